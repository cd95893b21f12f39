// lbm13_aux.cu -- initialisation, moment read-out and the FP64 reductions.
//
// Read-outs and reductions run in double precision in both storage modes
// (a float deviation converts to double exactly).  The reductions are
// deterministic: each thread sums its nodes in a fixed grid-stride order, a
// block combines its threads with warp shuffles and in warp order, and the last
// block to finish combines the per-block partials in a fixed order.
#include "lbm13_read.cuh"

namespace lbm13 {

namespace {

// ---------------------------------------------------------------- init

// f*_j = f_eq,j(rho, rho u, E) with E = rho (26 T - 28) + 13 rho |u|^2, stored as
// the deviation from the rest populations.
template <typename T>
__global__ void init_kernel(T *f, int nx, int ny, long long pitch, long long plane, const InitFix c,
                            const double *__restrict__ rho, const double *__restrict__ ux,
                            const double *__restrict__ uy, const double *__restrict__ Tf)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= nx) return;
    const long long i = (long long)y * nx + x;
    T *p = f + (long long)y * pitch + x;
    T g[Q];
    init_node(rho[i], ux[i], uy[i], Tf[i], c, g);
#pragma unroll
    for (int j = 0; j < Q; ++j) p[(long long)j * plane] = g[j];
}

// -------------------------------------------------------------- moments

// The selected fields of one node in FP64, in order: bits 0 .. 12 the absolute
// moments, then u_x, u_y, T, p and the Sec. 7 energy.  All: moments other than rho, E
// and the momentum may be among them (their 25 operations are left out otherwise).
constexpr unsigned kOtherMoments = 0x1fccu;
template <bool All, typename T, typename Put>
__device__ __forceinline__ void put_fields(const ReadArgs<T> &a, const double (&f)[Q], unsigned mask, Put put)
{
    Mom<double> d;
    forward(f, d);
    if (mask & 0x1u) put(1.0 + d.rho);
    if (mask & 0x2u) put(a.rest.E0 + d.E);
    if (All && (mask & 0x4u)) put(a.rest.eps0 + d.eps);
    if (All && (mask & 0x8u)) put(a.rest.vpi0 + d.vpi);
    if (mask & 0x10u) put(d.jx);
    if (mask & 0x20u) put(d.jy);
    if (All && (mask & 0x40u)) put(d.qx);
    if (All && (mask & 0x80u)) put(d.qy);
    if (All && (mask & 0x100u)) put(d.rx);
    if (All && (mask & 0x200u)) put(d.ry);
    if (All && (mask & 0x400u)) put(d.XX);
    if (All && (mask & 0x800u)) put(d.XY);
    if (All && (mask & 0x1000u)) put(d.XXe);
    if (!(mask >> 13)) return;
    const double T0 = a.rest.T0;
    double ux, uy, dT, dp;
    macro_dev(a, d.rho, d.E, d.jx, d.jy, ux, uy, dT, dp);
    if (mask & 0x2000u) put(ux);
    if (mask & 0x4000u) put(uy);
    if (mask & 0x8000u) put(T0 + dT);
    if (mask & 0x10000u) put(T0 + dp);
    if (mask & 0x20000u) put(a.rest.E0 + d.E - 6.5 * (ux * ux + uy * uy));
}
template <typename T>
__device__ __noinline__ void put_fields_plain(const ReadArgs<T> &a, const T (&raw)[Q], unsigned mask, double *o, long long n)
{
    double f[Q];
    widen(raw, f);
    put_fields<true>(a, f, mask, [&](double v) {
        *o = v;
        o += n;
    });
}

// The same for FP32 storage in integers.
template <typename Put>
__device__ __forceinline__ void put_fields_fixed(const ReadArgs<float> &a, const float (&f)[Q], unsigned mask, Put put,
                                                 double *o, long long n)
{
    FxSums s;
    FxMacro m;
    if (!fx_sums(f, s) || ((mask >> 13) != 0u && !fx_macro(s, a.fx, m))) {
        float g[Q];  // f itself stays in registers
#pragma unroll
        for (int j = 0; j < Q; ++j) g[j] = f[j];
        put_fields_plain(a, g, mask, o, n);
        return;
    }
    if (mask & 0x1u) put(1.0 + s.value(s.rho()));
    if (mask & 0x2u) put(a.rest.E0 + s.energy());
    if (mask & 0xcu) {
        const double f0 = s.value(s.f0), S1 = s.value(s.S1), S5 = s.value(s.S5), S9 = s.value(s.S9);
        if (mask & 0x4u) put(a.rest.eps0 + fma(34.0, S9, fma(-67.0, S5, fma(-2.0, S1, 140.0 * f0))));
        if (mask & 0x8u) put(a.rest.vpi0 + fma(-6.0, S5, fma(8.0, S1, fma(-12.0, f0, S9))));
    }
    if (mask & 0x10u) put(s.value(s.jx()));
    if (mask & 0x20u) put(s.value(s.jy()));
    if (mask & 0x40u) put(s.value(2 * s.b9 - 2 * s.b1 - s.dm));
    if (mask & 0x80u) put(s.value(2 * s.b10 - 2 * s.b2 - s.dp));
    if (mask & 0x100u) put(s.value(4 * s.b1 - 3 * s.dm + s.b9));
    if (mask & 0x200u) put(s.value(4 * s.b2 - 3 * s.dp + s.b10));
    if (mask & 0x400u) put(s.value(s.X1 + 4 * s.X9));
    if (mask & 0x800u) put(s.value(s.X5));
    if (mask & 0x1000u) put(s.value(s.X9 - 4 * s.X1));
    if (mask & 0x2000u) put(s.value(m.u));
    if (mask & 0x4000u) put(s.value(m.v));
    const double T0 = a.rest.T0;
    if (mask & 0x8000u) put(T0 + s.value(m.T));
    if (mask & 0x10000u) put(T0 + s.value(m.p));
    if (mask & 0x20000u) {
        const double ux = s.value(m.u), uy = s.value(m.v);
        put(a.rest.E0 + s.energy() - 6.5 * (ux * ux + uy * uy));
    }
}

// The selected fields of one node per thread.  The integer read-out of FP32 storage
// leaves one conversion and at most a few FP64 operations per selected field (8192^2
// FP32, rho, u and T: see the header of lbm13_fixed_io.cuh).
template <typename T>
__global__ void __launch_bounds__(128) moments_kernel(const ReadArgs<T> a, double *__restrict__ out, unsigned mask)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= a.nx) return;
    T f[Q];
    load_node(a, (long long)y * a.pitch + x, f);
    const long long n = (long long)a.nx * a.ny;
    double *o = out + (long long)y * a.nx + x;
    const auto put = [&](double v) {
        *o = v;
        o += n;
    };
    if constexpr (sizeof(T) == 8) {
        if (mask & kOtherMoments)
            put_fields<true>(a, f, mask, put);
        else
            put_fields<false>(a, f, mask, put);
    } else {
        put_fields_fixed(a, f, mask, put, o, n);
    }
}

// ----------------------------------------------------------- reductions

// Sums of the N = 8 values over the lanes of a warp, value i left in the lanes
// 4 i .. 4 i + 3: a lane hands half of its values on at each of the first three
// exchanges, 9 additions instead of 40 (64 clocks of the FP64 pipe each).
__device__ __forceinline__ double warp_sums(double (&v)[8])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 4, o = 16; h > 0; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double mine = up ? v[i + h] : v[i], theirs = up ? v[i] : v[i + h];
            v[i] = mine + __shfl_xor_sync(0xffffffffu, theirs, o);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    return v[0];
}

// Largest of non-negative doubles, compared as integers (their order); NaN is
// passed over.
__device__ __forceinline__ void keep_largest(unsigned long long &m, double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    if (b <= 0x7ff0000000000000ull && b > m) m = b;
}
__device__ __forceinline__ unsigned long long warp_largest(unsigned long long m)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, m, o);
        m = t > m ? t : m;
    }
    return m;
}

constexpr int kSums = 8, kMax = 2;  // of a pass: sums, then maxima

// The 8 sums and 2 maxima of the block's threads into dst[10], in a fixed order.
__device__ __forceinline__ void block_combine(double (&s)[kSums], unsigned long long (&mx)[kMax], double *dst)
{
    __shared__ double sh[kReduceThreads / 32][kSums + kMax];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const double t = warp_sums(s);
    if ((lane & 3) == 0) sh[wid][lane >> 2] = t;
#pragma unroll
    for (int i = 0; i < kMax; ++i) {
        const unsigned long long m = warp_largest(mx[i]);
        if (lane == 0) sh[wid][kSums + i] = __longlong_as_double((long long)m);
    }
    __syncthreads();
    if (threadIdx.x < kSums) {
        double r = 0.0;
        for (int w = 0; w < kReduceThreads / 32; ++w) r += sh[w][threadIdx.x];
        dst[threadIdx.x] = r;
    } else if (threadIdx.x < kSums + kMax) {
        unsigned long long m = 0;
        for (int w = 0; w < kReduceThreads / 32; ++w) keep_largest(m, sh[w][threadIdx.x]);
        dst[threadIdx.x] = __longlong_as_double((long long)m);
    }
}

// Whether this block is the last of its pass to have written its partials (then
// every block's are visible to it); *count is left at zero.
__device__ __forceinline__ bool last_block(unsigned *count, int nblocks)
{
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(count, 1u) == unsigned(nblocks - 1);
        if (last) *count = 0u;
        __threadfence();
    }
    __syncthreads();
    return last;
}

// The partials of all blocks combined, slot by slot: a warp a slot, lane by lane
// in block order, then over the lanes.
__device__ __forceinline__ void combine_partials(const double *partials, int nblocks, double *res)
{
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < kSums + kMax; i += kReduceThreads / 32) {
        if (i < kSums) {
            double t = 0.0;
            for (int b = lane; b < nblocks; b += 32) t += __ldcg(partials + (long long)b * kPartials + i);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) res[i] = t;
        } else {
            unsigned long long m = 0;
            for (int b = lane; b < nblocks; b += 32) keep_largest(m, __ldcg(partials + (long long)b * kPartials + i));
            m = warp_largest(m);
            if (lane == 0) res[i] = __longlong_as_double((long long)m);
        }
    }
    __syncthreads();
}

// First pass of block `block` of a lattice: velocity and temperature of every
// node, and the partial sums 0 drho, 1 jx, 2 jy, 3 dE, 4 ux, 5 uy, 6 T - T0, 7
// non-finite populations, largest 0 |u|^2.  The last block leaves in stats: 0 mean
// ux, 1 mean uy, 2 mean T, 3 .. 12 the combined slots.
template <typename T>
__device__ __forceinline__ void fields_pass(const ReadArgs<T> &a, const ReduceBufs &b, int block)
{
    __shared__ double res[kSums + kMax];
    const long long n = (long long)a.nx * a.ny;
    const double T0 = a.rest.T0;
    double s[kSums] = {0, 0, 0, 0, 0, 0, 0, 0};
    unsigned long long mx[kMax] = {0, 0};
    for (long long i = (long long)block * kReduceThreads + threadIdx.x; i < n; i += (long long)b.nblocks * kReduceThreads) {
        const int y = int(i / a.nx), x = int(i - (long long)y * a.nx);
        const NodeDev d = node_dev(a, (long long)y * a.pitch + x);
        b.fields[i] = d.ux;
        b.fields[n + i] = d.uy;
        b.fields[2 * n + i] = T0 + d.T;
        s[0] += d.rho;
        s[1] += d.jx;
        s[2] += d.jy;
        s[3] += d.E;
        s[4] += d.ux;
        s[5] += d.uy;
        s[6] += d.T;
        if (d.bad != 0.0) s[7] += d.bad;
        keep_largest(mx[0], d.ux * d.ux + d.uy * d.uy);
    }
    block_combine(s, mx, b.partials + (long long)block * kPartials);
    if (!last_block(b.done, b.nblocks)) return;
    combine_partials(b.partials, b.nblocks, res);
    if (threadIdx.x < kSums + kMax) b.stats[3 + threadIdx.x] = res[threadIdx.x];
    if (threadIdx.x < 3) b.stats[threadIdx.x] = (threadIdx.x == 2 ? T0 : 0.0) + res[4 + threadIdx.x] / double(n);
}

// Second pass: partial sums 0 .. 2 (F - snap)^2, 3 .. 5 (F - mean F)^2 for F = ux,
// uy, T, 6 Nusselt; largest 0 S_u^2, 1 S_T.  The last block writes the results.
template <typename T>
__device__ __forceinline__ void residual_pass(const ReadArgs<T> &a, const ReduceBufs &b, const ReduceConf &c,
                                              const unsigned *err, double *out, int block)
{
    __shared__ double res[kSums + kMax];
    const long long n = (long long)a.nx * a.ny;
    const double mean[3] = {b.stats[0], b.stats[1], b.stats[2]};
    const double Tref_asym = c.asym_walls ? c.Tasym : mean[2];
    double s[kSums] = {0, 0, 0, 0, 0, 0, 0, 0};
    unsigned long long mx[kMax] = {0, 0};
    const double *F[3] = {b.fields, b.fields + n, b.fields + 2 * n};
    for (long long i = (long long)block * kReduceThreads + threadIdx.x; i < n; i += (long long)b.nblocks * kReduceThreads) {
        const int y = int(i / a.nx), x = int(i - (long long)y * a.nx);
        double v[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            v[q] = F[q][i];
            if (c.have_snap) {
                const double dv = v[q] - b.snap[q * n + i];
                s[q] += dv * dv;
            }
            const double e = v[q] - mean[q];
            s[3 + q] += e * e;
            b.snap[q * n + i] = v[q];
        }
        if (c.nusselt) {
            const double *Tf = F[2];
            double dTdx;
            if (x == 0) dTdx = (-3.0 * Tf[i] + 4.0 * Tf[i + 1] - Tf[i + 2]) / 2.0;
            else if (x == a.nx - 1) dTdx = (3.0 * Tf[i] - 4.0 * Tf[i - 1] + Tf[i - 2]) / 2.0;
            else dTdx = (Tf[i + 1] - Tf[i - 1]) / 2.0;
            s[6] += v[0] * (v[2] - c.Tref) - c.kappa * dTdx;
        }
        const long long m = (long long)(a.ny - 1 - y) * a.nx + (a.nx - 1 - x);
        const double sx = v[0] + F[0][m], sy = v[1] + F[1][m];
        keep_largest(mx[0], sx * sx + sy * sy);
        keep_largest(mx[1], fabs((v[2] - Tref_asym) + (F[2][m] - Tref_asym)));
    }
    block_combine(s, mx, b.partials + (long long)block * kPartials);
    if (!last_block(b.done, b.nblocks)) return;
    combine_partials(b.partials, b.nblocks, res);
    if (threadIdx.x != 0) return;
    // the velocity is one vector field: both components over its variation
    const double floor_ = 1e-6 * sqrt(double(n));
    for (int q = 0; q < 4; ++q) out[q] = 0.0;
    if (c.have_snap && c.K > 0) {
        const double du = fmax(sqrt(res[3] + res[4]), floor_), dT = fmax(sqrt(res[5]), floor_);
        const double K = double(c.K);
        out[1] = sqrt(res[0]) / (K * du);
        out[2] = sqrt(res[1]) / (K * du);
        out[3] = sqrt(res[2]) / (K * dT);
        out[0] = fmax(sqrt(res[0] + res[1]) / (K * du), out[3]);
    }
    const double *p1 = b.stats + 3;
    out[4] = double(n) + p1[0];
    out[5] = p1[1];
    out[6] = p1[2];
    out[7] = double(n) * a.rest.E0 + p1[3];
    out[8] = c.nusselt ? res[6] / (double(a.ny) * c.kappa * c.dT) : 0.0;
    out[9] = sqrt(res[8]);  // the square root keeps the order
    out[10] = res[9];
    out[11] = sqrt(p1[8]);
    out[12] = p1[7];
    out[13] = c.have_snap ? double(c.K) : 0.0;
    out[14] = double(c.step);
    out[15] = b.stats[2];
    if (err) out[16] = double(*err);
}

// One lattice's reduction, a launch a pass (the last block of each combines the
// partials, which took two more launches of one block).
template <typename T>
__global__ void __launch_bounds__(kReduceThreads) fields_kernel(const ReduceJob<T> j)
{
    fields_pass(j.a, j.b, blockIdx.x);
}
template <typename T>
__global__ void __launch_bounds__(kReduceThreads) residual_kernel(const ReduceJob<T> j)
{
    residual_pass(j.a, j.b, j.c, j.err, j.out, blockIdx.x);
}

// The reductions of many lattices, a launch a pass for all of them: block i works
// for the last lattice whose first block is not after i.
template <typename T>
__device__ __forceinline__ const ReduceJob<T> &job_of(const ReduceJob<T> *jobs, int count)
{
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].first <= int(blockIdx.x)) lo = mid;
        else hi = mid - 1;
    }
    return jobs[lo];
}
template <typename T>
__global__ void __launch_bounds__(kReduceThreads) fields_batch_kernel(const ReduceJob<T> *__restrict__ jobs, int count)
{
    const ReduceJob<T> &j = job_of(jobs, count);
    fields_pass(j.a, j.b, int(blockIdx.x) - j.first);
}
template <typename T>
__global__ void __launch_bounds__(kReduceThreads) residual_batch_kernel(const ReduceJob<T> *__restrict__ jobs, int count)
{
    const ReduceJob<T> &j = job_of(jobs, count);
    residual_pass(j.a, j.b, j.c, j.err, j.out, int(blockIdx.x) - j.first);
}

// --------------------------------------------------------- projections

// Per-block partials of the Fourier projections, [block][kProj]:
// slot 4 f + 2 h + c = sum F_f trig_c(2 pi (h + 1) m / N), m = (kx x ny + ky y nx) mod N
// (kx, ky already reduced to [0, nx) x [0, ny)).
template <typename T>
__global__ void __launch_bounds__(kReduceThreads) project_kernel(const ReadArgs<T> a, long long kx, long long ky,
                                                                 double *partials, unsigned *done, double *out)
{
    const long long n = (long long)a.nx * a.ny;
    double s[kProj];
#pragma unroll
    for (int i = 0; i < kProj; ++i) s[i] = 0.0;
    for (long long i = (long long)blockIdx.x * kReduceThreads + threadIdx.x; i < n;
         i += (long long)gridDim.x * kReduceThreads) {
        const int y = int(i / a.nx), x = int(i - (long long)y * a.nx);
        const NodeDev d = node_dev(a, (long long)y * a.pitch + x);
        const double v[6] = {d.rho, d.ux, d.uy, d.T, d.E, d.p};
        const long long m = ((kx * x) % a.nx * a.ny + (ky * y) % a.ny * a.nx) % n;
        double c1, s1, c2, s2;
        sincospi(2.0 * double(m) / double(n), &s1, &c1);
        sincospi(2.0 * double((2 * m) % n) / double(n), &s2, &c2);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            s[4 * q + 0] += v[q] * c1;
            s[4 * q + 1] += v[q] * s1;
            s[4 * q + 2] += v[q] * c2;
            s[4 * q + 3] += v[q] * s2;
        }
    }
    __shared__ double sh[kReduceThreads / 32][kProj];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int g = 0; g < kProj / 8; ++g) {
        double v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = s[8 * g + i];
        const double t = warp_sums(v);
        if ((lane & 3) == 0) sh[wid][8 * g + (lane >> 2)] = t;
    }
    __syncthreads();
    if (threadIdx.x < kProj) {
        double t = 0.0;
        for (int w = 0; w < kReduceThreads / 32; ++w) t += sh[w][threadIdx.x];
        partials[(long long)blockIdx.x * kProj + threadIdx.x] = t;
    }
    // the last block combines the partials, a warp a slot
    if (!last_block(done, gridDim.x)) return;
    for (int i = wid; i < kProj; i += kReduceThreads / 32) {
        double t = 0.0;
        for (int b = lane; b < int(gridDim.x); b += 32) t += __ldcg(partials + (long long)b * kProj + i);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) out[i] = t;
    }
}

} // namespace

template <typename T>
cudaError_t launch_init(T *f, int nx, int ny, long long pitch, long long plane, const InitFix &x, const double *rho,
                        const double *ux, const double *uy, const double *Tf, cudaStream_t s)
{
    dim3 block(128), grid((nx + 127) / 128, ny);
    init_kernel<T><<<grid, block, 0, s>>>(f, nx, ny, pitch, plane, x, rho, ux, uy, Tf);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_moments(const ReadArgs<T> &a, double *out, unsigned mask, cudaStream_t s)
{
    dim3 block(128), grid((a.nx + 127) / 128, a.ny);
    moments_kernel<T><<<grid, block, 0, s>>>(a, out, mask);
    return cudaGetLastError();
}

// ------------------------------------------------------ y-slab halos
//
// Entry i of a packed halo [2 rows][4 populations][nx]: pack reads the rows
// next to the halo rows of `side` (south: 2, 3; north: ny-4, ny-3) for the
// populations that move across it (south: v_y < 0; north: v_y > 0); unpack
// writes the halo rows (south: 0, 1; north: ny-2, ny-1) for the populations
// that move in (south: v_y > 0; north: v_y < 0).
__device__ __forceinline__ int halo_plane(bool up, int k)
{
    return up ? (k == 0 ? 2 : k == 1 ? 5 : k == 2 ? 6 : 10) : (k == 0 ? 4 : k == 1 ? 7 : k == 2 ? 8 : 12);
}

template <typename T>
__global__ void halo_kernel(T *__restrict__ f, int nx, int ny, long long pitch, long long plane, int side, int pack,
                            T *__restrict__ buf)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 8LL * nx) return;
    const int x = int(i % nx), k = int((i / nx) % 4), r = int(i / (4LL * nx));
    const bool south = side == SOUTH;
    const int y = pack ? (south ? 2 + r : ny - 4 + r) : (south ? r : ny - 2 + r);
    const bool up = pack ? !south : south;
    T *p = f + (long long)halo_plane(up, k) * plane + (long long)y * pitch + x;
    if (pack)
        buf[i] = *p;
    else
        *p = buf[i];
}

template <typename T>
cudaError_t launch_halo(T *f, int nx, int ny, long long pitch, long long plane, int side, bool pack, T *buf,
                        cudaStream_t s)
{
    const long long n = 8LL * nx;
    halo_kernel<T><<<unsigned((n + 255) / 256), 256, 0, s>>>(f, nx, ny, pitch, plane, side, pack ? 1 : 0, buf);
    return cudaGetLastError();
}

template cudaError_t launch_halo<double>(double *, int, int, long long, long long, int, bool, double *, cudaStream_t);
template cudaError_t launch_halo<float>(float *, int, int, long long, long long, int, bool, float *, cudaStream_t);

int reduce_blocks(int nx, int ny)
{
    const long long n = (long long)nx * ny;
    long long b = (n + kReduceThreads - 1) / kReduceThreads;
    const long long cap = 8LL * device_sm_count();  // eight blocks per SM
    return int(b < cap ? (b < 1 ? 1 : b) : cap);
}

template <typename T>
cudaError_t launch_reduce(const ReduceJob<T> &j, cudaStream_t s)
{
    fields_kernel<T><<<j.b.nblocks, kReduceThreads, 0, s>>>(j);
    residual_kernel<T><<<j.b.nblocks, kReduceThreads, 0, s>>>(j);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_reduce_batch(const ReduceJob<T> *jobs, int count, int blocks, cudaStream_t s)
{
    fields_batch_kernel<T><<<blocks, kReduceThreads, 0, s>>>(jobs, count);
    residual_batch_kernel<T><<<blocks, kReduceThreads, 0, s>>>(jobs, count);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_project(const ReadArgs<T> &a, int kx, int ky, double *partials, int nblocks, unsigned *done,
                           double *out_dev, cudaStream_t s)
{
    const long long kxm = ((long long)kx % a.nx + a.nx) % a.nx, kym = ((long long)ky % a.ny + a.ny) % a.ny;
    project_kernel<T><<<nblocks, kReduceThreads, 0, s>>>(a, kxm, kym, partials, done, out_dev);
    return cudaGetLastError();
}

template cudaError_t launch_init<double>(double *, int, int, long long, long long, const InitFix &, const double *,
                                         const double *, const double *, const double *, cudaStream_t);
template cudaError_t launch_init<float>(float *, int, int, long long, long long, const InitFix &, const double *,
                                        const double *, const double *, const double *, cudaStream_t);
template cudaError_t launch_moments<double>(const ReadArgs<double> &, double *, unsigned, cudaStream_t);
template cudaError_t launch_moments<float>(const ReadArgs<float> &, double *, unsigned, cudaStream_t);
template cudaError_t launch_reduce<double>(const ReduceJob<double> &, cudaStream_t);
template cudaError_t launch_reduce<float>(const ReduceJob<float> &, cudaStream_t);
template cudaError_t launch_reduce_batch<double>(const ReduceJob<double> *, int, int, cudaStream_t);
template cudaError_t launch_reduce_batch<float>(const ReduceJob<float> *, int, int, cudaStream_t);

template cudaError_t launch_project<double>(const ReadArgs<double> &, int, int, double *, int, unsigned *, double *,
                                            cudaStream_t);
template cudaError_t launch_project<float>(const ReadArgs<float> &, int, int, double *, int, unsigned *, double *,
                                           cudaStream_t);

} // namespace lbm13
