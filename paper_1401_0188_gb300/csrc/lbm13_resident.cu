// lbm13_resident.cu -- many time steps of one small lattice in one launch, the
// populations resident in shared memory.
//
// A lattice of up to a few hundred nodes squared is bound by latency, not by
// bandwidth or arithmetic: a launch per step costs the gap between two kernels
// and, inside each, the round trips to L2 of its loads.  Here one cooperative
// launch advances the lattice by up to 1024 steps.  Each block keeps a tile of
// it in shared memory and exchanges with its neighbours only, every K steps,
// through numbered units in L2 (lbm13_resident.h): one step costs the collisions
// of a tile plus 1/K of one trip to L2 and back.
//
// Microseconds per step, per-step launches (32-step graphs) and this kernel: FP32
// 64^2 periodic 3.3 and 1.15, 64^2 cavity 4.2 and 1.65, 256^2 cavity 4.9 and 2.3,
// 1024 x 128 channel 8.0 and 3.4, 512^2 periodic 6.3 and 4.2; FP64 (collision in
// integers in both) 64^2 periodic 5.4 and 2.8, 256^2 cavity 10.4 and 9.9, 1024 x
// 128 channel 14.5 and 15.7.  What bounds it is the chain of one node's step (450
// instructions in FP32, 1365 in FP64, at two to four clocks each with the few
// warps that a tile gives) between two barriers; an exchange through flags and
// fences instead of numbered units took 2.4 us instead of 0.8.
//
// Every node is pulled with the same links, wall rules and collision as in the
// per-step kernels, so the states are bit-identical to theirs.
//
// Every wait is bounded: a block that waits longer than timeout_ns for its
// neighbours' units records it in the error word and leaves, and so do the blocks
// that wait for it; the host reports LBM13_ETIMEOUT at its next synchronisation.
// Co-residency of all blocks is guaranteed by the cooperative launch.
#include <atomic>

#include "lbm13_internal.h"
#include "lbm13_resident.h"

// One launch reads what its other blocks wrote: loads go to L2, never to a
// possibly stale L1 line.
#define LBM13_LDG(p) __ldcg(p)
#include "lbm13_stepdev.cuh"

namespace lbm13 {

namespace {

// Population j of node (x, y) from the shared array (ox, oy: the coordinates of
// its first column and row): how the walls' states are read.
template <typename T, typename C, int EX>
struct SharedSrc {
    const T *sm;
    int ox, oy, rows;
    __device__ __forceinline__ C operator()(const StepArgs<T, C> &a, int j, int x, int y) const
    {
        int r = y - oy, c = x - ox;
#ifdef LBM13_DEBUG
        if (r < 0 || r >= rows || c < 0 || c >= EX) {
            atomicAdd(a.bad, 1ull);
            r = c = 0;
        }
#endif
        return C(sm[(r * Q + j) * EX + c]);
    }
};

// Debug builds: a population of the shared rows [0, n) reached by pointer; an access
// outside is counted and goes to the first one instead.
template <typename T, typename C>
__device__ __forceinline__ T *chk_shared(const StepArgs<T, C> &a, T *rows, size_t n, T *p)
{
#ifdef LBM13_DEBUG
    if (p < rows || p >= rows + n) {
        atomicAdd(a.bad, 1ull);
        return rows;
    }
#endif
    return p;
}

// One 16-byte unit of the exchange buffer, written and read as one access.
struct Unit {
    unsigned long long lo, hi;
};
__device__ __forceinline__ void unit_store(void *p, Unit u)
{
    asm volatile("{\n .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t;\n}" ::"l"(p),
                 "l"(u.lo), "l"(u.hi)
                 : "memory");
}
__device__ __forceinline__ Unit unit_load(const void *p)
{
    Unit u;
    asm volatile("{\n .reg .b128 t;\n ld.relaxed.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}"
                 : "=l"(u.lo), "=l"(u.hi)
                 : "l"(p)
                 : "memory");
    return u;
}

// A node's 13 populations as words.
__device__ __forceinline__ unsigned res_word(const float (&f)[Q], int i) { return i < Q ? __float_as_uint(f[i]) : 0u; }
__device__ __forceinline__ unsigned res_word(const double (&f)[Q], int i)
{
    return i >= 2 * Q ? 0u : unsigned((i & 1) ? __double2hiint(f[i >> 1]) : __double2loint(f[i >> 1]));
}
__device__ __forceinline__ void res_value(const unsigned *w, float &v, int j) { v = __uint_as_float(w[j]); }
__device__ __forceinline__ void res_value(const unsigned *w, double &v, int j)
{
    v = __hiloint2double(int(w[2 * j + 1]), int(w[2 * j]));
}

__device__ __forceinline__ unsigned long long res_clock()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Lattice coordinates of (x, y), wrapped where the axis is periodic; false for
// a node beyond a wall.
template <typename T, typename C>
__device__ __forceinline__ bool res_wrap(const StepArgs<T, C> &a, int &x, int &y)
{
    if (x < 0 || x >= a.nx) {
        if (!a.per_x) return false;
        x %= a.nx;
        x += x < 0 ? a.nx : 0;
    }
    if (y < 0 || y >= a.ny) {
        if (!a.per_y) return false;
        y %= a.ny;
        y += y < 0 ? a.ny : 0;
    }
    return true;
}

// States: the walls' states are evaluated once a step, one position along a wall a
// thread, in a pass and behind a barrier of their own, instead of by each of the up
// to ten links that use one.
// Tile `block` of the lattice of arguments a; force: whether it has a body force
// (a constant, but in a plan's kernel).
template <typename T, typename C, int EX, bool States>
__device__ __forceinline__ void resident_tile(const StepArgs<T, C> &a, bool force, const ResShape &s, int block,
                                              int nsteps, unsigned char *xchg, unsigned tag, unsigned *err,
                                              unsigned long long timeout_ns)
{
    extern __shared__ __align__(16) unsigned char res_mem[];
    __shared__ StepArgs<T, C> sa;  // for the edge nodes: a periodic axis without ends
    __shared__ ResRegion regs[kResMaxK];
    constexpr int kFar = 1 << 24;  // where a periodic axis' node 0 lies in sa's coordinates
    constexpr int kUnits = res_units(sizeof(T));
    T *const sm = reinterpret_cast<T *>(res_mem);
    const size_t held = size_t(s.rows) * Q * EX;
    T *const links = sm + held;  // [13][span]
    const int along = res_along(s);
    T *const states = links + size_t(s.edges) * Q;  // [4][along] pairs: the walls' density and energy
    unsigned *const found = reinterpret_cast<unsigned *>(states + size_t(8) * along);  // [13][span]
    unsigned *const places = found + size_t(s.edges) * Q;
    const int tid = threadIdx.x, K = s.K, threads = blockDim.x;
    const ResTile t = res_tile(s, a.nx, a.ny, block);
    const int fx = a.per_x ? kFar : 0, fy = a.per_y ? kFar : 0;
    const size_t nodes = size_t(a.nx) * a.ny;
    if (tid == 0) {
        sa = a;
        if (a.per_x) sa.nx = 1 << 28;
        if (a.per_y) sa.ny = 1 << 28;
    }
    if (tid < K) regs[tid] = res_region(t, a.nx, a.ny, a.per_x != 0, a.per_y != 0, 2 * tid, threads);
    int off = 2;  // rows that the array stands below its first row
    for (int i = tid; i < t.ew * t.eh; i += threads) {
        const int r = i / t.ew, c = i - r * t.ew;
        int x = t.ox + c, y = t.oy + r;
        if (!res_wrap(a, x, y)) continue;
        T *p = sm + (r + off) * Q * EX + c;
        T v[Q];
#pragma unroll
        for (int j = 0; j < Q; ++j)
            v[j] = __ldcg(chk(a, a.fin, a.fin + (long long)y * a.pitch + x + (long long)j * a.plane));
#pragma unroll
        for (int j = 0; j < Q; ++j) *chk_shared(a, sm, held, p + j * EX) = v[j];
    }
    __syncthreads();
    // the edge nodes, numbered as in the largest region: column and row in the
    // shared array
    const ResRegion &wide = regs[K - 1];
    const int edges = res_edge_count(wide), span = (edges + 31) & ~31;
    // the walls here whose state enters
    const bool has[4] = {wide.el > 0 && a.wall[WEST].needs_data, wide.er > 0 && a.wall[EAST].needs_data,
                         wide.ya < wide.elo && a.wall[SOUTH].needs_data, wide.yb > wide.ehi && a.wall[NORTH].needs_data};
    const bool pass = States && (has[WEST] || has[EAST] || has[SOUTH] || has[NORTH]);
    for (int r = wide.ya + tid / 32; r < wide.yb && edges > 0; r += threads / 32)
        for (int c = wide.xa + (tid & 31); c < wide.xb; c += 32)
            if (r < wide.elo || r >= wide.ehi || c - wide.xa < wide.el || c >= wide.xb - wide.er)
                places[res_edge_index(wide, c, r)] = unsigned(r - t.oy) << 16 | unsigned(c - t.ox);
    __syncthreads();
    // their links: where each comes from (an index into the rows) and what is
    // done to it, the same for every step
    for (int i = tid; i < Q * span; i += threads) {
        const int j = i / span, n = i - j * span;
        if (n >= edges) {
            found[i] = 0u;
            continue;
        }
        const unsigned at = places[n];
        const int x = int(at & 0xffffu) + t.ox + fx, y = int(at >> 16) + t.oy + fy;
        int js, xs, ys;
        const unsigned flags = resolve_link(sa, j, x, y, js, xs, ys);
        found[i] = flags << 16 | unsigned(((ys - t.oy - fy) * Q + js) * EX + xs - t.ox - fx);
    }
    __syncthreads();
    const int between = res_between(K, nsteps);
    for (int done = 0, e = 0; done < nsteps; ++e) {
        const int kk = min(between, nsteps - done);
        const bool last = done + kk >= nsteps;
        if (e > 0) {
            // the nodes around the tile, as soon as the neighbours have written them
            bool ok = true;
            const unsigned char *const in = xchg + size_t(e & 1) * kUnits * 16 * nodes;
            const unsigned want = tag + unsigned(e);
            for (int i = tid; i < res_halo_count(t) && ok; i += threads) {
                int x, y;
                res_halo_node(t, K, i, x, y);
                T *p = sm + (y - t.oy + off) * Q * EX + x - t.ox;
                if (!res_wrap(a, x, y)) continue;
                const unsigned char *g = in + (size_t(y) * a.nx + x) * 16;
                unsigned w[3 * kUnits];
                unsigned long long end = 0;
                for (;;) {
                    bool all = true;
#pragma unroll
                    for (int u = 0; u < kUnits; ++u) {
                        const Unit v = unit_load(g + size_t(u) * 16 * nodes);
                        w[3 * u] = unsigned(v.lo);
                        w[3 * u + 1] = unsigned(v.lo >> 32);
                        w[3 * u + 2] = unsigned(v.hi);
                        all = all && unsigned(v.hi >> 32) == want;
                    }
                    if (all) break;
                    const unsigned long long now = res_clock();
                    if (end == 0) end = now + timeout_ns;
                    if (now > end) {
                        atomicExch(err, 1u);
                        ok = false;
                        break;
                    }
                }
#pragma unroll
                for (int j = 0; j < Q; ++j) {
                    T v;
                    res_value(w, v, j);
                    *chk_shared(a, sm, held, p + j * EX) = v;
                }
            }
            if (__syncthreads_or(!ok)) return;
        }
        unsigned char *const out = xchg + size_t((e + 1) & 1) * kUnits * 16 * nodes;
        const unsigned mine = tag + unsigned(e + 1);
        for (int k = kk - 1; k >= 0; --k) {
            const ResRegion &g = regs[k];
            // every link of every edge node, four of them in flight in each
            // thread: the wall rules are the longest chain of a step, so that the
            // warps share it instead of leaving it to those that step the edge
            // nodes (nodes that only a larger region needs are of no use here, but
            // their places are inside the array)
            const T *const rows0 = sm + off * Q * EX;
            if (pass) {
                const SharedSrc<T, C, EX> src{sm, t.ox + fx, t.oy + fy - off, s.rows};
#pragma unroll
                for (int side = 0; side < 4; ++side) {
                    if (!has[side]) continue;
                    const bool xw = side <= EAST;
                    const int first = xw ? wide.ya - t.oy : wide.xa - t.ox;
                    const int n = xw ? wide.yb - wide.ya : wide.xb - wide.xa;
                    // each wall starts at a warp of its own
                    int i = tid - side * ((threads / 4) & ~31);
                    if (i < 0) i += threads;
                    for (; i < n; i += threads) {
                        const int at = first + i;
                        const WallState<C> st = wall_state_body(sa, side, at + (xw ? t.oy + fy : t.ox + fx), src);
                        states[2 * (side * along + at)] = T(st.rho);
                        states[2 * (side * along + at) + 1] = T(st.E);
                    }
                }
                __syncthreads();
            }
            for (int i0 = tid; i0 < Q * span; i0 += 4 * threads) {
                unsigned at[4];
                C v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = i0 + u * threads;
                    at[u] = i < Q * span ? found[i] : 0u;
                    v[u] = C(rows0[at[u] & 0xffffu]);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = i0 + u * threads;
                    if (i >= Q * span) break;
                    const unsigned f = at[u] >> 16;
                    C w = (f & kLinkNeg) ? -v[u] : v[u];
                    if (f & (kLinkX | kLinkY)) {
                        const unsigned place = places[i % span];
                        const int pc = int(place & 0xffffu), pr = int(place >> 16);
                        if constexpr (States) {
                            w = corrected_link(sa, f, pc, pr, w, [&](int side, int at) {
                                const T *p = states + 2 * (side * along + at);
                                return WallState<C>{C(p[0]), C(p[1])};
                            });
                        } else {
                            const SharedSrc<T, C, EX> src{sm, t.ox + fx, t.oy + fy - off, s.rows};
                            w = corrected_link(sa, f, pc + t.ox + fx, pr + t.oy + fy, w, [&](int side, int at) {
                                return wall_state_body(sa, side, at, src);
                            });
                        }
                    }
                    links[i] = T(w);
                }
            }
            const bool up = off == 2;  // rows move to the front: lowest rows first
            const int shift = up ? -2 * Q * EX : 2 * Q * EX, chunks = g.chunks;
            for (int c = 0; c < chunks; ++c) {
                const int ca = g.ya + (up ? c : chunks - 1 - c) * g.chunk, cb = min(ca + g.chunk, g.yb);
                int x = 0, y = 0;
                bool edge = false;
                const bool valid = res_item(g, ca, cb, tid, x, y, edge);
                T *const p = sm + (y - t.oy + off) * Q * EX + x - t.ox;
                C f[Q];
                if (valid && !edge) {
#pragma unroll
                    for (int j = 0; j < Q; ++j) f[j] = C(*chk_shared(a, sm, held, p + ((j - Q * cvy(j)) * EX - cvx(j))));
                }
                __syncthreads();  // every read of the chunk before its writes
                if (valid) {
                    if (edge) {
                        const T *l = links + res_edge_index(wide, x, y);
#pragma unroll
                        for (int j = 0; j < Q; ++j) f[j] = C(l[j * span]);
                    }
                    if (force)
                        collide<true>(f, a.k);
                    else
                        collide<false>(f, a.k);
#pragma unroll
                    for (int j = 0; j < Q; ++j) *chk_shared(a, sm, held, p + (j * EX + shift)) = T(f[j]);
                    if (k == 0 && last) {
                        store(a, x, y, f);
                    } else if (k == 0 && (x < t.x0 + 2 * K || x >= t.x1 - 2 * K || y < t.y0 + 2 * K ||
                                          y >= t.y1 - 2 * K)) {
                        unsigned char *q = out + (size_t(y) * a.nx + x) * 16;
#pragma unroll
                        for (int u = 0; u < kUnits; ++u) {
                            const unsigned w0 = res_word(f, 3 * u), w1 = res_word(f, 3 * u + 1),
                                           w2 = res_word(f, 3 * u + 2);
                            unit_store(q + size_t(u) * 16 * nodes,
                                       Unit{w0 | (unsigned long long)w1 << 32, w2 | (unsigned long long)mine << 32});
                        }
                    }
                }
            }
            off ^= 2;
            __syncthreads();
        }
        done += kk;
    }
}

template <typename T, typename C, bool Force, int EX, bool States>
__global__ void __launch_bounds__(res_threads(sizeof(T)), 1)
    resident_kernel(const StepArgs<T, C> a, const ResShape s, int nsteps, unsigned char *xchg, unsigned tag,
                    unsigned *err, unsigned long long timeout_ns)
{
    resident_tile<T, C, EX, States>(a, Force, s, blockIdx.x, nsteps, xchg, tag, err, timeout_ns);
}

// The lattices of a plan: each block takes its tile's lattice and shape from the
// table, the lattice's arguments (of the plan's parity) into shared memory; the
// collision's coefficients read there cost 2 to 5% against constants (256^2 cavity
// 2.33 and 2.38 us a step).  Served cavities and channels of 64 to 192 columns in one
// plan, microseconds a step by single launches (32-step graphs) and here: 2 solves
// 3.7 and 2.0, 5: 3.9 and 2.2, 12: 6.0 and 3.7, 24 (247,040 nodes, all 152 SMs): 9.1
// and 6.3; the nodes of the fullest tile bound the last.
template <int EX, bool States>
__global__ void __launch_bounds__(res_threads(4), 1)
    resident_plan_kernel(const BatchDesc<float, float> *__restrict__ descs, const ResPlanTile *__restrict__ tiles,
                         int parity, int nsteps, unsigned char *xchg, unsigned tag, unsigned *err,
                         unsigned long long timeout_ns)
{
    __shared__ StepArgs<float, float> args;
    __shared__ ResPlanTile tile;
    if (threadIdx.x == 0) tile = tiles[blockIdx.x];
    __syncthreads();
    const BatchDesc<float, float> &d = descs[tile.lattice];
    static_assert(sizeof(StepArgs<float, float>) % 4 == 0, "copied word by word");
    const unsigned *src = reinterpret_cast<const unsigned *>(&d.a[parity]);
    for (int i = threadIdx.x; i < int(sizeof(args) / 4); i += blockDim.x) reinterpret_cast<unsigned *>(&args)[i] = src[i];
    __syncthreads();
    if (threadIdx.x == 0 && nsteps % 2 == 0) args.fout = const_cast<float *>(args.fin);
    __syncthreads();
    resident_tile<float, float, EX, States>(args, d.force != 0, tile.s, tile.tile, nsteps, xchg + tile.offset, tag, err,
                                            timeout_ns);
}

// The shared-memory allowance is a per-device attribute: raised once on each device
// that launches the kernel.
cudaError_t res_allow(const void *fn, std::atomic<unsigned long long> &raised)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (!bit || !(raised.load() & bit)) {
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmem);
        if (e != cudaSuccess) return e;
        raised.fetch_or(bit);
    }
    return cudaSuccess;
}

template <typename T, typename C, bool States>
const void *resident_fn(int ex, bool force)
{
    if (ex == 24)
        return force ? reinterpret_cast<const void *>(&resident_kernel<T, C, true, 24, States>)
                     : reinterpret_cast<const void *>(&resident_kernel<T, C, false, 24, States>);
    if (ex == 32)
        return force ? reinterpret_cast<const void *>(&resident_kernel<T, C, true, 32, States>)
                     : reinterpret_cast<const void *>(&resident_kernel<T, C, false, 32, States>);
    return force ? reinterpret_cast<const void *>(&resident_kernel<T, C, true, 48, States>)
                 : reinterpret_cast<const void *>(&resident_kernel<T, C, false, 48, States>);
}

// The kernel of a split, its allowance raised.
template <typename T, typename C>
cudaError_t resident_ready(const ResShape &s, bool force, bool states, const void *&fn)
{
    fn = states ? resident_fn<T, C, true>(s.ex, force) : resident_fn<T, C, false>(s.ex, force);
    static std::atomic<unsigned long long> raised[4 * kResWidths];
    const int which = (s.ex == 24 ? 0 : s.ex == 32 ? 1 : 2) + (force ? kResWidths : 0) + (states ? 2 * kResWidths : 0);
    return res_allow(fn, raised[which]);
}
cudaError_t resident_plan_ready(int ex, bool states, const void *&fn)
{
    const bool wide = ex == kResPlanWidths[1];
    fn = wide ? (states ? reinterpret_cast<const void *>(&resident_plan_kernel<kResPlanWidths[1], true>)
                        : reinterpret_cast<const void *>(&resident_plan_kernel<kResPlanWidths[1], false>))
              : (states ? reinterpret_cast<const void *>(&resident_plan_kernel<kResPlanWidths[0], true>)
                        : reinterpret_cast<const void *>(&resident_plan_kernel<kResPlanWidths[0], false>));
    static std::atomic<unsigned long long> raised[4];
    return res_allow(fn, raised[(wide ? 2 : 0) + (states ? 1 : 0)]);
}

int res_capacity(const void *fn, int threads, size_t smem)
{
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return per * device_sm_count();
}

} // namespace

template <typename T, typename C>
cudaError_t launch_resident(const StepArgs<T, C> &a, bool force, int nsteps, const ResShape &s, void *xchg,
                            unsigned tag, unsigned *err, unsigned long long timeout_ns, cudaStream_t stream, int absent)
{
    const void *fn = nullptr;
    const cudaError_t e = resident_ready<T, C>(s, force, res_states_pass(a.wall), fn);
    if (e != cudaSuccess) return e;
    StepArgs<T, C> pa = a;
    if (nsteps % 2 == 0) pa.fout = const_cast<T *>(a.fin);
    ResShape ps = s;
    unsigned char *px = static_cast<unsigned char *>(xchg);
    void *args[] = {&pa, &ps, &nsteps, &px, &tag, &err, &timeout_ns};
    return cudaLaunchCooperativeKernel(fn, dim3(s.gx * s.gy - absent), dim3(s.threads), args,
                                       res_smem(s, int(sizeof(T))), stream);
}

template <typename T, typename C>
int resident_capacity(const ResShape &s, bool force, const WallArgs<C> *wall)
{
    const void *fn = nullptr;
    if (resident_ready<T, C>(s, force, res_states_pass(wall), fn) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return res_capacity(fn, s.threads, res_smem(s, int(sizeof(T))));
}
int resident_plan_capacity(int ex, int threads, size_t smem, bool states)
{
    const void *fn = nullptr;
    if (resident_plan_ready(ex, states, fn) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return res_capacity(fn, threads, smem);
}

cudaError_t launch_resident_plan(const BatchDesc<float, float> *descs, const ResPlanTile *tiles, int ntiles, int ex,
                                 int threads, size_t smem, bool states, int parity, int nsteps, void *xchg,
                                 unsigned tag, unsigned *err, unsigned long long timeout_ns, cudaStream_t stream)
{
    const void *fn = nullptr;
    const cudaError_t e = resident_plan_ready(ex, states, fn);
    if (e != cudaSuccess) return e;
    unsigned char *px = static_cast<unsigned char *>(xchg);
    void *args[] = {&descs, &tiles, &parity, &nsteps, &px, &tag, &err, &timeout_ns};
    return cudaLaunchCooperativeKernel(fn, dim3(ntiles), dim3(threads), args, smem, stream);
}

template int resident_capacity<double, double>(const ResShape &, bool, const WallArgs<double> *);
template int resident_capacity<float, float>(const ResShape &, bool, const WallArgs<float> *);
template cudaError_t launch_resident<double, double>(const StepArgs<double, double> &, bool, int, const ResShape &,
                                                     void *, unsigned, unsigned *, unsigned long long, cudaStream_t, int);
template cudaError_t launch_resident<float, float>(const StepArgs<float, float> &, bool, int, const ResShape &, void *,
                                                   unsigned, unsigned *, unsigned long long, cudaStream_t, int);

} // namespace lbm13
