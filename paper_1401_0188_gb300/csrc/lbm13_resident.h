// lbm13_resident.h -- many steps of one small lattice in one launch, its
// populations resident in shared memory (resident_kernel, lbm13_resident.cu):
// the split of the lattice into tiles, the work items of a tile, and the launch.
#pragma once

#include <vector>

#include "lbm13_internal.h"

namespace lbm13 {

// The lattice is split into gx x gy tiles, one block (and one SM) each.  A block
// holds its tile and 2 K nodes around it, steps K times on a region that shrinks
// by two nodes a step, and then exchanges: it writes the outer 2 K nodes of its
// tile to an exchange buffer and reads the 2 K nodes around its tile from it.
// There is no flag and no fence: the buffer holds units of 16 bytes, three words
// of a node's populations and the exchange's number, written and read as one
// access, and a reader repeats its loads until every unit carries the number it
// waits for.  Two copies alternate; a block writes a copy again only after it has
// read what its neighbours wrote later than their last read of it.
//
// Shared memory is [row][plane][ex columns] with two spare rows: a step moves
// every node two rows down or up (in turn), so that it can be done in place: the
// nodes are taken in chunks of whole rows, all reads of a chunk before its
// writes, and what a chunk overwrites no later chunk reads.
// largest number of threads of a block, one node each at a time (64 registers in
// FP32, 128 in FP64)
LBM13_HD constexpr int res_threads(int elem) { return elem == 4 ? 1024 : 512; }
constexpr int kResMaxTiles = 256;
// 16-byte units of a node's 13 populations: 13 or 26 words, three to a unit
LBM13_HD constexpr int res_units(int elem) { return (Q * elem / 4 + 2) / 3; }
LBM13_HD constexpr size_t res_exchange_bytes(int nx, int ny, int elem)
{
    return size_t(2) * res_units(elem) * 16 * size_t(nx) * size_t(ny);
}
constexpr int kResMaxK = 4;
constexpr int kResSmem = 222 * 1024;  // rows and edge links of one tile; the rest of 227 KB holds the arguments
constexpr int kResWidths = 3;
LBM13_HD constexpr int res_width(int i) { return i == 0 ? 24 : i == 1 ? 32 : 48; }

struct ResShape {
    int ex;      // columns of a shared row (0: the lattice is not stepped this way)
    int K;       // steps between exchanges
    int gx, gy;  // tiles
    int rows;    // shared rows, the two spare ones included
    int threads; // of a block
    int edges;   // room for this many edge nodes' links, a multiple of 32
};

// Shared memory: the rows; for the edge nodes the values of their links
// [13][edges]; the states of the four walls by column or row of the array; the
// links resolved [13][edges], and the edge nodes' places.
LBM13_HD constexpr int res_along(const ResShape &s) { return s.edges == 0 ? 0 : s.ex > s.rows ? s.ex : s.rows; }
LBM13_HD constexpr size_t res_smem(const ResShape &s, int elem)
{
    return size_t(s.rows) * Q * s.ex * elem + size_t(s.edges) * (Q * (elem + 4) + 4) +
           size_t(8) * res_along(s) * elem;
}
// a resolved link's source is a 16-bit index into the rows
static_assert(kResSmem / 4 < 65536, "shared rows indexed with 16 bits");

// Rows and columns of tile b of n tiles of an axis: first node of tile i is
// len * i / n, so tiles differ by one node at most.
LBM13_HD int res_edge(int len, int i, int n) { return int((long long)len * i / n); }

struct ResTile {
    int x0, x1, y0, y1;  // the tile's nodes
    int ox, oy;          // node in the shared array's column 0, row 0
    int ew, eh;          // columns and rows of the tile and the nodes around it
};

LBM13_HD ResTile res_tile(const ResShape &s, int nx, int ny, int b)
{
    const int bx = b % s.gx, by = b / s.gx;
    ResTile t;
    t.x0 = res_edge(nx, bx, s.gx);
    t.x1 = res_edge(nx, bx + 1, s.gx);
    t.y0 = res_edge(ny, by, s.gy);
    t.y1 = res_edge(ny, by + 1, s.gy);
    t.ox = t.x0 - 2 * s.K;
    t.oy = t.y0 - 2 * s.K;
    t.ew = t.x1 - t.x0 + 4 * s.K;
    t.eh = t.y1 - t.y0 + 4 * s.K;
    return t;
}

// The nodes stepped when r more nodes around the tile are still needed: the
// tile grown by r, cut at walls.  Nodes within two of a wall (edge nodes) are
// work items of their own, resolved link by link; the others pull from fixed
// offsets.
struct ResRegion {
    int xa, xb, ya, yb;
    int el, er;        // edge columns at the left and right end
    int elo, ehi;      // rows below elo and from ehi on are edge rows
    int wd;            // other columns
    unsigned magic;    // d / wd = (d * magic) >> 16 for d < 1024, wd <= 48
    int chunk, chunks;  // rows of one chunk (its items fit the block's threads), chunks
};

LBM13_HD ResRegion res_region(const ResTile &t, int nx, int ny, bool per_x, bool per_y, int r, int threads)
{
    ResRegion g;
    g.xa = t.x0 - r;
    g.xb = t.x1 + r;
    g.ya = t.y0 - r;
    g.yb = t.y1 + r;
    g.el = g.er = 0;
    g.elo = -(1 << 30);
    g.ehi = 1 << 30;
    if (!per_x) {
        g.xa = g.xa > 0 ? g.xa : 0;
        g.xb = g.xb < nx ? g.xb : nx;
        // the four columns next to the walls, as far as they are here
        const int l = (2 < g.xb ? 2 : g.xb) - g.xa, e = g.xb - (nx - 2 > g.xa ? nx - 2 : g.xa);
        g.el = l > 0 ? l : 0;
        g.er = e > 0 ? e : 0;
    }
    if (!per_y) {
        g.ya = g.ya > 0 ? g.ya : 0;
        g.yb = g.yb < ny ? g.yb : ny;
        g.elo = 2;
        g.ehi = ny - 2;
    }
    const int w = g.xb - g.xa;
    g.wd = w - g.el - g.er;
    g.magic = g.wd > 0 ? (65536u + unsigned(g.wd) - 1u) / unsigned(g.wd) : 0u;
    const bool edges = !per_x || !per_y;
    const int most = (threads - (edges ? 31 : 0)) / w;
    const int rows = g.yb - g.ya, least = (rows + most - 1) / most;
    g.chunk = (rows + least - 1) / least;
    g.chunks = (rows + g.chunk - 1) / g.chunk;
    return g;
}

// Item i of the rows [ca, cb) of a region: its node, and whether it is an edge
// node; false when there is none.  Edge nodes come first and fill whole warps.
LBM13_HD bool res_item(const ResRegion &g, int ca, int cb, int i, int &x, int &y, bool &edge)
{
    const int rows = cb - ca;
    if (g.el + g.er == 0 && ca >= g.elo && cb <= g.ehi) {  // no edge nodes
        const int r = int((unsigned(i) * g.magic) >> 16);
        edge = false;
        x = g.xa + i - r * g.wd;
        y = ca + r;
        return r < rows;
    }
    const int w = g.xb - g.xa;
    int nb = g.elo - ca, nt = cb - g.ehi;  // edge rows at the low and high end
    nb = nb < 0 ? 0 : nb > rows ? rows : nb;
    nt = nt < 0 ? 0 : nt > rows - nb ? rows - nb : nt;
    const int ec = g.el + g.er, mid = rows - nb - nt, ym = ca + nb;
    const int ne = (nb + nt) * w + mid * ec, pad = (ne + 31) & ~31;
    edge = i < pad;
    if (edge) {
        if (i >= ne) return false;
        if (i < (nb + nt) * w) {
            const int r = i / w;
            x = g.xa + i - r * w;
            y = r < nb ? ca + r : ym + mid + r - nb;
            return true;
        }
        const int k = i - (nb + nt) * w, r = k / ec, c = k - r * ec;
        x = c < g.el ? g.xa + c : g.xb - g.er + c - g.el;
        y = ym + r;
        return true;
    }
    const int d = i - pad;
    if (d >= mid * g.wd) return false;
    const int r = int((unsigned(d) * g.magic) >> 16);
    x = g.xa + g.el + d - r * g.wd;
    y = ym + r;
    return true;
}

// Edge nodes of a region (the largest one of a tile holds those of the others),
// and the number of the edge node at (x, y).
LBM13_HD int res_edge_rows(const ResRegion &g, int &low)
{
    const int rows = g.yb - g.ya;
    int nb = g.elo - g.ya, nt = g.yb - g.ehi;
    nb = nb < 0 ? 0 : nb > rows ? rows : nb;
    nt = nt < 0 ? 0 : nt > rows - nb ? rows - nb : nt;
    low = nb;
    return nb + nt;
}
LBM13_HD int res_edge_count(const ResRegion &g)
{
    int low;
    const int er = res_edge_rows(g, low);
    return er * (g.xb - g.xa) + (g.yb - g.ya - er) * (g.el + g.er);
}
LBM13_HD int res_edge_index(const ResRegion &g, int x, int y)
{
    int low;
    const int er = res_edge_rows(g, low), w = g.xb - g.xa, mid = g.yb - g.ya - er;
    const int r = y - g.ya;
    if (r < low) return r * w + x - g.xa;
    if (r >= low + mid) return (r - mid) * w + x - g.xa;
    const int c = x - g.xa < g.el ? x - g.xa : x - g.xb + g.er + g.el;
    return er * w + (r - low) * (g.el + g.er) + c;
}

// Node i of the nodes around the tile (those of the shared array outside it):
// the rows below and above, then the columns left and right; lattice
// coordinates, not wrapped.
LBM13_HD int res_halo_count(const ResTile &t) { return t.ew * t.eh - (t.x1 - t.x0) * (t.y1 - t.y0); }
LBM13_HD void res_halo_node(const ResTile &t, int K, int i, int &x, int &y)
{
    const int band = 2 * K * t.ew;
    if (i < 2 * band) {
        const int r = i / t.ew;
        x = t.ox + i - r * t.ew;
        y = r < 2 * K ? t.oy + r : t.y1 + r - 2 * K;
        return;
    }
    const int k = i - 2 * band, r = k / (4 * K), c = k - r * 4 * K;
    x = c < 2 * K ? t.ox + c : t.x1 + c - 2 * K;
    y = t.y0 + r;
}

// Every split of an nx x ny lattice into `tiles` tiles or fewer that fits the SMs'
// shared memory (rows of `width` columns, or of any where that is 0), with the
// estimated clocks of a step: each(shape, clocks).
template <typename F>
inline void res_splits(int nx, int ny, bool per_x, bool per_y, int elem, int tiles, int width, F each)
{
    for (int i = 0; i < kResWidths; ++i)
        for (int K = 1; K <= kResMaxK; ++K) {
            const int ex = res_width(i), wide = ex - 4 * K, most_rows = kResSmem / (Q * ex * elem) - 2 - 4 * K;
            if (wide < 2 * K || most_rows < 2 * K || (width && ex != width)) continue;
            const int gx = (nx + wide - 1) / wide;
            if (gx > tiles || (gx > 1 && nx / gx < 2 * K)) continue;
            for (int gy = (ny + most_rows - 1) / most_rows; gy <= tiles / gx; ++gy) {
                if (gy > 1 && ny / gy < 2 * K) break;
                // the largest tile's time per step, in clocks
                const int w = (nx + gx - 1) / gx, h = (ny + gy - 1) / gy;
                ResShape s{ex, K, gx, gy, h + 4 * K + 2, 0, 0};
                // as many threads as the largest region has nodes, if so many may be
                const int largest = (w + 4 * (K - 1)) * (h + 4 * (K - 1)) + 31;
                s.threads = largest < 256 ? 256 : largest < res_threads(elem) ? largest & ~31 : res_threads(elem);
                // edge rows and columns of one tile: of one wall, or of both
                const int er = per_y ? 0 : gy == 1 || h + 4 * K >= ny - 2 ? 4 : 2;
                const int ec = per_x ? 0 : gx == 1 || w + 4 * K >= nx - 2 ? 4 : 2;
                s.edges = (er * (w + 4 * K) + ec * (h + 4 * K) + 31) & ~31;
                if (res_smem(s, elem) > size_t(kResSmem)) continue;
                const ResTile t{0, w, 0, h, -2 * K, -2 * K, w + 4 * K, h + 4 * K};
                // fitted to 865 measured splits of 64^2 .. 512^2 lattices (8% rms): an
                // exchange, the nodes around the tile, a chunk (two barriers and one
                // node's chain) and its nodes
                double clocks = elem == 4 ? 2500.0 + 3.2 * res_halo_count(t) : 3900.0;
                for (int k = 0; k < K; ++k) {
                    const ResRegion g = res_region(t, 1 << 28, 1 << 28, true, true, 2 * k, s.threads);
                    const double nodes = double(g.xb - g.xa) * (g.yb - g.ya);
                    clocks += elem == 4 ? 330.0 * g.chunks + 3.1 * nodes : 1840.0 * g.chunks + 16.0 * nodes;
                }
                each(s, clocks / K);
            }
        }
}

// The split of an nx x ny lattice for `sms` SMs and populations of elem bytes:
// the one with the smallest estimated time of a step, or ex = 0 where no split
// fits the SMs' shared memory.
inline ResShape res_shape(int nx, int ny, bool per_x, bool per_y, int elem, int sms)
{
    ResShape best{0, 0, 0, 0, 0, 0, 0};
    double best_t = 1e300;
    res_splits(nx, ny, per_x, per_y, elem, sms < kResMaxTiles ? sms : kResMaxTiles, 0, [&](const ResShape &s, double t) {
        if (t < best_t) {
            best_t = t;
            best = s;
        }
    });
    return best;
}

// The splits of many lattices that share the SMs: every lattice starts with the
// fewest tiles that hold it, and the one with the longest step takes more as long
// as there are SMs for them.  One width of the shared rows for all.  Returns the
// longest step in clocks and the shapes in out, or 0 where they do not fit.
struct ResLattice {
    int nx, ny;
    bool per_x, per_y;
};
inline double res_plan_shapes(const std::vector<ResLattice> &lats, int elem, int sms, int width,
                              std::vector<ResShape> &out)
{
    const int tiles = sms < kResMaxTiles ? sms : kResMaxTiles, count = int(lats.size());
    out.clear();
    if (count > tiles) return 0.0;
    struct Split {
        ResShape s;
        double t;
    };
    // by lattice, the best split into n + 1 tiles or fewer (equal lattices share one)
    std::vector<std::vector<Split>> by;
    std::vector<int> which(count), n(count, 0);
    int used = 0;
    for (int i = 0; i < count; ++i) {
        const ResLattice &l = lats[i];
        int k = 0;
        while (k < i && !(lats[k].nx == l.nx && lats[k].ny == l.ny && lats[k].per_x == l.per_x && lats[k].per_y == l.per_y))
            ++k;
        if (k < i) {
            which[i] = which[k];
        } else {
            which[i] = int(by.size());
            std::vector<Split> v(size_t(tiles), Split{ResShape{0, 0, 0, 0, 0, 0, 0}, 1e300});
            res_splits(l.nx, l.ny, l.per_x, l.per_y, elem, tiles, width, [&](const ResShape &s, double t) {
                Split &w = v[size_t(s.gx * s.gy - 1)];
                if (t < w.t) w = Split{s, t};
            });
            for (int m = 1; m < tiles; ++m)
                if (!(v[m].t < v[m - 1].t)) v[m] = v[m - 1];
            by.push_back(v);
        }
        const std::vector<Split> &v = by[which[i]];
        while (n[i] < tiles && v[n[i]].s.ex == 0) ++n[i];
        if (n[i] == tiles) return 0.0;
        used += n[i] + 1;
        if (used > tiles) return 0.0;
    }
    for (;;) {
        int slow = 0;
        for (int i = 1; i < count; ++i)
            if (by[which[i]][n[i]].t > by[which[slow]][n[slow]].t) slow = i;
        const std::vector<Split> &v = by[which[slow]];
        int m = n[slow] + 1;
        while (m < tiles && !(v[m].t < v[n[slow]].t)) ++m;
        if (m == tiles || used + m - n[slow] > tiles) {
            for (int i = 0; i < count; ++i) out.push_back(by[which[i]][n[i]].s);
            return v[n[slow]].t;
        }
        used += m - n[slow];
        n[slow] = m;
    }
}

// nsteps steps from a.fin (the state) in one cooperative launch; the new state is
// in a.fout, or after an even number of steps in a.fin again: the buffers end up as
// after single steps, also for a captured graph that holds them.  A block reads
// a.fin once, before its first exchange, and writes its tile after it has seen the
// first exchange of every block that reads nodes of that tile.  xchg: res_exchange_bytes bytes, zeroed once; the launch's exchanges
// are numbered tag + 1, tag + 2, ... (res_exchanges of them), which must not have
// been used before.  A wait that runs out (timeout_ns) sets *err, and the block
// leaves without writing.  absent: that many tiles, the last ones, are not launched,
// so that the waits for them run out (a self-check).
// Steps between two exchanges of a launch: at least one exchange for two steps or more.
LBM13_HD constexpr int res_between(int K, int nsteps) { return nsteps > K ? K : (nsteps + 1) / 2; }
LBM13_HD constexpr int res_exchanges(int K, int nsteps)
{
    return (nsteps + res_between(K, nsteps) - 1) / res_between(K, nsteps) - 1;
}
template <typename T, typename C>
cudaError_t launch_resident(const StepArgs<T, C> &a, bool force, int nsteps, const ResShape &s, void *xchg,
                            unsigned tag, unsigned *err, unsigned long long timeout_ns, cudaStream_t stream,
                            int absent = 0);

// Blocks of such a launch that the SMs hold at once (0 where it cannot be launched).
template <typename T, typename C>
int resident_capacity(const ResShape &s, bool force, const WallArgs<C> *wall);

// The same for the lattices of a plan, block i stepping tile[i].  All shapes have
// rows of `ex` columns (kResPlanWidths); xchg holds the lattices' exchange buffers
// at their offsets.  states: evaluate the walls' states once a step
// (res_states_pass of any of the lattices).
// A tile may take an SM's registers and shared memory whole, and a launch lasts up to
// 1024 steps: with a tile on every SM, kernels of other streams wait for its end (a
// server's admission beside a round of 24 solves, a new 128^2 lattice set and read once,
// took 3.5 ms instead of 0.45).  A plan leaves kResFree SMs to them where the split that
// does is at most kResShare times as slow by the estimate: 0.65 ms; the round 5% longer.
// One lattice does not: a 256^2 cavity would be 9 to 15% slower.
constexpr int kResFree = 4;
constexpr double kResShare = 1.05;
struct ResPlanTile {
    ResShape s;
    int lattice, tile;
    long long offset;  // of the lattice's exchange buffer, bytes
};
constexpr int kResPlanWidths[2] = {32, 48};
// Where walls of both axes need data, the tile in their corner resolves links that
// need two states each: microseconds a step with the states by link and in a pass
// of their own, 187 x 211 box FP32 3.84 and 3.03, FP64 11.9 and 7.8.  Walls of one
// axis, 256^2 cavity FP32: zero flux (three loads a state) 2.34 and 2.56,
// extrapolated density (26 loads) 2.70 and 2.82: the pass costs a barrier.
template <typename C>
bool res_states_pass(const WallArgs<C> *wall)
{
    return (wall[WEST].needs_data || wall[EAST].needs_data) && (wall[SOUTH].needs_data || wall[NORTH].needs_data);
}
int resident_plan_capacity(int ex, int threads, size_t smem, bool states);
cudaError_t launch_resident_plan(const BatchDesc<float, float> *descs, const ResPlanTile *tiles, int ntiles, int ex,
                                 int threads, size_t smem, bool states, int parity, int nsteps, void *xchg,
                                 unsigned tag, unsigned *err, unsigned long long timeout_ns, cudaStream_t stream);

}  // namespace lbm13
