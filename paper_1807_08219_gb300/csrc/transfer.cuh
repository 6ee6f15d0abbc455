// transfer.cuh -- node binning, spreading S* and interpolation S
// (Sec. "Interpolation Scheme"; Algorithm steps 2 and 4), and the FP64
// conservation sums.
//
// Binning. Every node is assigned the cell c = floor(x n/L) of its box. For
// both kernels and all three MAC lattices its stencil lies inside cells
// c-2 .. c+2 per axis. Boxes are cut into tiles, so large that a stencil meets at
// most two of them per axis.
// FP32: tiles of 4 to 16 cells a side and own lists: for every tile, the nodes whose
// cell lies in it. A tile's own nodes are spread and interpolated in shared boxes of
// the tile and its halo, which are added to the grid (transfer_tile_kernel; in a
// fixed order where the spread is reproducible, tile_combine_kernel).
// FP64: tiles of 5 cells or more (the last per axis up to t + 4) and candidate
// lists: for every tile, the nodes whose stencil meets it, by node number. Spreading
// is owner-computes: every value is accumulated by one thread at a time in the order
// of the nodes and written once, without atomics. Interpolation gathers per node.
#pragma once
#include <type_traits>

#include "common.cuh"

namespace ifem {

struct TileInfo {
    int box;
    int start[3];
    int edge[3];
};

__device__ inline int box_of_tile(const DevGrid &g, long long tile)
{
    int lo = 0, hi = g.n_boxes - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (g.boxes[mid].tile_base <= tile)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

__device__ inline TileInfo decode_tile(const DevGrid &g, long long tile)
{
    TileInfo ti;
    ti.box = box_of_tile(g, tile);
    const BoxDev &B = g.boxes[ti.box];
    long long local = tile - B.tile_base;
    int j[3] = {(int)(local % B.T), (int)((local / B.T) % B.T), (int)(local / ((long long)B.T * B.T))};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        ti.start[a] = tile_start(j[a], B.t);
        ti.edge[a] = tile_edge(j[a], B.t, B.T, B.n);
    }
    return ti;
}

__device__ __forceinline__ float mac_off(int d, int a) { return a == d ? 0.f : 0.5f; }

// ---------------------------------------------------------------- binning
// Cell of a node from its coordinates xa (all finite: true, else the cell is
// zero from the first non-finite axis on); s receives the lattice coordinates.
template <typename real>
__device__ inline bool node_cell_xyz(const InstDev &I, const BoxDev &B, const real xa[3], int c[3], real s[3])
{
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        ok = ok && isfinite(xa[a]);
        int I0;
        s[a] = LatCoord<real>::get(I, B, a, xa[a], real(0), I0);
        if constexpr (std::is_same<real, float>::value) {
            // 32-bit integer arithmetic while the cell is within 2^30 of the
            // particle's origin cell (every node near its box): with 64-bit
            // arithmetic for the cell and the own-list key the FP64 pipe was
            // 40 % busy in the binning pass
            const float fl = floorf(s[a]);
            if (fabsf(fl) < 1073741824.f && I0 > -1073741824 && I0 < 1073741824) {
                const int ci = I0 + (int)fl;
                int cw;
                if (ci >= 0 && ci < 2 * B.n) {
                    cw = ci >= B.n ? ci - B.n : ci;
                } else {
                    cw = ci % B.n;
                    cw += cw < 0 ? B.n : 0;
                }
                c[a] = ok ? cw : 0;
                continue;
            }
        }
        long long ci = (long long)I0 + (long long)floor(s[a]);
        int cw;
        if (ci >= 0 && ci < 2LL * B.n)
            cw = ci >= B.n ? (int)ci - B.n : (int)ci;
        else
            cw = wrapi(ci, B.n);
        c[a] = ok ? cw : 0;
    }
    return ok;
}

template <typename real>
__device__ inline bool node_cell(const InstDev &I, const BoxDev &B, const real *x, long long N, int node,
                                 int c[3])
{
    const real xa[3] = {x[node], x[N + node], x[2 * N + node]};
    real s[3];
    return node_cell_xyz<real>(I, B, xa, c, s);
}

// Own-list key of a cell: (tile, 4^3 sub-block of the tile). Nodes come out
// of the binning grouped by position, which keeps the gathers of
// neighbouring lanes on shared cache lines.
// 32-bit: the workspace holds fewer than 2^31 - 1 keys (n_tiles * kOwnSub3,
// checked when it is set up). r receives the cell within its tile.
__device__ __forceinline__ int own_key(const BoxDev &B, const int c[3], int r[3])
{
    int o[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        o[a] = tile_of(c[a], B.t, B.T);
        r[a] = c[a] - tile_start(o[a], B.t);
    }
    return ((int)B.tile_base + (o[2] * B.T + o[1]) * B.T + o[0]) * kOwnSub3 +
           ((r[2] >> 2) * kOwnSub + (r[1] >> 2)) * kOwnSub + (r[0] >> 2);
}

// Warp-aggregated list append: lanes with the same tile share one global
// atomic (count pass: the count; fill pass: the slot range). Every lane of
// the warp must call this (invalid lanes pass valid = false).
template <bool FILL>
__device__ __forceinline__ int agg_append(int *count, int *cursor, int *list, long long tile, bool valid,
                                           int node)
{
    const unsigned key = valid ? (unsigned)tile : 0xffffffffu;
    const unsigned grp = __match_any_sync(0xffffffffu, key);
    if (!valid)
        return -1;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(grp) - 1;
    if (!FILL) {
        if (lane == leader)
            atomicAdd(&count[tile], __popc(grp));
        return -1;
    }
    int base = 0;
    if (lane == leader)
        base = atomicAdd(&cursor[tile], __popc(grp));
    base = __shfl_sync(grp, base, leader);
    const int slot = base + __popc(grp & ((1u << lane) - 1u));
    list[slot] = node;
    return slot;
}

// Programmatic dependent launch: a kernel launched so (launch_after) may start
// once every CTA of the one before it has triggered, and waits for that one's end
// and its stores before it reads them. Without the attribute both do nothing.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Clears a binning's counters and counts, and the field to be spread into where
// that is small (a kernel, not a memset, for own_count_kernel to follow without a
// gap).
static __global__ void __launch_bounds__(256) clear_kernel(int *__restrict__ p, size_t words, int *__restrict__ f,
                                                           size_t f_words)
{
    pdl_trigger();
    for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < words; i += (size_t)gridDim.x * 256)
        p[i] = 0;
    for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < f_words; i += (size_t)gridDim.x * 256)
        f[i] = 0;
}

// A node's lattice coordinate f0 + x n/L from the cell that begins at fl, with what
// the coordinate itself, tens of cells, rounds off: that was most of the error of the
// interpolation. A little outside [0, 1) where the rounded coordinate is in the next
// cell: stencils from there are the same to second order, and within the boxes up to
// the limits set here (coordinates of 1e5 cells and more).
__device__ __forceinline__ float node_frac(float f0, float x, const BoxDev &B, float fl)
{
    const float p = __fmul_rn(x, B.inv_h_f), pe = fmaf(x, B.inv_h_lo, fmaf(x, B.inv_h_f, -p));
    float e;
    const float s = two_sum(f0, p, e);
    return fminf(fmaxf((s - fl) + (e + pe), -0.015625f), 1.015625f);
}

// One-pass own-list binning (FP32): per node its rank within its
// own-list key (the old value of the key's count, one atomic per group of
// lanes with the same key) and its record -- fractional lattice coordinates
// and cell within the tile, 8-bit x | y << 8 | z << 16 -- kept by node for
// own_scatter_kernel; the leader of each group also marks the key's tile as
// owning nodes. Nodes that are not finite or not in the box get the key -1
// and are counted in ST_DOMAIN. kBinPer nodes per thread, node
// (blockIdx.x * kBinPer + j) * blockDim.x + threadIdx.x of instance
// blockIdx.y, each phase's loads, atomics and stores issued for all of them
// before their results are used: with one node per thread the pass is a
// chain of dependent latencies.
constexpr int kBinPer = 4;
static __global__ void __launch_bounds__(256) own_count_kernel(DevBatch b, DevGrid g, DevWork w, const float *__restrict__ x)
{
    pdl_trigger();
    const InstDev I = b.inst[blockIdx.y];
    const BoxDev B = g.boxes[I.box];
    const long long N = b.N;
    const int lane = threadIdx.x & 31;
    int node[kBinPer];
    bool in[kBinPer];
    float xa[kBinPer][3];
#pragma unroll
    for (int j = 0; j < kBinPer; ++j) {
        const int k = (blockIdx.x * kBinPer + j) * blockDim.x + threadIdx.x;
        in[j] = k < I.n_nodes;
        node[j] = I.node_off + (in[j] ? k : 0);
        xa[j][0] = xa[j][1] = xa[j][2] = 0.f;
        if (in[j]) {
            xa[j][0] = x[node[j]];
            xa[j][1] = x[N + node[j]];
            xa[j][2] = x[2 * N + node[j]];
        }
    }
    pdl_wait();   // for the clearing (which began after the positions were there)
    bool ok[kBinPer];
    int key[kBinPer];
#pragma unroll
    for (int j = 0; j < kBinPer; ++j) {
        int c[3] = {0, 0, 0};
        float sl[3];
        ok[j] = in[j] && node_cell_xyz<float>(I, B, xa[j], c, sl);
        if (in[j] && !ok[j])
            status_add(w.status, ST_DOMAIN, 1);
        int r[3];
        key[j] = own_key(B, c, r);
        if (ok[j]) {
            const unsigned pk = (unsigned)r[0] | ((unsigned)r[1] << 8) | ((unsigned)r[2] << 16);
            float fr[3];
#pragma unroll
            for (int a = 0; a < 3; ++a)
                fr[a] = node_frac(I.f0[a], xa[j][a], B, floorf(sl[a]));
            w.node_rec[node[j]] = make_float4(fr[0], fr[1], fr[2], __uint_as_float(pk));
        }
    }
    // every lane takes part in the votes and shuffles (invalid lanes form
    // their own group under the key 0xffffffff, which no valid key reaches)
    unsigned grp[kBinPer];
    int base[kBinPer];
#pragma unroll
    for (int j = 0; j < kBinPer; ++j) {
        grp[j] = __match_any_sync(0xffffffffu, ok[j] ? (unsigned)key[j] : 0xffffffffu);
        base[j] = 0;
        if (ok[j] && lane == __ffs(grp[j]) - 1) {
            base[j] = atomicAdd(&w.own_count[key[j]], __popc(grp[j]));
            w.own_flag[key[j] / kOwnSub3] = 1;
        }
    }
#pragma unroll
    for (int j = 0; j < kBinPer; ++j) {
        const int rank = __shfl_sync(0xffffffffu, base[j], __ffs(grp[j]) - 1) + __popc(grp[j] & ((1u << lane) - 1u));
        if (in[j])
            w.node_key[node[j]] = make_int2(ok[j] ? key[j] : -1, rank);
    }
}

// FILL = false: count candidate pairs per tile; FILL = true: write them
// (FP64; FP32 bins with own_count_kernel and own_scatter_kernel). Block size
// must be a multiple of 32 (every lane reaches the warp votes).
template <typename real, bool FILL>
__global__ void bin_kernel(DevBatch b, DevGrid g, DevWork w, const real *__restrict__ x)
{
    const InstDev I = b.inst[blockIdx.y];
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = k < I.n_nodes;
    const BoxDev B = g.boxes[I.box];
    const int node = I.node_off + (in ? k : 0);
    int c[3] = {0, 0, 0};
    bool ok = false;
    if (in) {
        ok = node_cell<real>(I, B, x, b.N, node, c);
        if (!FILL && !ok)
            status_add(w.status, ST_DOMAIN, 1);
    }
    int tl[3][2], nt[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        int lo = c[a] - 2, hi = c[a] + 2;
        lo += lo < 0 ? B.n : 0;
        hi -= hi >= B.n ? B.n : 0;
        tl[a][0] = tile_of(lo, B.t, B.T);
        tl[a][1] = tile_of(hi, B.t, B.T);
        nt[a] = tl[a][0] == tl[a][1] ? 1 : 2;
    }
#pragma unroll
    for (int slot = 0; slot < 8; ++slot) {
        const int ix = slot & 1, iy = (slot >> 1) & 1, iz = slot >> 2;
        const bool valid = ok && ix < nt[0] && iy < nt[1] && iz < nt[2];
        if (!__any_sync(0xffffffffu, valid))
            continue;   // most nodes meet one or two tiles: skip empty slots warp-wide
        const long long tile = B.tile_base + ((long long)tl[2][iz] * B.T + tl[1][iy]) * B.T + tl[0][ix];
        agg_append<FILL>(w.cand_count, w.cand_cursor, w.cand_nodes, tile, valid, node);
    }
}

// Exclusive scan of the counts (FP32: per own sub-block, FP64: candidates per
// tile): block-local scan, whose last block to finish scans the block sums -> add +
// cursors + active lists (scan_finish_kernel, FP64; in FP32 own_scatter_kernel adds
// the block offsets itself).

__device__ inline int block_exclusive_scan(int v, int *sh, int &total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o)
            incl += t;
    }
    if (lane == 31)
        sh[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        int s = lane < nw ? sh[lane] : 0;
        int si = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, si, o);
            if (lane >= o)
                si += t;
        }
        if (lane < nw)
            sh[lane] = si - s;
        if (lane == nw - 1)
            sh[32] = si;
    }
    __syncthreads();
    int r = sh[wid] + incl - v;
    total = sh[32];
    __syncthreads();
    return r;
}

static __global__ void scan_local_kernel(long long n, const int *__restrict__ count, int *__restrict__ off,
                                         int *__restrict__ bsum, int *__restrict__ ticket, int *__restrict__ total)
{
    pdl_trigger();
    pdl_wait();
    __shared__ int sh[33];
    __shared__ int last;
    const long long base = (long long)blockIdx.x * kScanBlock + (long long)threadIdx.x * kScanPer;
    int v[kScanPer], s = 0;
#pragma unroll
    for (int q = 0; q < kScanPer; ++q) {
        v[q] = base + q < n ? count[base + q] : 0;
        s += v[q];
    }
    int t;
    int e = block_exclusive_scan(s, sh, t);
#pragma unroll
    for (int q = 0; q < kScanPer; ++q) {
        if (base + q < n)
            off[base + q] = e;
        e += v[q];
    }
    // block sums out, then a ticket: the block that takes the last one sees
    // every block's sum (fence before the ticket, L2 loads after it)
    if (threadIdx.x == 0) {
        bsum[blockIdx.x] = t;
        __threadfence();
        last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last)
        return;
    __threadfence();
    const int nb = (int)gridDim.x;
    int run = 0;
    for (int b0 = 0; b0 < nb; b0 += blockDim.x) {
        const int i = b0 + threadIdx.x;
        const int u = i < nb ? __ldcg(&bsum[i]) : 0;
        int w;
        const int x = block_exclusive_scan(u, sh, w);
        if (i < nb)
            bsum[i] = x + run;
        run += w;
    }
    if (threadIdx.x == 0)
        *total = run;
}

// n tiles (candidate lists). Adds the block offsets, sets the fill cursors,
// writes the terminal offset and the lists of tiles with candidates, by class of their number, most first: a warp takes up to
// 0.1 us a candidate, so the few long lists of a dense spot, begun last, were
// the tail of the FP64 spread.
// Class 0, lists that several warps walk (spread_det_warp_kernel), begins at 0.6
// of the candidates that a quarter of an SM has to walk in all: a unit longer
// than that would be the spread's length.
__device__ __forceinline__ int tile_class(int count, int limit)
{
    return count >= limit ? 0 : (2 * count >= limit ? 1 : (4 * count >= limit ? 2 : 3));
}
struct ActiveTiles {
    int count[kTileClasses], total;
    __device__ explicit ActiveTiles(const DevWork &w) : total(0)
    {
#pragma unroll
        for (int k = 0; k < kTileClasses; ++k)
            total += count[k] = w.counters[10 + k];
    }
    __device__ int tile(const DevGrid &g, const DevWork &w, int i) const
    {
        const int *list = w.active;
#pragma unroll
        for (int k = 0; k < kTileClasses - 1; ++k)
            if (i >= count[k]) {
                i -= count[k];
                list += g.n_tiles;
            } else {
                break;
            }
        return list[i];
    }
};
static __global__ void scan_finish_kernel(long long n, DevWork w, int n_sm)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i > n)
        return;
    int c1 = 0;
    if (i == n) {
        w.cand_off[n] = w.counters[4];
    } else {
        c1 = w.cand_count[i];
        const int o1 = w.cand_off[i] + w.scan_blocks[i / kScanBlock];
        w.cand_off[i] = o1;
        w.cand_cursor[i] = o1;
    }
    const unsigned act = __activemask();
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(act) - 1;
    const int limit = max(256, (int)(9LL * w.counters[4] / (20 * n_sm)));   // 3 lattices, 4 quarters
#pragma unroll
    for (int k = 0; k < kTileClasses; ++k) {
        const unsigned m = __ballot_sync(act, c1 > 0 && tile_class(c1, limit) == k);
        int at = 0;
        if (lane == leader && m)
            at = atomicAdd(&w.counters[10 + k], __popc(m));
        at = __shfl_sync(act, at, leader);
        if (m >> lane & 1u)
            w.active[k * n + at + __popc(m & ((1u << lane) - 1u))] = (int)i;
    }
}

// Deterministic mode: sort each tile's candidate list by node id (bitonic
// sort in shared memory). Lists longer than kSortCap are flagged.
constexpr int kSortCap = 4096;
static __global__ void sort_segments_kernel(DevGrid g, DevWork w)
{
    __shared__ int key[kSortCap];
    const ActiveTiles active(w);
    for (int it = blockIdx.x; it < active.total; it += gridDim.x) {
        const int tile = active.tile(g, w, it);
        const int beg = w.cand_off[tile], len = w.cand_off[tile + 1] - beg;
        if (len > kSortCap) {
            if (threadIdx.x == 0)
                status_add(w.status, ST_CAPACITY, 1);
            continue;
        }
        int P = 1;
        while (P < len)
            P <<= 1;
        for (int i = threadIdx.x; i < P; i += blockDim.x)
            key[i] = i < len ? w.cand_nodes[beg + i] : 0x7fffffff;
        __syncthreads();
        for (int k = 2; k <= P; k <<= 1)
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int i = threadIdx.x; i < P; i += blockDim.x) {
                    int l = i ^ j;
                    if (l > i) {
                        int a = key[i], bb = key[l];
                        bool up = (i & k) == 0;
                        if ((a > bb) == up) {
                            key[i] = bb;
                            key[l] = a;
                        }
                    }
                }
                __syncthreads();
            }
        for (int i = threadIdx.x; i < len; i += blockDim.x)
            w.cand_nodes[beg + i] = key[i];
        __syncthreads();
    }
}

// --------------------------------------------------------- stencil per axis
// Peskin: i0 = floor(s) - 1 (relative to I0), phi[m] = phi4(s - (i0 + m)).
template <typename real>
__device__ __forceinline__ long long peskin_axis(real s, real ph[4])
{
    long long i0 = (long long)floor(s) - 1;
#pragma unroll
    for (int m = 0; m < 4; ++m)
        ph[m] = phi4<real>(s - (real)(i0 + m));
    return i0;
}

// FP64 Peskin stencils of every node, thread per (node, axis): the weights of
// the two offsets that the lattices have along the axis (the same expressions as
// the gather and the spread, same compilation), bit for bit. Bound by the FP64
// pipe: 24 weights a node, where the three lattices' nine axes took 36 (133 k
// nodes 230 us, 135 now). Non-finite nodes are never binned and never read.
static __global__ void det_weights_kernel(DevBatch b, DevGrid g, DetW *__restrict__ wt, const double *__restrict__ x)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long N = b.N;
    if (t >= 3 * N)
        return;
    const int a = (int)(t / N);
    const long long node = t - a * N;
    const InstDev &I = b.inst[b.node_inst[node]];
    const BoxDev &B = g.boxes[I.box];
    const double xa = x[t];
    if (!isfinite(xa))
        return;
    DetW &W = wt[node];
#pragma unroll
    for (int o = 0; o < 2; ++o) {
        int I0;
        double ph[4];
        W.base[a][o] = wrapi(peskin_axis<double>(LatCoord<double>::get(I, B, a, xa, o ? 0.5 : 0.0, I0), ph), B.n);
#pragma unroll
        for (int m = 0; m < 4; ++m)
            W.ph[a][o][m] = ph[m];
    }
}

// Per-thread partial sums as unevaluated float pairs (hi + lo, Knuth's
// TwoSum and the FMA product error): about 44 significant bits, at FP32
// speed; the FP64 pipe of this GPU is far narrower than its FP32 pipe.
struct DF {
    float hi, lo;
};
__device__ __forceinline__ void df_add(DF &x, float v)
{
    const float s = x.hi + v;
    const float bv = s - x.hi;
    const float e = (x.hi - (s - bv)) + (v - bv);
    const float t = x.lo + e;
    x.hi = s + t;
    x.lo = t - (x.hi - s);
}
// x += y for two float pairs, with both the high and the low sums made exact
// by TwoSum before renormalising (relative error a few 2^-48).
__device__ __forceinline__ void df_add_df(DF &x, DF y)
{
    const float s = x.hi + y.hi;
    const float bs = s - x.hi;
    float e = (x.hi - (s - bs)) + (y.hi - bs);
    const float t = x.lo + y.lo;
    const float bt = t - x.lo;
    const float f = (x.lo - (t - bt)) + (y.lo - bt);
    e += t;
    const float h = s + e;
    e = (e - (h - s)) + f;
    x.hi = h + e;
    x.lo = e - (x.hi - h);
}
__device__ __forceinline__ void df_add_prod(DF &x, float a, float b)
{
    const float p = a * b;
    const float pe = fmaf(a, b, -p);
    df_add(x, p);
    x.lo += pe;
}

// The four Peskin weights of one axis share one square root: with
// r = s - floor(s) in [0, 1) and q = sqrt(1 + 4r - 4r^2),
//   phi(1 + r) = (3 - 2r - q)/8, phi(r) = (3 - 2r + q)/8,
//   phi(1 - r) = (1 + 2r + q)/8, phi(2 - r) = (1 + 2r - q)/8
// (the radicands of both branches of phi reduce to the same 1 + 4r - 4r^2,
// which lies in [1, 2], so sqrt(t) = t * rsqrt(t) needs no special cases).
// The even and the odd weights each sum to 1/2: the larger one of a pair is rounded, the
// other is what it leaves of 1/2, exactly, so that the roundings of a pair cancel but for
// the difference of the field over two cells (velocities of 600 mixed cells against 64
// bits: relative error 6.5e-8 with each weight rounded for itself, 4.8e-8).
// PAIRED = false rounds each weight for itself: the cell-centred interpolation, for which
// the compiler keeps fewer loads in flight with the pairs (600 mixed cells, six
// components 538 us, 574).
// Used by the FP32 kernels; the FP64 kernels evaluate phi point by point.
template <bool PAIRED = true>
__device__ __forceinline__ void peskin_frac(float r, float ph[4])
{
    const float t = 1.f + 4.f * r - 4.f * r * r;   // in [1, 2] for r in [0, 1), at least 0.93 for node_frac's
    const float q = t * rsqrtf(t);
    if (!PAIRED) {
        ph[0] = (3.f - 2.f * r - q) * 0.125f;
        ph[1] = (3.f - 2.f * r + q) * 0.125f;
        ph[2] = (1.f + 2.f * r + q) * 0.125f;
        ph[3] = (1.f + 2.f * r - q) * 0.125f;
        return;
    }
    ph[2] = 0.5f - (3.f - 2.f * r - q) * 0.125f;
    ph[1] = 0.5f - (1.f + 2.f * r - q) * 0.125f;
    ph[0] = 0.5f - ph[2];
    ph[3] = 0.5f - ph[1];
}
__device__ __forceinline__ int peskin_axis_fast(float s, float ph[4])
{
    const float fl = floorf(s);
    peskin_frac<false>(s - fl, ph);
    return (int)fl - 1;
}

// Fire-and-forget adds performed at L2 (no value returned, so the SM does not
// wait for the line): the tile flush adds its sums to the grid this way.
__device__ __forceinline__ void red_add_v4(float *p, float a, float b, float c, float d)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(__cvta_generic_to_global(p)), "f"(a),
                 "f"(b), "f"(c), "f"(d)
                 : "memory");
}
__device__ __forceinline__ void red_add_v2(float *p, float a, float b)
{
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(__cvta_generic_to_global(p)), "f"(a), "f"(b)
                 : "memory");
}
__device__ __forceinline__ void red_add(float *p, float a)
{
    asm volatile("red.global.add.f32 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "f"(a) : "memory");
}

// n-periodic wrap of an index that is normally already in (-n, 2n)
__device__ __forceinline__ int wrap_near(int v, int n)
{
    if (v < 0)
        v += n;
    else if (v >= n)
        v -= n;
    if ((unsigned)v >= (unsigned)n)
        v = wrapi(v, n);
    return v;
}

// Periodic wrap of a box coordinate in [-n, 2n): the boxes of a grid have
// at least 8 cells and the halos at most 4, so one correction suffices.
__device__ __forceinline__ int wrap1(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// A sum of non-negative floats that does not depend on their order: 64-bit
// integers, one per 32 binades, in units of 2^(32 bin - 131), values rounded up
// to them (at most 2^-4 of a value at the low end of a bin; 2^27 of the largest
// values fit). A value that is not finite counts as the largest float.
__device__ __forceinline__ void fsum_add(unsigned long long *bins, float v)
{
    if (!(v <= 3.402823466e38f))
        v = 3.402823466e38f;
    if (v == 0.f)
        return;
    const int bin = __float_as_int(v) >> 28;   // exponent field / 32
    // the unit's reciprocal in two factors that are floats
    const float q = ceilf(v * __int_as_float((127 + 67 - 16 * bin) << 23) * __int_as_float((127 + 64 - 16 * bin) << 23));
    atomicAdd(bins + bin, (unsigned long long)q);
}
__device__ __forceinline__ float fsum_get(const unsigned long long *__restrict__ bins)
{
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < kFsumBins; ++k) {
        const unsigned long long q = bins[k];
        if (q)
            s += (double)q * __hiloint2double((1023 + 32 * k - 131) << 20, 0);
    }
    return (float)s;
}

// FP32, after the scan: every binned node goes to its slot (the
// scanned offset of its key plus its rank from own_count_kernel) as one
// 32-byte record: what own_count_kernel kept of it, its force (0 without F)
// and its id, kBinPer nodes per thread as in own_count_kernel (loads first,
// then the offsets, then the stores). With the force in the record the
// transfer reads its nodes in two consecutive 16-byte loads, without a gather
// through the node id. The tiles that own nodes are listed (tile_slot: a
// tile's place in the list, or -1; for a reproducible spread also the tiles that
// a box reaches, near_tile, counters[9] of them), counters[3] of them, with everything the
// transfer needs of a tile: it fetches an item in one copy, without walking
// empty tiles or decoding tile numbers. The list keeps roughly the tile order
// (in order within each warp's append), so items running at the same time are
// spatial neighbours whose velocity rows and grid lines share L2 (listing the
// largest tiles first measured slower).
// With the forces F given, the placement also sums |F_d| over each tile's
// own nodes into tile_fsum (zeroed with the counts): the transfer's
// fixed-point scale of item (tile, d) comes from that sum instead of a pass
// over the item's forces. Lanes of a warp hold consecutive nodes, so the
// tiles come in runs: a segmented shuffle scan sums each run and its last
// lane adds it with one atomic per lattice (the order of those atomics is
// not fixed; the transfer's bound allows for it).
// xn (a step with the position update, which the transfer writes for the nodes it
// visits): the update of nodes that are in no tile, as ab2_kernel does it. (In the
// transfer, which knows too, the test cost 0.8% of a step of 600 particles.)
// Grid: as own_count_kernel along x and y, at least n_tiles threads in all.
static __global__ void __launch_bounds__(256) own_scatter_kernel(DevBatch b, DevGrid g, DevWork w,
                                                                 const float *__restrict__ F, int det,
                                                                 const float *__restrict__ x, const float *__restrict__ v,
                                                                 const float *__restrict__ vp, float *__restrict__ xn,
                                                                 float dt)
{
    pdl_trigger();
    pdl_wait();   // for the scan
    const InstDev I = b.inst[blockIdx.y];
    const long long N = b.N;
    const int lane = threadIdx.x & 31;
    int node[kBinPer];
    int2 kr[kBinPer];
    float4 rec[kBinPer];
    float fa[kBinPer][3];
#pragma unroll
    for (int j = 0; j < kBinPer; ++j) {
        const int k = (blockIdx.x * kBinPer + j) * blockDim.x + threadIdx.x;
        node[j] = I.node_off + k;
        kr[j] = make_int2(-1, 0);
        fa[j][0] = fa[j][1] = fa[j][2] = 0.f;
        if (k < I.n_nodes) {
            kr[j] = w.node_key[node[j]];
            rec[j] = w.node_rec[node[j]];
            if (F) {
                fa[j][0] = F[node[j]];
                fa[j][1] = F[N + node[j]];
                fa[j][2] = F[2 * N + node[j]];
            }
            if (xn && kr[j].x < 0)
#pragma unroll 1
                for (int d = 0; d < 3; ++d) {
                    const long long i = d * N + node[j];
                    xn[i] = ab2_value(x[i], v[i], vp[i], dt);
                }
        }
    }
    int off[kBinPer];
#pragma unroll
    for (int j = 0; j < kBinPer; ++j)
        off[j] = kr[j].x >= 0 ? w.own_cursor[kr[j].x] + w.scan_blocks[kr[j].x / kScanBlock] : 0;
#pragma unroll
    for (int j = 0; j < kBinPer; ++j) {
        if (kr[j].x >= 0) {
            float4 *slot = w.own_rec + 2LL * (off[j] + kr[j].y);
            slot[0] = rec[j];
            slot[1] = make_float4(fa[j][0], fa[j][1], fa[j][2], __int_as_float(node[j]));
        }
    }
    if (F) {   // the same for every thread of the grid
#pragma unroll
        for (int j = 0; j < kBinPer; ++j) {
            const int tile = kr[j].x >= 0 ? kr[j].x / kOwnSub3 : -1;
            const int prev = __shfl_up_sync(0xffffffffu, tile, 1);
            const int next = __shfl_down_sync(0xffffffffu, tile, 1);
            const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || prev != tile);
            // first lane of this lane's run
            const int seg = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
#pragma unroll
            for (int d = 0; d < 3; ++d)
                fa[j][d] = fabsf(fa[j][d]);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const float t = __shfl_up_sync(0xffffffffu, fa[j][d], o);
                    if (lane - o >= seg)
                        fa[j][d] += t;
                }
            }
            if (tile >= 0 && (lane == 31 || next != tile)) {
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    if (det)
                        fsum_add(w.tile_fbin + kFsumBins * (3LL * tile + d), fa[j][d]);
                    else
                        atomicAdd(&w.tile_fsum[3LL * tile + d], fa[j][d]);
                }
            }
        }
    }
    const long long nthr = (long long)gridDim.x * gridDim.y * blockDim.x;
    const long long tid = ((long long)blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x;
    for (long long t0 = tid - lane; t0 < g.n_tiles; t0 += nthr) {   // warp-uniform bounds
        const long long t = t0 + lane;
        bool has = false;
        if (t < g.n_tiles) {
            has = w.own_flag[t] != 0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, has);
        int base = 0;
        if (lane == 0 && m)
            base = atomicAdd(&w.counters[3], __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        const int slot = base + __popc(m & ((1u << lane) - 1u));
        if (t < g.n_tiles)
            w.tile_slot[t] = has ? slot : -1;
        if (has) {
            const TileInfo ti = decode_tile(g, t);
            const BoxDev &B = g.boxes[ti.box];
            const long long i = t * kOwnSub3, j = i + kOwnSub3;
            TileDesc td;
            td.tile = (int)t;
            td.n = B.n;
            td.beg = w.own_cursor[i] + w.scan_blocks[i / kScanBlock];
            td.end = t + 1 < g.n_tiles ? w.own_cursor[j] + w.scan_blocks[j / kScanBlock] : w.counters[5];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                td.start[a] = ti.start[a];
                td.edge[a] = ti.edge[a];
            }
            td.grid_off = B.grid_off;
            td.h3 = B.h3;
            td.scale_f = B.scale_f;
            td.slot = slot;
            w.tile_desc[slot] = td;
        }
        if (det) {   // tiles reached by a box: those with nodes in them or in a neighbour
            bool near = false;
            int box = 0;
            if (t < g.n_tiles) {
                box = box_of_tile(g, t);
                const BoxDev &B = g.boxes[box];
                const int T = B.T, local = (int)(t - B.tile_base);
                const int jx = local % T, jy = (local / T) % T, jz = local / (T * T);
                int any = 0;
#pragma unroll
                for (int k = 0; k < 27; ++k)
                    any |= w.own_flag[B.tile_base + (wrap1(jz + k / 9 - 1, T) * T + wrap1(jy + k / 3 % 3 - 1, T)) * T +
                                      wrap1(jx + k % 3 - 1, T)];
                near = any != 0;
            }
            const unsigned mn = __ballot_sync(0xffffffffu, near);
            if (lane == 0 && mn)
                base = atomicAdd(&w.counters[9], __popc(mn));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (near)
                w.near_tile[base + __popc(mn & ((1u << lane) - 1u))] = make_int2((int)t, box);
        }
    }
}

// --------------------------------------- tile transfer, FP32, own nodes only
// Spreading, interpolation, or both fused (Algorithm steps 2 and 4 use the same
// stencil weights of the same positions), with the position update of Eq.
// Bashforth_eqn on request, for both kernels and scatter modes. Work
// item = (tile, lattice) over the tiles with own nodes (own_scatter_kernel),
// taken from a global counter. Each node is visited only by the tile that
// holds its cell. Boxes of shared memory cover the tile plus a halo, 2 cells
// in y and z and 4 in x (so that its 16-byte quads are quads of the grid),
// which holds every stencil point of every own node: U, the velocity values
// the item's stencils read, and A, the spread accumulator (int32 fixed point,
// scale from the bound sum_k |g_k| / 8 over the tile's own nodes, from the sum
// of |F_d| that the binning's placement keeps per tile; integer addition is
// associative, so a box does not depend on the order of its nodes).
//
// Two boxes of each kind, and two kinds of warps. While the node warps work on
// item i (one (node, lattice) unit per thread: the Peskin weights, v_d = sum
// phi u_d from U, 64 contributions added to A with shared-memory reductions),
// the box warps copy the velocities of item i + 1 into the other U (cp.async)
// and flush the other A, of item i - 1, and clear it. IFEM_SCATTER_ATOMIC with
// the Peskin kernel: every non-zero value is added to the grid with an L2
// reduction (the halos of neighbouring tiles combine there; the order of a
// value's terms across tiles is not fixed). Otherwise (STORE) only values whose
// terms have no order are added like that: on a cleared field those that at most
// two boxes reach, else (add) those that one does. The others go to a buffer, and
// tile_combine_kernel sums their terms in a fixed order and writes the sum or adds
// it, so that repeated runs give the same bits. One
// barrier per item. With the copy, the node loop and the flush one after the
// other, each waited out its own memory latency.
//
// Measured, 600-particle suspension (1.33 M nodes, 256^3, 16-cell tiles, fused):
// 291 us against 375 us for the kernel before it (one box of each kind, three
// CTAs of 128 threads per SM, stencils in z-y-x order, a status atomic per warp
// and item); 64 boxes of 32 to 96 cells 240 against 437 us. What bounds it now:
// instruction issue (51 %) and the shared-memory pipe (44 %) of an SM whose two
// kinds of warps wait for each other once per item; alone, the node loops take
// 174 us, the copies 172, the flushes' scans 121.
//
// The boxes store the cell (x, y, z) in bank (x & 3) | (z & 3) << 2 | (y & 1)
// << 4 of the 128-byte line (x >> 2, z >> 2, y >> 1). A unit's 4 x 4 x 4 points
// fall on every bank exactly twice, and each lane walks its points starting
// from its own bank: lane l takes, at step (t0, t1, t2), the point in bank
// ((l + t0) & 3) | ((l >> 2) + t1 & 3) << 2 | ((l >> 4) + t2 & 1) << 4, so the
// 32 lanes are on 32 different banks at every step wherever their nodes lie.
// (In plain z-y-x order the lanes' banks are random: 2.7 wavefronts per load
// and 3.4 per reduction on the 600-particle suspension, by a count over its
// stencils.) The Peskin weights are rotated into that order once per unit; the
// interpolation adds its terms in pairs that no rotation separates, so v does
// not depend on the lane.

// red.shared.add without a compiler memory clobber: for accumulators that
// no thread reads before the next barrier (the caller places a compiler
// fence before it).
__device__ __forceinline__ void red_shared_add_nc(unsigned a, int v)
{
    asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(a), "r"(v));
}

// Accumulator width of the spread: red_add of a value in fixed point at a byte offset
// of the box of 32-bit words, and the box's quads.
template <typename Acc>
struct TileAcc;
template <>
struct TileAcc<int> {
    using Quad = int4;
    static __device__ __forceinline__ void add(unsigned A, int off, float v)
    {
        red_shared_add_nc(A + (unsigned)off, __float2int_rn(v));
    }
    static __device__ __forceinline__ unsigned some(int q) { return min((unsigned)q, 1u); }
};
template <>
struct TileAcc<long long> {
    struct alignas(16) Quad {
        long long x, y, z, w;
    };
    static __device__ __forceinline__ void add(unsigned A, int off, float v)
    {
        asm volatile("red.shared.add.u64 [%0], %1;" ::"r"(A + 2u * (unsigned)off), "l"(__float2ll_rn(v)));
    }
    static __device__ __forceinline__ unsigned some(long long q) { return q != 0; }
};

__device__ __forceinline__ void cp_async16(unsigned dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(__cvta_generic_to_global(src))
                 : "memory");
}
__device__ __forceinline__ void cp_async4(unsigned dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(__cvta_generic_to_global(src))
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Work counter of a launch: the three lattices of each listed tile, in list
// order (lattice < 0, counters[2]), or lattice d of each listed tile
// (counters[1], [6], [7] for d = 0, 1, 2), so that one launch per lattice
// completes row d of v at its end.
__device__ __forceinline__ int *tile_counter(const DevWork &w, int lattice)
{
    return &w.counters[lattice < 0 ? 2 : (lattice == 0 ? 1 : (lattice == 1 ? 6 : 7))];
}

// Shapes by the width W = 20, 16, 12 of the boxes in y and z (tiles of at most
// 16, 12, 8 cells): lines per axis, node and box threads. A box thread keeps
// one (x >> 2, z, y & 1) and walks y in kYStep phases; two phases where that
// measured faster (64 boxes of odd sizes, 16-cell tiles: 243 against 284 us;
// 600 particles 292 against 291).
template <int W>
struct TileShape {
    static constexpr int NX = W / 4 + 1, NZ = W / 4, NY = W / 2;
    static constexpr int kWords = 32 * NX * NZ * NY;                  // of one box
    static constexpr int kColumn = (8 * NX * NZ + 31) / 32 * 32;       // box threads per y phase: 256, 160, 96
    static constexpr int kYStep = W == 16 ? 1 : 2;                    // phases
    static constexpr int kBoxThreads = kColumn * kYStep;
    static constexpr int kNodeThreads = W == 20 ? 384 : (W == 16 ? 256 : 64);
    static constexpr int kThreads = kBoxThreads + kNodeThreads;
    static constexpr int kCtas = W == 20 ? 1 : (W == 16 ? 2 : 4);     // resident per SM, fused
};

struct TileItem {
    int tile, slot, d, beg, end;
    int sx, sy, sz, ex, ey, ez;
    int n;
    long long grid_off;
    float sd;
};
__device__ __forceinline__ TileItem tile_item(const TileDesc &td, int d, int density)
{
    return TileItem{td.tile, td.slot, d, td.beg, td.end, td.start[0], td.start[1], td.start[2], td.edge[0], td.edge[1],
                    td.edge[2], td.n, td.grid_off, density ? td.scale_f : 1.f};
}
// 16-byte access to the grid's quads: n, the tile's start and edge multiples of 4, the lattice aligned.
__device__ __forceinline__ bool tile_vec(const TileItem &it, const float *lat)
{
    return ((it.sx | it.n | it.ex) & 3) == 0 && (reinterpret_cast<uintptr_t>(lat) & 15) == 0;
}

// Fixed-point unit (y) of an item and its reciprocal (x), the scale: keep the
// bound sum |g_k| / 8 on any value (and the rounding of its terms) below 2^31.
// The unit is the smallest such one rounded up to three mantissa bits (the bits a
// different order of the placement's additions cannot reach), so that integers
// become values by an exact product (an FP64 division of each item's sum by the
// scale held up one of the node warps that the item waits for: steps of 600 mixed
// cells 460 us, of 64 boxes 418, now 453 and 407). A power of two instead left the field of one red cell with 1.5 to 1.9 times
// the error. fsum: the placement's atomic float sum of |F_d| over n nodes, within
// (n - 1) 2^-24 of the exact one in any order.
// An MLS weight is at most 1 (mls_weights_f32), for supports from 1/0.58 on 1/2 (0.493
// there, 0.487 for the default sqrt(3)): field of 48 mixed cells in 101^3, 16-cell tiles,
// error against 64 bits 2.0e-6 with 1, 1.1e-6.
template <int KER>
__device__ __forceinline__ float2 tile_scale(const TileItem &it, float fsum, float inv_support)
{
    const float n = (float)(it.end - it.beg);
    const float bound = fsum * (1.0002f + n * 1.1920929e-7f) * it.sd *
                        (KER == 0 ? 0.125f : (inv_support <= 0.58f ? 0.5f : 1.f));
    if (!(bound > 0.f && isfinite(bound)))
        return make_float2(1.f, 1.f);
    const float least = fminf(fmaxf(bound * 0x1p-31f, 0x1p-120f), 0x1p120f);
    const float unit = __uint_as_float((__float_as_uint(least) + 0xfffffu) & 0xfff00000u);
    return make_float2(1.f / unit, unit);
}

// Copies the velocity box of an item's lattice into U asynchronously: quads
// where the grid's quads are aligned, else single values. bt: box thread.
template <int W>
__device__ __forceinline__ void tile_stage(const TileItem &it, const float *__restrict__ u, unsigned sU, int bt)
{
    using S = TileShape<W>;
    const int n = it.n, nn = n * n;
    const float *ud = u + it.grid_off + (long long)it.d * nn * n;
    if (tile_vec(it, ud)) {
        const int y0 = bt / S::kColumn;
        bt -= y0 * S::kColumn;
        const int zl = bt & 3, yl = (bt >> 2) & 1, line = bt >> 3, gx = line % S::NX, lz = 4 * (line / S::NX) + zl;
        if (line >= S::NX * S::NZ || 4 * gx >= it.ex + 8 || lz >= it.ez + 4)
            return;
        const float *src = ud + wrap1(it.sz - 2 + lz, n) * nn + wrap1(it.sx - 4 + 4 * gx, n);
        const unsigned dst = sU + 16u * (unsigned)bt;   // (line, yl, zl) in this order
#pragma unroll
        for (int k = 0; k < S::NY / S::kYStep; ++k) {
            const int yb = y0 + k * S::kYStep;
            const int ly = 2 * yb + yl;
            if (ly < it.ey + 4)
                cp_async16(dst + 128u * (unsigned)(yb * S::NZ * S::NX), src + wrap1(it.sy - 2 + ly, n) * n);
        }
    } else {
        // lanes take the 32 cells of a line, warps the lines
        const int xl = bt & 3, zl = (bt >> 2) & 3, yl = (bt >> 4) & 1;
        for (int c = bt >> 5; c < S::NX * S::NY; c += S::kBoxThreads / 32) {
            const int yb = c / S::NX, gx = c - yb * S::NX, ly = 2 * yb + yl, lx = 4 * gx + xl;
            if (lx < 2 || lx >= it.ex + 6 || ly >= it.ey + 4)
                continue;
            const float *row = ud + wrap1(it.sy - 2 + ly, n) * n + wrap1(it.sx - 4 + lx, n);
            const unsigned dst = sU + 4u * (unsigned)(bt & 31) + 128u * (unsigned)(yb * S::NZ * S::NX + gx);
#pragma unroll
            for (int zb = 0; zb < S::NZ; ++zb) {
                const int lz = 4 * zb + zl;
                if (lz < it.ez + 4)
                    cp_async4(dst + 128u * (unsigned)(zb * S::NX), row + wrap1(it.sz - 2 + lz, n) * nn);
            }
        }
    }
}

// Adds every non-zero value of A to the grid and clears it; returns the exact
// integer sum and counts the non-zero values inside the tile itself. STORE:
// values that three or more boxes can reach, those within 2 cells of a tile's
// faces along two axes or three, go to the item's box of the buffer instead, in
// A's own order, zero or not; the others have at most two terms, whose sum from
// zero is the same in either order. add (f is not cleared): values that two boxes
// can reach, near a face along one axis, go there too. buf: the item's place in the
// buffer. bt: box thread.
template <int W, bool STORE, typename Acc = int>
__device__ __forceinline__ long long tile_flush(const TileItem &it, float *__restrict__ f, float *__restrict__ buf,
                                                typename TileAcc<Acc>::Quad *A, float inv, int bt, bool add,
                                                unsigned &touched)
{
    using S = TileShape<W>;
    const int n = it.n;
    float *fd = f + it.grid_off + (long long)it.d * n * n * n;
    const bool vec = tile_vec(it, fd);
    const int y0 = bt / S::kColumn;
    bt -= y0 * S::kColumn;
    const int zl = bt & 3, yl = (bt >> 2) & 1, line = bt >> 3, gx = line % S::NX, lz = 4 * (line / S::NX) + zl;
    if (line >= S::NX * S::NZ || lz >= it.ez + 4)   // cells beyond the box stay zero
        return 0;
    float *plane = fd + wrap1(it.sz - 2 + lz, n) * n * n;
    const bool in_z = (unsigned)(lz - 2) < (unsigned)it.ez;
    const bool in_xz = in_z && (unsigned)(4 * gx - 4) < (unsigned)it.ex;
    if (vec)
        plane += wrap1(it.sx - 4 + 4 * gx, n);
    // STORE: cells of the quad that are near a face along x, and the row along z
    const bool face_z = lz < 4 || lz >= it.ez;
    unsigned face_x = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c)
        face_x |= (4 * gx + c < 6 || 4 * gx + c >= it.ex + 2) ? 1u << c : 0u;
    float4 *out = reinterpret_cast<float4 *>(buf) + bt;
    long long qsum = 0;
    A += bt;
#pragma unroll
    for (int k = 0; k < S::NY / S::kYStep; ++k) {
        const int yb = y0 + k * S::kYStep, at = 8 * yb * S::NZ * S::NX, ly = 2 * yb + yl;
        const typename TileAcc<Acc>::Quad q = A[at];
        const bool zero = (q.x | q.y | q.z | q.w) == 0;
        float v0 = (float)q.x * inv, v1 = (float)q.y * inv, v2 = (float)q.z * inv, v3 = (float)q.w * inv;
        if constexpr (STORE) {
            const bool face_y = ly < 4 || ly >= it.ey;
            const bool any = add || face_y || face_z, whole = add ? face_y || face_z : face_y && face_z;
            if (whole || (any && face_x)) {
                if (ly < it.ey + 4)
                    out[at] = make_float4(v0, v1, v2, v3);
                const unsigned keep = whole ? 0u : ~face_x;
                v0 = keep & 1u ? v0 : 0.f;
                v1 = keep & 2u ? v1 : 0.f;
                v2 = keep & 4u ? v2 : 0.f;
                v3 = keep & 8u ? v3 : 0.f;
            }
        }
        if (zero)
            continue;
        A[at] = {0, 0, 0, 0};
        float *row = plane + wrap1(it.sy - 2 + ly, n) * n;
        qsum += ((long long)q.x + q.y) + ((long long)q.z + q.w);
        const bool in_y = (unsigned)(ly - 2) < (unsigned)it.ey;
        if (vec) {
            if (!STORE || v0 != 0.f || v1 != 0.f || v2 != 0.f || v3 != 0.f)
                red_add_v4(row, v0, v1, v2, v3);
            if (in_xz && in_y)
                touched += TileAcc<Acc>::some(q.x) + TileAcc<Acc>::some(q.y) + TileAcc<Acc>::some(q.z) +
                           TileAcc<Acc>::some(q.w);
        } else {
            const Acc qc[4] = {q.x, q.y, q.z, q.w};
            const float vc[4] = {v0, v1, v2, v3};
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (qc[c] != 0) {
                    if (!STORE || vc[c] != 0.f)
                        red_add(row + wrap1(it.sx - 4 + 4 * gx + c, n), vc[c]);
                    touched += in_z && in_y && (unsigned)(4 * gx + c - 4) < (unsigned)it.ex;
                }
        }
    }
    return qsum;
}

// A node's binning record, force and id (see own_scatter_kernel).
struct TileUnit {
    float4 rec, fn;
};
__device__ __forceinline__ TileUnit tile_unit(const DevWork &w, int q)
{
    const float4 *r = w.own_rec + 2LL * q;
    return TileUnit{r[0], r[1]};
}

// p[t] = p[(r + t) & 3]
__device__ __forceinline__ void rotate4(float p[4], int r)
{
    const bool one = r & 1, two = r & 2;
    const float a0 = one ? p[1] : p[0], a1 = one ? p[2] : p[1], a2 = one ? p[3] : p[2], a3 = one ? p[0] : p[3];
    p[0] = two ? a2 : a0;
    p[1] = two ? a3 : a1;
    p[2] = two ? a0 : a2;
    p[3] = two ? a1 : a3;
}

// mls_weights in FP32, every operation's rounding stated: the same bits in each
// kernel that uses it. y: the points' distances from the node per axis (cells),
// wt: z-outer, x-inner. The cubic's outer piece is 4/3 (1 - r)^3; the moments
// are summed along x, then y, then z (a third of the products of a sum over the
// 27 points). A distance is r2 * rsqrt(r2): with sqrtf the transfer of 48 mixed
// cells in 101^3 took 83 us, 74 now; the velocities' error, 1.9e-7, is the same.
// False where the moment matrix is singular: a pivot that is not positive, or a
// weight above 1. The weights of a regular matrix are at most 1 for every support
// (0.49 for the default sqrt(3)); rounding gives larger ones where the condition
// number passes 1e6 or so, which happens for supports below 1.25 (5e3 at 1.25).
__device__ __forceinline__ bool mls_weights_f32(const float y[3][3], float inv_support, float wt[27])
{
    float A00 = 0.f, A10 = 0.f, A11 = 0.f, A20 = 0.f, A21 = 0.f, A22 = 0.f, A30 = 0.f, A31 = 0.f, A32 = 0.f, A33 = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float B00 = 0.f, B10 = 0.f, B11 = 0.f, B20 = 0.f, B21 = 0.f, B22 = 0.f;   // of the plane
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const float yz = fmaf(y[2][c], y[2][c], __fmul_rn(y[1][b], y[1][b]));
            float s0 = 0.f, s1 = 0.f, s2 = 0.f;   // of the row
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float r2 = fmaxf(fmaf(y[0][a], y[0][a], yz), 1e-30f);
                const float r = __fmul_rn(__fmul_rn(r2, rsqrtf(r2)), inv_support);
                const float q = fmaxf(__fadd_rn(1.f, -r), 0.f), qq = __fmul_rn(q, q);
                const float W = r <= 0.5f ? fmaf(-4.f * q, __fmul_rn(r, r), 2.f / 3.f) : __fmul_rn(4.f / 3.f * q, qq);
                wt[(c * 3 + b) * 3 + a] = W;
                const float Wy = __fmul_rn(W, y[0][a]);
                s0 = __fadd_rn(s0, W);
                s1 = __fadd_rn(s1, Wy);
                s2 = fmaf(Wy, y[0][a], s2);
            }
            const float t0 = __fmul_rn(s0, y[1][b]);
            B00 = __fadd_rn(B00, s0);
            B10 = __fadd_rn(B10, s1);
            B11 = __fadd_rn(B11, s2);
            B20 = __fadd_rn(B20, t0);
            B21 = fmaf(s1, y[1][b], B21);
            B22 = fmaf(t0, y[1][b], B22);
        }
        const float t0 = __fmul_rn(B00, y[2][c]);
        A00 = __fadd_rn(A00, B00);
        A10 = __fadd_rn(A10, B10);
        A11 = __fadd_rn(A11, B11);
        A20 = __fadd_rn(A20, B20);
        A21 = __fadd_rn(A21, B21);
        A22 = __fadd_rn(A22, B22);
        A30 = __fadd_rn(A30, t0);
        A31 = fmaf(B10, y[2][c], A31);
        A32 = fmaf(B20, y[2][c], A32);
        A33 = fmaf(t0, y[2][c], A33);
    }
    // A z = e1 by A = L D L^T with unit L; the pivots are those of the Cholesky factor, squared
    const float d0 = A00, i0 = __frcp_rn(d0);
    const float l10 = __fmul_rn(A10, i0), l20 = __fmul_rn(A20, i0), l30 = __fmul_rn(A30, i0);
    const float d1 = fmaf(-l10, A10, A11), i1 = __frcp_rn(d1);
    const float u21 = fmaf(-l20, A10, A21), u31 = fmaf(-l30, A10, A31);
    const float l21 = __fmul_rn(u21, i1), l31 = __fmul_rn(u31, i1);
    const float d2 = fmaf(-l21, u21, fmaf(-l20, A20, A22)), i2 = __frcp_rn(d2);
    const float u32 = fmaf(-l31, u21, fmaf(-l30, A20, A32));
    const float l32 = __fmul_rn(u32, i2);
    const float d3 = fmaf(-l32, u32, fmaf(-l31, u31, fmaf(-l30, A30, A33)));
    if (!(d0 > 0.f && d1 > 0.f && d2 > 0.f && d3 > 0.f))
        return false;
    const float f1 = -l10, f2 = fmaf(-l21, f1, -l20), f3 = fmaf(-l32, f2, fmaf(-l31, f1, -l30));
    const float z3 = __fmul_rn(f3, __frcp_rn(d3));
    const float z2 = fmaf(-l32, z3, __fmul_rn(f2, i2));
    const float z1 = fmaf(-l31, z3, fmaf(-l21, z2, __fmul_rn(f1, i1)));
    const float z0 = fmaf(-l30, z3, fmaf(-l20, z2, fmaf(-l10, z1, i0)));
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const float zz = fmaf(z2, y[1][b], fmaf(z3, y[2][c], z0));
#pragma unroll
            for (int a = 0; a < 3; ++a)
                wt[(c * 3 + b) * 3 + a] = __fmul_rn(wt[(c * 3 + b) * 3 + a], fmaf(z1, y[0][a], zz));
        }
    if (inv_support > 0.75f) {
        float most = 0.f;
#pragma unroll
        for (int J = 0; J < 27; ++J)
            most = fmaxf(most, fabsf(wt[J]));
        return most <= 1.0001f;
    }
    return true;
}

// One (node, lattice) unit: spreads into A, interpolates from U, or both
// (gq: the node's force times the item's fixed-point scale).
// MLS units take their 27 points in plain order: the weights (a 4 x 4 moment
// system, mls_weights_f32) cost more than the banks. 48 mixed cells in a 101^3
// grid, transfers of a step: 202 us with a spread over candidate lists that
// evaluated a node's weights in each of its tiles, plus the interpolation; 85 us.
template <int KER, int W, bool SPREAD, bool INTERP, typename Acc = int>
__device__ __forceinline__ void tile_node(const TileItem &cur, const DevWork &w, const TileUnit &un, float gsc,
                                          const unsigned char *U, unsigned sA, float *__restrict__ v,
                                          const float *__restrict__ x, const float *__restrict__ vp,
                                          float *__restrict__ xn, float dt, float inv_support, long long N)
{
    using S = TileShape<W>;
    const int lane = threadIdx.x & 31, d = cur.d;
    const int node = __float_as_int(un.fn.w);
    const float gq = (d == 0 ? un.fn.x : (d == 1 ? un.fn.y : un.fn.z)) * gsc;
    const unsigned pk = __float_as_uint(un.rec.w);
    const float fr[3] = {un.rec.x, un.rec.y, un.rec.z};
    int l0[3];
    bool inside = true;
    auto put = [&](float out) {
        const long long i = d * N + node;
        v[i] = out;
        if (xn)   // Eq. Bashforth_eqn
            xn[i] = ab2_value(x[i], out, vp[i], dt);
    };
    if constexpr (KER == 1) {
        float y[3][3], wt[27];
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            const float s = ax == d ? fr[ax] : fr[ax] - 0.5f;   // from the node's cell
            const float base = floorf(s + 0.5f) - 1.f;
#pragma unroll
            for (int m = 0; m < 3; ++m)
                y[ax][m] = (base + (float)m) - s;
            l0[ax] = (int)((pk >> (8 * ax)) & 255u) + (int)base + 2;
            inside = inside && (unsigned)l0[ax] <= (unsigned)(ax == 0 ? cur.ex : (ax == 1 ? cur.ey : cur.ez)) + 1u;
        }
        const bool regular = mls_weights_f32(y, inv_support, wt);
        if (!inside || !regular) {   // a singular moment matrix (or an inconsistent record: never expected)
            status_add(w.status, ST_DOMAIN, SPREAD && INTERP ? 2 : 1);   // once per transfer
            if constexpr (INTERP)
                put(0.f);
            return;
        }
        int xo[3], yo[3], zo[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const int lx = l0[0] + 2 + m, ly = l0[1] + m, lz = l0[2] + m;
            xo[m] = 4 * (lx & 3) + 128 * (lx >> 2);
            zo[m] = 16 * (lz & 3) + 128 * S::NX * (lz >> 2);
            yo[m] = 64 * (ly & 1) + 128 * S::NX * S::NZ * (ly >> 1);
        }
        float out = 0.f;
        int J = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int bb = 0; bb < 3; ++bb)
#pragma unroll
                for (int a = 0; a < 3; ++a, ++J) {
                    const int o = zo[c] + yo[bb] + xo[a];
                    if constexpr (INTERP)
                        out = fmaf(wt[J], *reinterpret_cast<const float *>(U + o), out);
                    if constexpr (SPREAD)
                        TileAcc<Acc>::add(sA, o, __fmul_rn(wt[J], gq));
                }
        if constexpr (INTERP)
            put(out);
        return;
    }
    float ph[3][4];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        // lattice d sits at the cell coordinate, the other two half a
        // cell lower: s = t - 1/2 has floor(t) - 1 and fraction r + 1/2
        // below r = 1/2, so the stencil starts 2 (not 1) cells below
        const int c = (int)((pk >> (8 * ax)) & 255u);   // cell within the tile
        int sh = 1;
        float r = fr[ax];
        if (ax != d) {
            const bool low = r < 0.5f;
            r = low ? r + 0.5f : r - 0.5f;
            sh = low ? 0 : 1;
        }
        peskin_frac(r, ph[ax]);
        l0[ax] = c + sh;   // first stencil cell, from 2 cells below the tile
        inside = inside && l0[ax] <= (ax == 0 ? cur.ex : (ax == 1 ? cur.ey : cur.ez));
    }
    if (!inside) {   // a record inconsistent with this tile: never expected
        status_add(w.status, ST_DOMAIN, 1);
        return;
    }
    // byte offsets of the lane's points in step order (see above)
    int xo[4], zo[4], yo[2];
    const int xl = (l0[0] + 2) & 3, xq = (l0[0] + 2) >> 2;   // the box starts 4 cells below in x
    const int zl = l0[2] & 3, zq = l0[2] >> 2, yl = l0[1] & 1, yq = l0[1] >> 1;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int tx = (lane + t) & 3, tz = ((lane >> 2) + t) & 3;
        xo[t] = 4 * tx + 128 * (xq + (tx < xl));
        zo[t] = 16 * tz + 128 * S::NX * (zq + (tz < zl));
    }
    const int ry = ((lane >> 4) ^ yl) & 1;   // y offset (0 or 1) of step t2 = 0
#pragma unroll
    for (int t = 0; t < 2; ++t)
        yo[t] = 64 * ((lane >> 4) ^ t) + 128 * S::NX * S::NZ * (yq + (yl & (ry ^ t)));
    rotate4(ph[0], lane - xl);
    rotate4(ph[2], (lane >> 2) - zl);
    const float py0 = ry ? ph[1][1] : ph[1][0], py2 = ry ? ph[1][3] : ph[1][2];
    const float py1 = ry ? ph[1][0] : ph[1][1], py3 = ry ? ph[1][2] : ph[1][3];
    constexpr int kRow2 = 128 * S::NX * S::NZ;   // two y rows further
    float p[4];
#pragma unroll
    for (int t0 = 0; t0 < 4; ++t0) {
        float qz[4];
        const float gx = ph[0][t0] * gq;
#pragma unroll
        for (int t1 = 0; t1 < 4; ++t1) {
            const int oa = xo[t0] + zo[t1] + yo[0], ob = xo[t0] + zo[t1] + yo[1];
            if constexpr (INTERP) {
                const float ua = *reinterpret_cast<const float *>(U + oa);
                const float uc = *reinterpret_cast<const float *>(U + oa + kRow2);
                const float ub = *reinterpret_cast<const float *>(U + ob);
                const float ue = *reinterpret_cast<const float *>(U + ob + kRow2);
                const float sa = fmaf(py2, uc, __fmul_rn(py0, ua)), sb = fmaf(py3, ue, __fmul_rn(py1, ub));
                qz[t1] = __fmul_rn(ph[2][t1], __fadd_rn(sa, sb));
            }
            if constexpr (SPREAD) {
                const float gz = gx * ph[2][t1];
                TileAcc<Acc>::add(sA, oa, py0 * gz);
                TileAcc<Acc>::add(sA, oa + kRow2, py2 * gz);
                TileAcc<Acc>::add(sA, ob, py1 * gz);
                TileAcc<Acc>::add(sA, ob + kRow2, py3 * gz);
            }
        }
        if constexpr (INTERP)
            p[t0] = __fmul_rn(ph[0][t0], __fadd_rn(__fadd_rn(qz[0], qz[2]), __fadd_rn(qz[1], qz[3])));
    }
    if constexpr (INTERP)
        put(__fadd_rn(__fadd_rn(p[0], p[2]), __fadd_rn(p[1], p[3])));
}

template <int KER, int W, bool SPREAD, bool INTERP, bool STORE>
__global__ void __launch_bounds__(TileShape<W>::kThreads, TileShape<W>::kCtas)
    transfer_tile_kernel(DevBatch b, DevWork w, const float *__restrict__ x, float *__restrict__ f, int density,
                         const float *__restrict__ u, float *__restrict__ v, const float *__restrict__ vp,
                         float *__restrict__ xn, float dt, float inv_support, int lattice, int add)
{
    using S = TileShape<W>;
    constexpr int kBox = 4 * S::kWords, kBoxWarps = S::kBoxThreads / 32, kRing = 8;
    extern __shared__ __align__(128) unsigned char tile_smem[];
    unsigned char *U = tile_smem, *A = tile_smem + (INTERP ? 2 * kBox : 0);
    __shared__ long long s_red[2][kBoxWarps];
    __shared__ float2 s_scale[4];   // fixed-point scale and unit of item i in i % 4
    // items i of this CTA in slot i % kRing: lattice (-1: none) and descriptor
    __shared__ int s_d[kRing];
    __shared__ __align__(16) TileDesc s_desc[kRing];
    const long long N = b.N;
    const int lane = threadIdx.x & 31;
    const bool box = threadIdx.x < S::kBoxThreads;
    const int bt = threadIdx.x, nt = (int)threadIdx.x - S::kBoxThreads;
    // a kernel launched after this one with programmatic serialization (the
    // next lattice of the same step, which reads nothing this one writes) may
    // start at once: the grid is sized to be resident, so its CTAs take the
    // SMs that this grid's CTAs leave when the items run out
    pdl_trigger();
    if constexpr (SPREAD)
        for (int i = threadIdx.x; i < 2 * kBox / 16; i += S::kThreads)
            reinterpret_cast<int4 *>(A)[i] = make_int4(0, 0, 0, 0);
    if (lattice < 0)
        pdl_wait();   // for the binning's placement
    // the first box warp takes the items: the counter's answer for item i + 3
    // travels during item i, the descriptor of item i + 2 is copied during it
    const int n_items = w.counters[3] * (lattice < 0 ? 3 : 1);
    int *counter = tile_counter(w, lattice);
    // Fewer than 3 items per CTA: strided over the CTAs, so that the longest CTA
    // has as few as can be and no counter is waited for (one cell in 128^3, 150
    // items for 304 CTAs: 17.7 us with three each, 8.4 now). Else each CTA begins with three neighbours (of
    // one tile, mostly) and takes the rest as it gets to them.
    const bool few = n_items < 3 * (int)gridDim.x;
    int ahead = 0;   // its lane 0: number of the next item to be copied
    auto fetch = [&](int it, int i) {
        const int q = lattice < 0 ? it / 3 : it, slot = i % kRing;
        if (lane == 0)
            s_d[slot] = it < n_items ? (lattice < 0 ? it - 3 * q : lattice) : -1;
        if (lane < (int)sizeof(TileDesc) / 16 && it < n_items)
            cp_async16(smem_u32(&s_desc[slot]) + 16u * lane,
                       reinterpret_cast<const char *>(w.tile_desc + q) + 16 * lane);
    };
    if (threadIdx.x < 32) {
        int first = blockIdx.x;
        if (!few) {
            if (lane == 0)
                first = atomicAdd(counter, 3);
            first = __shfl_sync(0xffffffffu, first, 0);
        }
        const int step = few ? gridDim.x : 1;
        ahead = first + 2 * step;
        fetch(first, 0);
        fetch(first + step, 1);
        cp_async_wait_all();
    }
    __syncthreads();
    if (s_d[0] < 0)
        return;
    if (INTERP && box) {
        tile_stage<W>(tile_item(s_desc[0], s_d[0], density), u, smem_u32(U), bt);
        cp_async_wait_all();
    }
    // a node thread's first unit of the next item
    TileUnit un{};
    auto unit_ahead = [&](int i) {
        if (s_d[i % kRing] < 0)
            return;
        const TileDesc &td = s_desc[i % kRing];
        if (td.beg + nt < td.end)
            un = tile_unit(w, td.beg + nt);
    };
    auto put_scale = [&](int i, float fsum) {   // one thread
        s_scale[i & 3] = tile_scale<KER>(tile_item(s_desc[i % kRing], s_d[i % kRing], density), fsum, inv_support);
    };
    auto get_fsum = [&](int i) {
        const long long at = 3LL * s_desc[i % kRing].tile + s_d[i % kRing];
        return STORE ? fsum_get(w.tile_fbin + kFsumBins * at) : w.tile_fsum[at];
    };
    auto write_sum = [&](int i) {   // one thread: the exact integer sum of a flushed item, scaled, times h^3
        const TileDesc &td = s_desc[i % kRing];
        long long vsum = 0;
#pragma unroll
        for (int q = 0; q < kBoxWarps; ++q)
            vsum += s_red[i & 1][q];
        w.red_tile[3LL * td.tile + s_d[i % kRing]] = (double)vsum * (double)s_scale[i & 3].y * td.h3;
    };
    if (!box)
        unit_ahead(0);
    if (SPREAD && threadIdx.x == 32)
        put_scale(0, get_fsum(0));
    __syncthreads();
    unsigned touched = 0;
    int i = 0;
    for (;; ++i) {
        const bool valid = s_d[i % kRing] >= 0;
        if (!box) {
            if (SPREAD && i > 1 && nt == S::kNodeThreads - 1)
                write_sum(i - 2);
            if (valid) {
                const TileItem cur = tile_item(s_desc[i % kRing], s_d[i % kRing], density);
                const float gsc = SPREAD ? cur.sd * s_scale[i & 3].x : 0.f;
                TileUnit mine = un;
                int q = cur.beg + nt;
                const bool more = q + S::kNodeThreads < cur.end;
                if (more)
                    un = tile_unit(w, q + S::kNodeThreads);
                else
                    unit_ahead(i + 1);
                const unsigned char *Ui = U + (i & 1) * kBox;
                const unsigned sA = smem_u32(A) + (unsigned)((i & 1) * kBox);
                if (q < cur.end)
                    tile_node<KER, W, SPREAD, INTERP>(cur, w, mine, gsc, Ui, sA, v, x, vp, xn, dt, inv_support, N);
                if (more) {
#pragma unroll 1
                    for (q += S::kNodeThreads; q < cur.end; q += S::kNodeThreads) {
                        mine = un;
                        if (q + S::kNodeThreads < cur.end)
                            un = tile_unit(w, q + S::kNodeThreads);
                        tile_node<KER, W, SPREAD, INTERP>(cur, w, mine, gsc, Ui, sA, v, x, vp, xn, dt, inv_support, N);
                    }
                    unit_ahead(i + 1);
                }
            }
        } else {
            const bool scales = SPREAD && threadIdx.x == 32 && s_d[(i + 1) % kRing] >= 0;
            const float fsum = scales ? get_fsum(i + 1) : 0.f;
            if (valid) {
                if (threadIdx.x < 32) {
                    fetch(__shfl_sync(0xffffffffu, ahead, 0), i + 2);
                    if (lane == 0)
                        ahead = few ? n_items : atomicAdd(counter, 1);
                }
                if (INTERP && s_d[(i + 1) % kRing] >= 0)
                    tile_stage<W>(tile_item(s_desc[(i + 1) % kRing], s_d[(i + 1) % kRing], density), u,
                                  smem_u32(U) + (unsigned)(((i + 1) & 1) * kBox), bt);
            }
            if (SPREAD && i > 0) {
                // this flush's sum is written during the next item, by a node
                // thread; the next item's scale by a thread of the second warp
                const TileItem old = tile_item(s_desc[(i - 1) % kRing], s_d[(i - 1) % kRing], density);
                int4 *box_A = reinterpret_cast<int4 *>(A + ((i - 1) & 1) * kBox);
                const float inv = s_scale[(i - 1) & 3].y;
                float *buf = w.box_buf + ((long long)w.box_lattices * old.slot + (w.box_lattices == 3 ? old.d : 0)) * S::kWords;
                long long qsum = tile_flush<W, STORE>(old, f, buf, box_A, inv, bt, add != 0, touched);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    qsum += __shfl_down_sync(0xffffffffu, qsum, o);
                if (lane == 0)
                    s_red[(i - 1) & 1][threadIdx.x >> 5] = qsum;
            }
            if (scales)
                put_scale(i + 1, fsum);
            cp_async_wait_all();
        }
        asm volatile("" ::: "memory");   // the node threads' reductions stay before the barrier
        __syncthreads();
        if (!valid)
            break;
    }
    if constexpr (SPREAD) {
        if (threadIdx.x == 0)
            write_sum(i - 1);   // i >= 1: the CTA had an item
        // one update per warp and launch: one per warp and item, all on this
        // one word, took longer than the rest of the kernel
        touched = __reduce_add_sync(0xffffffffu, touched);
        if (lane == 0)
            status_add(w.status, ST_TOUCHED, touched);
    }
}

// The reproducible spread with 64-bit accumulators, on request (ifem_ctx_create): small
// forces beside large ones keep their digits. One box, a CTA per item, whose threads
// first take its nodes and then flush it: twice the memory leaves no room for the box
// that would be worked on meanwhile. Interpolation is a launch of its own. 27 bits of
// scale more than tile_scale's, so that the sum of a whole box fits 64 bits. Steps of 72
// mixed cells, 128^3: 226 us (95 with 32 bits); 48 with MLS, 101^3: 205 (110).
template <int KER, int W>
__global__ void __launch_bounds__(TileShape<W>::kBoxThreads)
    spread_wide_kernel(DevWork w, float *__restrict__ f, int density, float inv_support, int lattice, int add)
{
    using S = TileShape<W>;
    using Quad = TileAcc<long long>::Quad;
    constexpr int T = S::kBoxThreads;
    extern __shared__ __align__(128) unsigned char tile_smem[];
    Quad *A = reinterpret_cast<Quad *>(tile_smem);
    __shared__ long long s_red[T / 32];
    for (int i = threadIdx.x; i < S::kWords / 4; i += T)
        A[i] = {0, 0, 0, 0};
    pdl_wait();   // for the binning's placement
    const int per_tile = lattice < 0 ? 3 : 1, n_items = per_tile * w.counters[3];
    unsigned touched = 0;
    for (int i = blockIdx.x; i < n_items; i += gridDim.x) {
        const TileDesc td = w.tile_desc[i / per_tile];
        const TileItem it = tile_item(td, lattice < 0 ? i % 3 : lattice, density);
        const float2 sc = tile_scale<KER>(it, fsum_get(w.tile_fbin + kFsumBins * (3LL * it.tile + it.d)), inv_support);
        const float unit = fmaxf(sc.y * 0x1p-27f, 0x1p-120f);
        __syncthreads();   // the box is clear
        for (int q = it.beg + (int)threadIdx.x; q < it.end; q += T)
            tile_node<KER, W, true, false, long long>(it, w, tile_unit(w, q), it.sd * (1.f / unit), nullptr, smem_u32(A),
                                                      nullptr, nullptr, nullptr, nullptr, 0.f, inv_support, 0);
        asm volatile("" ::: "memory");   // the reductions stay before the barrier
        __syncthreads();
        float *buf = w.box_buf + ((long long)w.box_lattices * it.slot + (w.box_lattices == 3 ? it.d : 0)) * S::kWords;
        long long qsum = tile_flush<W, true, long long>(it, f, buf, A, unit, threadIdx.x, add != 0, touched);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            qsum += __shfl_down_sync(0xffffffffu, qsum, o);
        if ((threadIdx.x & 31) == 0)
            s_red[threadIdx.x >> 5] = qsum;
        __syncthreads();
        if (threadIdx.x == 0) {
            long long vsum = 0;
            for (int k = 0; k < T / 32; ++k)
                vsum += s_red[k];
            w.red_tile[3LL * it.tile + it.d] = (double)vsum * (double)unit * td.h3;
        }
    }
    touched = __reduce_add_sync(0xffffffffu, touched);
    if ((threadIdx.x & 31) == 0)
        status_add(w.status, ST_TOUCHED, touched);
}

// The reproducible spread's second half: the values of the cleared field f that
// three or more boxes can reach (tile_flush), each the sum of its boxes' terms
// in a fixed order; with add those that two or more can reach, the sum added to f.
// Unit = (tile, lattice); L = 1: of the lattice given. Every tile has at least 4 cells per
// axis (own_tiling), so a value near a face has one neighbour there, along two
// axes or three of them; along an axis of one or two tiles the neighbour is the
// tile itself or the same one on both sides, with different cells of its box.
// Bound by the loads' latency: an item, two cells of x, has its 4 or 8 loads in
// flight together, and what a unit needs to know of its tile and neighbours is read
// during the unit before it. 16% of a 16-cell tile's values come here (58% with
// add): 10 us for 72 mixed cells in a 128^3 grid, after 46 of the transfer. Storing
// whole boxes and summing every value took 27 (47 when only their non-zero quads were
// written and read, by a mask); single values where the grid's quads are not aligned
// made a step of 64 boxes of any size 606 us, 566 in pairs. The spread over candidate
// lists that this replaces (every tile visits each node whose stencil reaches it)
// took 106 after an interpolation of 37.
// add: adding the sums of the reached tiles' values where they belong. Clearing a
// second field, spreading into it and adding it reads and writes every value of every
// box: steps of one red cell in 256^3 203 us, 49 now; 72 mixed cells, 128^3, 125 and
// 117; 600, 256^3, 701 and 635; 64 boxes 777 and 705.
struct CombineUnit {
    int slot[27], start[3], edge[3], prev[3], n;   // neighbours' boxes; first cell, cells, the previous tile's cells
    long long off;
};
constexpr int kCombineThreads = 128;

// An item is two cells along x, or one at the end of an odd row. EVEN: the tile and
// the one before it have an even number of cells along x, so that both cells lie in
// one pair of every box; else the x neighbours' values are loaded one by one (the
// two cells may even have different ones), the others in pairs from even cells on.
// L: lattices whose boxes are kept (DevWork::box_lattices; known when compiled, 117 us
// for a step of 72 mixed cells with add, 125 with the product at run time).
template <int W, int L, bool EVEN>
__device__ __forceinline__ void combine_unit(const CombineUnit &un, const float *__restrict__ boxes, float *__restrict__ fd,
                                             bool add)
{
    using S = TileShape<W>;
    constexpr long long kStride = (long long)L * S::kWords;   // between the boxes of two tiles
    const int n = un.n, ex = un.edge[0], ey = un.edge[1], ez = un.edge[2];
    const bool vec = ((un.start[0] | n) & 1) == 0 && (reinterpret_cast<uintptr_t>(fd) & 7) == 0;
    // rows near a face along y and z: all of x; rows near one of them: the two ends of x.
    // add: rows near a face along y or z: all of x; the others: the ends
    const int nx = (ex + 1) / 2, one_z = 4 * (ey - 4), one = one_z + 4 * (ez - 4);
    const int whole = nx * (add ? 16 + one : 16), part = 2 * (add ? (ey - 4) * (ez - 4) : one);
    auto near = [](int k, int e) { return k < 2 ? k : e - 4 + k; };
    // neighbour along an axis, and the cell in the neighbour's box (halo h)
    auto side = [](int c, int e) { return c < 2 ? -1 : (c >= e - 2 ? 1 : 0); };
    auto other = [](int c, int e, int prev, int h) { return c < 2 ? c + prev + h : c - e + h; };
    auto word_x = [](int l) { return 32 * (l >> 2) + (l & 3); };
    auto word_y = [](int l) { return 32 * S::NX * S::NZ * (l >> 1) + 16 * (l & 1); };
    auto word_z = [](int l) { return 32 * S::NX * (l >> 2) + 4 * (l & 3); };
    for (int i = threadIdx.x; i < whole + part; i += kCombineThreads) {
        int x, y, z, r;   // r: the row, first the 16 near both, then those near one, then the others
        if (i < whole) {
            r = i / nx;
            x = 2 * (i - r * nx);
        } else {
            const int j = i - whole;
            r = (j >> 1) + (add ? 16 + one : 16);
            x = j & 1 ? ex - 2 : 0;
        }
        if (r < 16) {
            z = near(r & 3, ez);
            y = near(r >> 2, ey);
        } else if (r < 16 + one_z) {
            z = near(r & 3, ez);
            y = 2 + ((r - 16) >> 2);
        } else if (r < 16 + one) {
            y = near((r - 16 - one_z) & 3, ey);
            z = 2 + ((r - 16 - one_z) >> 2);
        } else {
            z = (r - 16 - one) / (ey - 4);
            y = 2 + r - 16 - one - z * (ey - 4);
            z += 2;
        }
        const bool two = EVEN || x + 1 < ex;
        const int o[3] = {side(x, ex), side(y, ey), side(z, ez)}, o1 = EVEN ? o[0] : (two ? side(x + 1, ex) : 0);
        const int wx[2] = {word_x(x + 4), word_x(other(x, ex, un.prev[0], 4))};
        const int wx1[2] = {word_x(x + 5), word_x(other(x + 1, ex, un.prev[0], 4))};
        const int wy[2] = {word_y(y + 2), word_y(other(y, ey, un.prev[1], 2))};
        const int wz[2] = {word_z(z + 2), word_z(other(z, ez, un.prev[2], 2))};
        float2 q[8];
        bool any = false;
#pragma unroll
        for (int k = 0; k < 8; ++k) {   // own box first
            const int kx = k & 1, ky = k >> 1 & 1, kz = k >> 2;
            const int at = 13 + 3 * ky * o[1] + 9 * kz * o[2];
            const float *p = boxes + (ky ? wy[1] : wy[0]) + (kz ? wz[1] : wz[0]);
            const bool there = !(ky && !o[1]) && !(kz && !o[2]);
            q[k] = make_float2(0.f, 0.f);
            const int slot = un.slot[at + kx * o[0]];
            const bool first = there && slot >= 0 && !(kx && !o[0]);
            if (EVEN || (!kx && !(x & 1))) {   // an odd row's last pair ends outside the tile: a cell of the box
                if (first)
                    q[k] = __ldg(reinterpret_cast<const float2 *>(p + kStride * slot + (kx ? wx[1] : wx[0])));
            } else {
                const int slot1 = un.slot[at + kx * o1];
                if (first)
                    q[k].x = __ldg(p + kStride * slot + (kx ? wx[1] : wx[0]));
                if (two && there && slot1 >= 0 && !(kx && !o1)) {
                    q[k].y = __ldg(p + kStride * slot1 + (kx ? wx1[1] : wx1[0]));
                    any = true;
                }
            }
            any |= first;
        }
        if (!any)
            continue;
        float2 acc = q[0];
#pragma unroll
        for (int k = 1; k < 8; ++k) {
            acc.x += q[k].x;
            acc.y += q[k].y;
        }
        float *out = fd + ((long long)(un.start[2] + z) * n + un.start[1] + y) * n + un.start[0] + x;
        if (add) {   // one term a value; by reductions, so that calls on other streams may add to f too
            if (vec && two && !(x & 1)) {
                if (acc.x != 0.f || acc.y != 0.f)
                    red_add_v2(out, acc.x, acc.y);
            } else {
                if (acc.x != 0.f)
                    red_add(out, acc.x);
                if (two && acc.y != 0.f)
                    red_add(out + 1, acc.y);
            }
        } else if (vec && two && !(x & 1)) {
            *reinterpret_cast<float2 *>(out) = acc;
        } else {
            *out = acc.x;
            if (two)
                out[1] = acc.y;
        }
    }
}

template <int W, int L>
__global__ void __launch_bounds__(kCombineThreads, 8)
    tile_combine_kernel(DevGrid g, DevWork w, float *__restrict__ f, int add, int lattice)
{
    pdl_wait();
    using S = TileShape<W>;
    __shared__ CombineUnit s_unit[2];
    const int units = L * w.counters[9], lane = threadIdx.x;
    // first warp: lane k < 27 a neighbour's slot, lanes 27 to 29 an axis, lane 30 the box
    int3 got;
    long long off = 0;
    auto near_of = [&](int unit) {
        return unit < units ? w.near_tile[unit / L] : make_int2(-1, 0);   // tile, box
    };
    auto read = [&](int2 near) {
        if (near.x < 0)
            return;
        const BoxDev &B = g.boxes[near.y];
        const int T = B.T, local = (int)(near.x - B.tile_base);
        const int j[3] = {local % T, (local / T) % T, local / (T * T)};
        if (lane < 27) {
            const int jx = wrap1(j[0] + lane % 3 - 1, T), jy = wrap1(j[1] + lane / 3 % 3 - 1, T);
            const int jz = wrap1(j[2] + lane / 9 - 1, T);
            got.x = w.tile_slot[B.tile_base + (jz * T + jy) * T + jx];
        } else if (lane < 30) {
            const int ja = lane == 27 ? j[0] : (lane == 28 ? j[1] : j[2]);
            got = make_int3(tile_start(ja, B.t), tile_edge(ja, B.t, T, B.n), tile_edge(wrap1(ja - 1, T), B.t, T, B.n));
        } else if (lane == 30) {
            got.x = B.n;
            off = B.grid_off;
        }
    };
    auto keep = [&](CombineUnit &u) {
        if (lane < 27) {
            u.slot[lane] = got.x;
        } else if (lane < 30) {
            u.start[lane - 27] = got.x;
            u.edge[lane - 27] = got.y;
            u.prev[lane - 27] = got.z;
        } else if (lane == 30) {
            u.n = got.x;
            u.off = off;
        }
    };
    int2 next = make_int2(-1, 0);
    if (threadIdx.x < 32) {
        read(near_of(blockIdx.x));
        next = near_of(blockIdx.x + gridDim.x);
        keep(s_unit[0]);
    }
    __syncthreads();
    for (int unit = blockIdx.x, buf = 0; unit < units; unit += gridDim.x, buf ^= 1) {
        if (threadIdx.x < 32) {
            read(next);
            next = near_of(unit + 2 * gridDim.x);
        }
        const CombineUnit &un = s_unit[buf];
        const int d = L == 3 ? unit % 3 : lattice, n = un.n;
        float *fd = f + un.off + (long long)d * n * n * n;
        const float *boxes = w.box_buf + (L == 3 ? (long long)d * S::kWords : 0);
        if (((un.edge[0] | un.prev[0]) & 1) == 0)
            combine_unit<W, L, true>(un, boxes, fd, add != 0);
        else
            combine_unit<W, L, false>(un, boxes, fd, add != 0);
        if (threadIdx.x < 32)
            keep(s_unit[buf ^ 1]);
        __syncthreads();
    }
}

// ---------------------------------------- spread, FP64 deterministic, MLS
// Owner-computes gather: each thread owns up to kDetCells values of the tile
// (per lattice), starts from the current grid value and adds the
// contributions of the tile's candidate nodes in ascending node order:
// f = f + w*g with the node's MLS weight w of that value, g = F*scale. This is
// the oracle's per-value summation order, so the result is bit-identical.
// (The Peskin kernel has its own warp-per-unit kernel, spread_det_warp_kernel.)
constexpr int kDetThreads = 256;
constexpr int kDetCells = 4;     // owned values per thread and lattice (1024 per chunk; 2 CTAs per SM)
constexpr int kDetChunk = 32;    // candidates staged per round

struct DetCand {
    int lo[3];            // wrapped cell c-2 (union reach of all lattices)
    int base[3][3];       // [d][a] wrapped first stencil index
    double wt[3][27];     // [d][J] MLS weights
    double g[3];
    int ok;
};

static __global__ void __launch_bounds__(kDetThreads, 2) spread_det_mls_kernel(DevBatch b, DevGrid g, DevWork w,
                                                                 const double *__restrict__ x,
                                                                 const double *__restrict__ F,
                                                                 double *__restrict__ f, int density,
                                                                 double support)
{
    __shared__ DetCand cand[kDetChunk];
    __shared__ double red_sh[3][kDetThreads / 32];
    const long long N = b.N;
    const ActiveTiles active(w);
    const int n_active = active.total;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        status_add(w.status, ST_PAIRS, (unsigned long long)w.cand_off[g.n_tiles]);
        status_add(w.status, ST_ACTIVE, (unsigned long long)n_active);
    }
    for (int it = blockIdx.x; it < n_active; it += gridDim.x) {
        const int tile = active.tile(g, w, it);
        const TileInfo ti = decode_tile(g, tile);
        const BoxDev B = g.boxes[ti.box];
        const int ex = ti.edge[0], ey = ti.edge[1], ez = ti.edge[2];
        const int vol = ex * ey * ez;
        const long long n3 = (long long)B.n * B.n * B.n;
        double part[3] = {0.0, 0.0, 0.0};
        // owned values in chunks of kDetThreads * kDetCells; each chunk walks
        // every candidate of the tile in ascending node order
        for (int cbase = 0; cbase < vol; cbase += kDetThreads * kDetCells) {
            double accv[kDetCells][3], init[kDetCells][3];
            int cx[kDetCells], cy[kDetCells], cz[kDetCells];
#pragma unroll
            for (int q = 0; q < kDetCells; ++q) {
                int i = cbase + threadIdx.x + q * kDetThreads;
                int lx = i % ex, ly = (i / ex) % ey, lz = i / (ex * ey);
                cx[q] = ti.start[0] + lx;
                cy[q] = ti.start[1] + ly;
                cz[q] = ti.start[2] + lz;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    double v = 0.0;
                    if (i < vol)
                        v = f[B.grid_off + d * n3 + ((long long)cz[q] * B.n + cy[q]) * B.n + cx[q]];
                    accv[q][d] = v;
                    init[q][d] = v;
                }
            }
            const double scale = density ? B.scale : 1.0;
            const int beg = w.cand_off[tile], end = w.cand_off[tile + 1];
            for (int c0 = beg; c0 < end; c0 += kDetChunk) {
                const int nc = min(kDetChunk, end - c0);
                __syncthreads();
                // stage candidate data: one thread per (candidate, lattice)
                for (int t = threadIdx.x; t < nc * 3; t += blockDim.x) {
                    const int j = t / 3, d = t % 3;
                    const int node = w.cand_nodes[c0 + j];
                    DetCand &C = cand[j];
                    const InstDev I = b.inst[b.node_inst[node]];
                    double s[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        int I0;
                        s[a] = LatCoord<double>::get(I, B, a, x[a * N + node], (double)mac_off(d, a), I0);
                    }
                    if (d == 0) {
                        C.ok = 1;
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            int I0;
                            double sc = LatCoord<double>::get(I, B, a, x[a * N + node], 0.0, I0);
                            C.lo[a] = wrapi((long long)floor(sc) - 2, B.n);
                        }
                    }
                    C.g[d] = F[d * N + node] * scale;
                    int base[3];
                    if (!mls_weights<double>(s, support, base, C.wt[d])) {
                        status_add(w.status, ST_DOMAIN, 1);
                        C.g[d] = 0.0;
#pragma unroll
                        for (int J = 0; J < 27; ++J)
                            C.wt[d][J] = 0.0;
                    }
#pragma unroll
                    for (int a = 0; a < 3; ++a)
                        C.base[d][a] = wrapi(base[a], B.n);
                }
                __syncthreads();
                for (int j = 0; j < nc; ++j) {
                    const DetCand &C = cand[j];
#pragma unroll
                    for (int q = 0; q < kDetCells; ++q) {
                        if (cbase + threadIdx.x + q * kDetThreads >= vol)
                            break;
                        int rx = cx[q] - C.lo[0], ry = cy[q] - C.lo[1], rz = cz[q] - C.lo[2];
                        rx += rx < 0 ? B.n : 0;
                        ry += ry < 0 ? B.n : 0;
                        rz += rz < 0 ? B.n : 0;
                        if (rx > 4 || ry > 4 || rz > 4)
                            continue;
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            int mx = cx[q] - C.base[d][0], my = cy[q] - C.base[d][1], mz = cz[q] - C.base[d][2];
                            mx += mx < 0 ? B.n : 0;
                            my += my < 0 ? B.n : 0;
                            mz += mz < 0 ? B.n : 0;
                            if (mx <= 2 && my <= 2 && mz <= 2)
                                accv[q][d] = accv[q][d] + C.wt[d][(mz * 3 + my) * 3 + mx] * C.g[d];
                        }
                    }
                }
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < kDetCells; ++q) {
                int i = cbase + threadIdx.x + q * kDetThreads;
                if (i >= vol)
                    break;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    f[B.grid_off + d * n3 + ((long long)cz[q] * B.n + cy[q]) * B.n + cx[q]] = accv[q][d];
                    part[d] += accv[q][d] - init[q][d];
                }
            }
        }
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            double v = part[d];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0)
                red_sh[d][wid] = v;
        }
        __syncthreads();
        if (threadIdx.x < 3) {
            double v = 0.0;
            for (int q = 0; q < kDetThreads / 32; ++q)
                v += red_sh[threadIdx.x][q];
            w.red_tile[3LL * tile + threadIdx.x] = v * (1.0 / B.scale);
        }
    }
}

// FP64 deterministic Peskin spread, one warp per unit = (tile, lattice), the
// longest candidate lists first; the longest (tile_class 0) are walked by 8 warps,
// one per octant of the tile. The unit's owned values sit in a shared-memory
// accumulator loaded from f; the warp walks the tile's candidates in ascending
// node order, f = f + ((phi_x phi_y) phi_z) g, those whose points miss the unit
// left out 32 at a time, with a warp barrier between candidates, so every value
// receives its terms in the oracle's order. A candidate's points inside the unit
// (40% of them for 8-cell tiles) are dealt to consecutive lanes: 1.25 rounds of
// three products and an addition, 1.64 with a fixed lane per point. kDetAhead
// candidates' weights are computed before the first of them is added; the next
// candidates' stencils are copied from the binning's table (det_weights_kernel)
// meanwhile.
// Bound by the FP64 pipe, which is charged per warp instruction whatever the
// active lanes: 19 cycles on an SM, 64 between two of one warp, of about 6 a
// candidate; and at the end by the longest walks, about 700 cycles a candidate.
// 133 k nodes in 120^3, 8-cell tiles: 530 us; 788 with a lane fixed to each point,
// whole tiles in any order and each candidate's chain of products on the way of
// the next. 36 k nodes, a solid's tiles with up to 2200 candidates: 518 to 225.
// Other ways tried on the first: lanes that own cells by their residues mod 4, 2,
// without barriers, 640 (6.2 FP64 instructions a candidate for 4.9); the terms
// tabulated once per node, 182, and only added here, 672.
constexpr int kDetWarps = 4;    // units (warps) per CTA at most
constexpr int kDetAhead = 4;
constexpr int kDetStage = 32;   // candidates staged at a time, two stages
struct alignas(16) DetStage {
    double ph[3][4];
    double g;
    unsigned box;   // first cell (6 bits an axis), first point (2), points - 1 (2); top bit: none
    unsigned inv;   // 2^15 / points along x and, above it, along y
};
// Shared memory of one warp: the accumulator of the largest tile + staging.
__host__ __device__ inline size_t det_warp_bytes(int max_edge)
{
    const size_t e3 = (size_t)max_edge * max_edge * max_edge;
    return ((e3 + 1) & ~(size_t)1) * sizeof(double) + 2 * (kDetStage + kDetAhead) * sizeof(DetStage);
}

static __global__ void __launch_bounds__(32 * kDetWarps) spread_det_warp_kernel(DevBatch b, DevGrid g, DevWork w,
                                                                              const double *__restrict__ F,
                                                                              double *__restrict__ f, int density)
{
    extern __shared__ __align__(16) unsigned char det_smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    DetStage *stages = reinterpret_cast<DetStage *>(det_smem + wid * det_warp_bytes(g.max_edge));
    double *acc = reinterpret_cast<double *>(stages + 2 * (kDetStage + kDetAhead));
    const long long N = b.N;
    const ActiveTiles active(w);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        status_add(w.status, ST_PAIRS, (unsigned long long)w.cand_off[g.n_tiles]);
        status_add(w.status, ST_ACTIVE, (unsigned long long)active.total);
    }
    const int n_split = 24 * active.count[0], n_units = n_split + 3 * (active.total - active.count[0]);
    const int n_warps = gridDim.x * (blockDim.x >> 5);
    // each warp's first unit is given, long and short ones spread over the SMs
    // evenly; the rest are fetched
    for (int unit = wid * gridDim.x + blockIdx.x; unit < n_units;) {
        const bool split = unit < n_split;
        const int whole = split ? unit >> 3 : unit - (n_split / 8) * 7;   // (place in the list, lattice)
        const int tile = active.tile(g, w, whole / 3), d = whole % 3;
        const TileInfo ti = decode_tile(g, tile);
        const BoxDev &B = g.boxes[ti.box];
        int s[3], e[3];   // the unit's first cell and cells
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int lo = split && (unit >> a & 1) ? ti.edge[a] >> 1 : 0;
            e[a] = (split && !(unit >> a & 1) ? ti.edge[a] >> 1 : ti.edge[a]) - lo;
            s[a] = ti.start[a] + lo;
        }
        const int n = B.n, ex = e[0], ey = e[1], ez = e[2], vol = ex * ey * ez;
        const double scale = density ? B.scale : 1.0;
        double *fd = f + B.grid_off + (long long)d * n * n * n + ((long long)s[2] * n + s[1]) * n + s[0];
        const int beg = w.cand_off[tile], end = w.cand_off[tile + 1];

        // stages candidate node (-1: none) of each lane whose points meet the unit, in
        // order, and then entries without points up to a multiple of kDetAhead; returns
        // their number
        auto issue = [&](int node, DetStage *st) {
            bool in = node >= 0;
            unsigned box = 0, num_a[3] = {1, 1, 1};
            const DetW &W = w.wtab[max(node, 0)];
            if (in) {
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    int r = W.base[a][a == d ? 0 : 1] - s[a];
                    if (r >= e[a])
                        r -= n;
                    // a box of one tile holds all points, past its last cell from the first on
                    const int lo = max(r, 0), k = e[a] == n ? 4 : min(r + 4, e[a]) - lo;
                    in = in && k > 0;
                    num_a[a] = (unsigned)max(k, 1);
                    box |= (unsigned)lo << (6 * a) | (unsigned)((lo - r) & 3) << (18 + 2 * a) |
                           ((num_a[a] - 1) & 3) << (24 + 2 * a);
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, in);
            const int num = __popc(m), slot = __popc(m & ((1u << lane) - 1u));
            if (in) {
                DetStage &S = st[slot];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const double *ph = W.ph[a][a == d ? 0 : 1];
                    cp_async16(smem_u32(&S.ph[a][0]), ph);
                    cp_async16(smem_u32(&S.ph[a][2]), ph + 2);
                }
                S.box = box;
                S.inv = (32768u + num_a[0] - 1) / num_a[0] | ((32768u + num_a[1] - 1) / num_a[1]) << 16;
                S.g = F[d * N + node] * scale;
            }
            if (lane < kDetAhead)
                st[num + lane].box = 1u << 31;
            return num;
        };
        auto node_at = [&](int c) { return c + lane < end ? w.cand_nodes[c + lane] : -1; };
        int num = issue(node_at(beg), stages), ahead = node_at(beg + 32);
        for (int i = lane; i < vol; i += 32) {
            const int x = i % ex, y = i / ex % ey, z = i / (ex * ey);
            acc[i] = fd[((long long)z * n + y) * n + x];
        }
        for (int c = beg, buf = 0; c < end; c += 32, buf ^= 1) {
            const DetStage *st = stages + buf * (kDetStage + kDetAhead);
            const int count = num;
            cp_async_wait_all();
            __syncwarp();
            num = issue(ahead, stages + (buf ^ 1) * (kDetStage + kDetAhead));
            ahead = node_at(c + 64);
            for (int j = 0; j < count; j += kDetAhead) {
                int at[kDetAhead][2];
                double wg[kDetAhead][2];
#pragma unroll
                for (int q = 0; q < kDetAhead; ++q) {
                    at[q][0] = at[q][1] = -1;
                    const DetStage &S = st[j + q];
                    const unsigned box = S.box, inv = S.inv;
                    if (box >> 31)   // the same for the warp
                        continue;
                    const int kx = (box >> 24 & 3) + 1, ky = (box >> 26 & 3) + 1;
                    const int points = kx * ky * (int)((box >> 28 & 3) + 1);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int p = lane + 32 * h;
                        if (p < points) {
                            const int r = (int)(p * (inv & 0xffffu)) >> 15, lz = (int)(r * (inv >> 16)) >> 15;
                            const int lx = p - r * kx, ly = r - lz * ky;
                            int x = (int)(box & 63) + lx, y = (int)(box >> 6 & 63) + ly, z = (int)(box >> 12 & 63) + lz;
                            x -= x >= ex ? ex : 0;   // (a box of one tile)
                            y -= y >= ey ? ey : 0;
                            z -= z >= ez ? ez : 0;
                            at[q][h] = (z * ey + y) * ex + x;
                            const double t = S.ph[0][(box >> 18 & 3) + lx] * S.ph[1][(box >> 20 & 3) + ly];
                            wg[q][h] = (t * S.ph[2][(box >> 22 & 3) + lz]) * S.g;
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < kDetAhead; ++q) {
                    double s0 = 0.0, s1 = 0.0;   // both loads before the stores
                    if (at[q][0] >= 0)
                        s0 = acc[at[q][0]];
                    if (at[q][1] >= 0)
                        s1 = acc[at[q][1]];
                    if (at[q][0] >= 0)
                        acc[at[q][0]] = s0 + wg[q][0];
                    if (at[q][1] >= 0)
                        acc[at[q][1]] = s1 + wg[q][1];
                    __syncwarp();
                }
            }
            __syncwarp();   // the stage is free
        }
        // write back; the unit's FP64 sum of the values it added
        double part = 0.0;
        for (int i = lane; i < vol; i += 32) {
            const int x = i % ex, y = i / ex % ey, z = i / (ex * ey);
            double *p = fd + ((long long)z * n + y) * n + x;
            const double old = *p;
            *p = acc[i];
            part += acc[i] - old;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            part += __shfl_down_sync(0xffffffffu, part, o);
        if (lane == 0) {
            part *= 1.0 / B.scale;
            bool last = true;
            if (split) {   // the octants' sums are added in their order, by the last to finish
                double *parts = w.red_part + 8 * whole;
                parts[unit & 7] = part;
                __threadfence();
                last = atomicAdd(&w.red_done[whole], 1) == 7;
                if (last) {
                    __threadfence();
                    part = 0.0;
                    for (int k = 0; k < 8; ++k)
                        part += __ldcg(&parts[k]);
                }
            }
            if (last)
                w.red_tile[3LL * tile + d] = part;
            unit = n_warps + atomicAdd(&w.counters[2], 1);
        }
        unit = __shfl_sync(0xffffffffu, unit, 0);
    }
}

// ------------------------------------------------------- interp, FP64
// Thread per node, in the oracle's order: acc = acc + ((phi_x*phi_y)*phi_z)*u
// from 0, z-outer, x-inner. Bound by the FP64 pipe (200 warp instructions a
// lattice of 32 nodes). One lattice after the other and 64 threads a CTA: 133 k
// nodes 174 us, 36 k 45, where all three unrolled (their shared stencils kept in
// registers) in CTAs of 256 took 223 and 61.
constexpr int kInterpThreads = 64;
template <typename real, int KER>
__global__ void __launch_bounds__(kInterpThreads) interp_kernel(DevBatch b, DevGrid g, DevWork w,
                                                     const real *__restrict__ u, const real *__restrict__ x,
                                                     real *__restrict__ v, real support, int use_wtab)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= b.N)
        return;
    const int node = (int)idx;
    const InstDev I = b.inst[b.node_inst[node]];
    const BoxDev B = g.boxes[I.box];
    const long long N = b.N;
    const long long n3 = (long long)B.n * B.n * B.n;
    const int n = B.n;
    real xl[3];
    bool finite = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        xl[a] = x[a * N + node];
        finite = finite && isfinite(xl[a]);
    }
    if (!finite) {
        status_add(w.status, ST_DOMAIN, 1);
#pragma unroll
        for (int d = 0; d < 3; ++d)
            v[d * N + node] = xl[0] + xl[1] + xl[2];
        return;
    }
#pragma unroll 1
    for (int d = 0; d < 3; ++d) {
        const real *ud = u + B.grid_off + d * n3;
        real out = real(0);
        if constexpr (KER == 0) {
            real ph[3][4];
            int ix[4], iy[4], iz[4];
            // with use_wtab the stencil comes from the binning's per-node table
            // (det_weights_kernel: the same values, computed once per node)
            const DetW *wt = nullptr;
            if constexpr (std::is_same<real, double>::value)
                wt = use_wtab ? &w.wtab[node] : nullptr;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                long long i0;
                if (wt) {
                    i0 = wt->base[a][a == d ? 0 : 1];
#pragma unroll
                    for (int m = 0; m < 4; ++m)
                        ph[a][m] = (real)wt->ph[a][a == d ? 0 : 1][m];
                } else {
                    int I0;
                    real s = LatCoord<real>::get(I, B, a, xl[a], (real)mac_off(d, a), I0);
                    i0 = I0 + peskin_axis<real>(s, ph[a]);
                }
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    int wi = wrapi(i0 + m, n);
                    if (a == 0) ix[m] = wi;
                    else if (a == 1) iy[m] = wi;
                    else iz[m] = wi;
                }
            }
            real acc = real(0);
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int bb = 0; bb < 4; ++bb)
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        real wgt = (ph[0][a] * ph[1][bb]) * ph[2][c];
                        acc = acc + wgt * ud[((long long)iz[c] * n + iy[bb]) * n + ix[a]];
                    }
            out = acc;
        } else {
            real s[3];
            int I0[3];
#pragma unroll
            for (int a = 0; a < 3; ++a)
                s[a] = LatCoord<real>::get(I, B, a, xl[a], (real)mac_off(d, a), I0[a]);
            int base[3];
            real wt[27];
            if (!mls_weights<real>(s, support, base, wt)) {
                status_add(w.status, ST_DOMAIN, 1);
                out = real(0);
            } else {
                real acc = real(0);
                int J = 0;
#pragma unroll
                for (int c = 0; c < 3; ++c)
#pragma unroll
                    for (int bb = 0; bb < 3; ++bb)
#pragma unroll
                        for (int a = 0; a < 3; ++a, ++J) {
                            long long gi = ((long long)wrapi((long long)I0[2] + base[2] + c, n) * n
                                            + wrapi((long long)I0[1] + base[1] + bb, n)) * n
                                           + wrapi((long long)I0[0] + base[0] + a, n);
                            acc = acc + wt[J] * ud[gi];
                        }
                out = acc;
            }
        }
        v[d * N + node] = out;
    }
}

// ------------------------------------------- interpolation, cell-centred
// S of a cell-centred field with ncomp components (the conformation tensor
// C_J of Sec. "Interpolation Scheme"): all components at ((i,j,k) + 1/2) h.
// Thread per (node, component), component-major (neighbouring threads are
// neighbouring nodes of one component). FP64 in the oracle's order:
// acc = acc + w * c_J from 0, z-outer, x-inner, w = (phi_x * phi_y) * phi_z;
// FP32 Peskin in separable form (x rows, then y, then z). Field layout: box b
// holds ncomp blocks of n_b^3 values from (grid_off_b / 3) * ncomp; out:
// ncomp rows of N.
template <typename real, int KER>
__global__ void __launch_bounds__(256) interp_cc_kernel(DevBatch b, DevGrid g, DevWork w,
                                                        const real *__restrict__ field, int ncomp,
                                                        const real *__restrict__ x, real *__restrict__ out,
                                                        real support)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long N = b.N;
    if (idx >= N * ncomp)
        return;
    const int q = (int)(idx / N);
    const long long node = idx - q * N;
    const InstDev I = b.inst[b.node_inst[node]];
    const BoxDev B = g.boxes[I.box];
    const int n = B.n;
    const long long n3 = (long long)n * n * n;
    const real *cq = field + (B.grid_off / 3) * ncomp + q * n3;
    real xl[3];
    bool finite = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        xl[a] = x[a * N + node];
        finite = finite && isfinite(xl[a]);
    }
    if (!finite) {
        if (q == 0)
            status_add(w.status, ST_DOMAIN, 1);
        out[q * N + node] = xl[0] + xl[1] + xl[2];
        return;
    }
    real acc = real(0);
    if constexpr (KER == 0 && std::is_same<real, float>::value) {
        float ph[3][4];
        int ix[4], iy[4], iz[4];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            int I0;
            const float s = LatCoord<float>::get(I, B, a, xl[a], 0.5f, I0);
            const int base = wrap_near(I0 + peskin_axis_fast(s, ph[a]), n);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                int id = base + m;
                id -= id >= n ? n : 0;
                if (a == 0) ix[m] = id;
                else if (a == 1) iy[m] = id;
                else iz[m] = id;
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float accz = 0.f;
#pragma unroll
            for (int bb = 0; bb < 4; ++bb) {
                const float *row = cq + ((long long)iz[c] * n + iy[bb]) * n;
                float accy = ph[0][0] * __ldg(row + ix[0]);
#pragma unroll
                for (int a = 1; a < 4; ++a)
                    accy += ph[0][a] * __ldg(row + ix[a]);
                accz += ph[1][bb] * accy;
            }
            acc += ph[2][c] * accz;
        }
    } else if constexpr (KER == 0) {
        real ph[3][4];
        int ix[4], iy[4], iz[4];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            int I0;
            real s = LatCoord<real>::get(I, B, a, xl[a], real(0.5), I0);
            long long i0 = peskin_axis<real>(s, ph[a]);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                int wi = wrapi(I0 + i0 + m, n);
                if (a == 0) ix[m] = wi;
                else if (a == 1) iy[m] = wi;
                else iz[m] = wi;
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int bb = 0; bb < 4; ++bb)
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    real wgt = (ph[0][a] * ph[1][bb]) * ph[2][c];
                    acc = acc + wgt * cq[((long long)iz[c] * n + iy[bb]) * n + ix[a]];
                }
    } else {
        real s[3];
        int I0[3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
            s[a] = LatCoord<real>::get(I, B, a, xl[a], real(0.5), I0[a]);
        int base[3];
        real wt[27];
        if (!mls_weights<real>(s, support, base, wt)) {
            if (q == 0)
                status_add(w.status, ST_DOMAIN, 1);
            out[q * N + node] = real(0);
            return;
        }
        int J = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int bb = 0; bb < 3; ++bb)
#pragma unroll
                for (int a = 0; a < 3; ++a, ++J) {
                    long long gi = ((long long)wrapi((long long)I0[2] + base[2] + c, n) * n
                                    + wrapi((long long)I0[1] + base[1] + bb, n)) * n
                                   + wrapi((long long)I0[0] + base[0] + a, n);
                    acc = acc + wt[J] * cq[gi];
                }
    }
    out[q * N + node] = acc;
}

// ------------------------------------------------------------- reductions
// Block per instance: FP64 sums in a fixed order (per-thread strided sums,
// then a fixed shared-memory tree). Layout: 12 doubles per instance.
template <int NT>
__device__ inline double block_sum(double v, double *sh)
{
    sh[threadIdx.x] = v;
    __syncthreads();
#pragma unroll
    for (int s = NT / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    double r = sh[0];
    __syncthreads();
    return r;
}

// One launch for all conservation sums. Blocks [0, n_inst): one instance
// each -- partial sums of x, F, v and x (x) F (about the instance's local
// origin) per thread, float pairs for FP32 inputs (FP64 for FP64 inputs),
// then a fixed-order tree: FP32 partials are transposed through shared
// memory so that each warp reduces one or two quantities in float pairs and
// converts once to FP64. Torque about the centroid:
// sum (x - c) x F = sum x x F - c x sum F.
// Blocks [n_inst, n_inst + 3 n_boxes): box b, lattice d -- h^3 * sum of the
// values the last spread added, from the per-tile FP64 partials in tile order.
// parts selects what one launch writes: 1 the x/F sums (centroid, sum F,
// torque: entries 0..8), 2 sum v (entries 9..11) and the box blocks, 3 all;
// the sums of one quantity do not depend on parts.

constexpr int kReduceThreads = 256;

// Float-pair partials of one node's x, F and x (x) F terms (the x/F sums).
__device__ __forceinline__ void df_add_xF(DF q[9], const float xk[3], const float Fk[3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        df_add(q[a], xk[a]);
        df_add(q[3 + a], Fk[a]);
    }
    df_add_prod(q[6], xk[1], Fk[2]);
    df_add_prod(q[6], -xk[2], Fk[1]);
    df_add_prod(q[7], xk[2], Fk[0]);
    df_add_prod(q[7], -xk[0], Fk[2]);
    df_add_prod(q[8], xk[0], Fk[1]);
    df_add_prod(q[8], -xk[1], Fk[0]);
}

// Fixed-order total of kReduceThreads float-pair partials (one warp: lane
// sums over a stride of 32, then a shuffle tree); the value is in lane 0.
__device__ __forceinline__ double df_row_total(const float2 *row, int lane)
{
    DF s{0.f, 0.f};
    for (int k = lane; k < kReduceThreads; k += 32) {
        const float2 e = row[k];
        df_add_df(s, DF{e.x, e.y});
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const DF y{__shfl_down_sync(0xffffffffu, s.hi, o), __shfl_down_sync(0xffffffffu, s.lo, o)};
        df_add_df(s, y);
    }
    return (double)s.hi + (double)s.lo;
}

// Entries 0..8 of a particle's sums from the totals of x, F and x (x) F:
// centroid, sum F, torque about the centroid, sum (x - c) x F = sum x x F - c x sum F.
__device__ __forceinline__ void write_xF_sums(double *o, const double *tot, int n_nodes)
{
    const double c[3] = {tot[0] / n_nodes, tot[1] / n_nodes, tot[2] / n_nodes};
    const double *S = tot + 3;
    o[0] = c[0];
    o[1] = c[1];
    o[2] = c[2];
    o[3] = S[0];
    o[4] = S[1];
    o[5] = S[2];
    o[6] = tot[6] - (c[1] * S[2] - c[2] * S[1]);
    o[7] = tot[7] - (c[2] * S[0] - c[0] * S[2]);
    o[8] = tot[8] - (c[0] * S[1] - c[1] * S[0]);
}

template <typename real>
__global__ void __launch_bounds__(kReduceThreads) reduce_kernel(DevBatch b, DevGrid g,
                                                               const double *__restrict__ red_tile,
                                                               const real *__restrict__ x,
                                                               const real *__restrict__ F,
                                                               const real *__restrict__ v, double *__restrict__ red,
                                                               int parts)
{
    __shared__ double sh[kReduceThreads];
    __shared__ double tot[12];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (blockIdx.x >= b.n_inst) {
        const int k = blockIdx.x - b.n_inst, bx = k / 3, d = k - 3 * bx;
        const BoxDev B = g.boxes[bx];
        const long long nt = (long long)B.T * B.T * B.T;
        double s = 0.0;
        for (long long t = threadIdx.x; t < nt; t += blockDim.x)
            s += red_tile[3 * (B.tile_base + t) + d];
        const double r = block_sum<kReduceThreads>(s, sh);
        if (threadIdx.x == 0) {
            double *o = red + 12LL * b.n_inst + 6LL * bx;
            o[d] = r;
            o[3 + d] = 0.0;
        }
        return;
    }
    const InstDev I = b.inst[blockIdx.x];
    const long long N = b.N;
    if constexpr (std::is_same<real, float>::value) {
        __shared__ float2 part[12][kReduceThreads];
        DF q[12];
#pragma unroll
        for (int i = 0; i < 12; ++i)
            q[i] = DF{0.f, 0.f};
        if (parts & 1) {
#pragma unroll 4
            for (int k = threadIdx.x; k < I.n_nodes; k += blockDim.x) {
                const int node = I.node_off + k;
                float xk[3], Fk[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    xk[a] = x[a * N + node];
                    Fk[a] = F ? F[a * N + node] : 0.f;
                }
                df_add_xF(q, xk, Fk);
            }
        }
        if ((parts & 2) && v) {
#pragma unroll 4
            for (int k = threadIdx.x; k < I.n_nodes; k += blockDim.x) {
                const int node = I.node_off + k;
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    df_add(q[9 + a], v[a * N + node]);
            }
        }
#pragma unroll
        for (int i = 0; i < 12; ++i)
            part[i][threadIdx.x] = make_float2(q[i].hi, q[i].lo);
        __syncthreads();
        for (int i = wid; i < 12; i += nw) {
            const bool want = i < 9 ? (parts & 1) != 0 : (parts & 2) != 0;
            if (!want)
                continue;
            const double t = df_row_total(part[i], lane);
            if (lane == 0)
                tot[i] = t;
        }
    } else {
        double p[12];
#pragma unroll
        for (int i = 0; i < 12; ++i)
            p[i] = 0.0;
        for (int k = threadIdx.x; k < I.n_nodes; k += blockDim.x) {
            const int node = I.node_off + k;
            if (parts & 1) {
                double xk[3], Fk[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    xk[a] = (double)x[a * N + node];
                    Fk[a] = F ? (double)F[a * N + node] : 0.0;
                    p[a] += xk[a];
                    p[3 + a] += Fk[a];
                }
                p[6] += xk[1] * Fk[2] - xk[2] * Fk[1];
                p[7] += xk[2] * Fk[0] - xk[0] * Fk[2];
                p[8] += xk[0] * Fk[1] - xk[1] * Fk[0];
            }
            if (parts & 2) {
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    p[9 + a] += v ? (double)v[a * N + node] : 0.0;
            }
        }
#pragma unroll
        for (int i = 0; i < 12; ++i) {
            double t = p[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                t += __shfl_down_sync(0xffffffffu, t, o);
            if (lane == 0)
                sh[i * 8 + wid] = t;
        }
        __syncthreads();
        if (threadIdx.x < 12) {
            double t = 0.0;
            for (int k = 0; k < nw; ++k)
                t += sh[threadIdx.x * 8 + k];
            tot[threadIdx.x] = t;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double *o = red + 12LL * blockIdx.x;
        if (parts & 1)
            write_xF_sums(o, tot, I.n_nodes);
        if (parts & 2) {
            o[9] = tot[9];
            o[10] = tot[10];
            o[11] = tot[11];
        }
    }
}

}  // namespace ifem
