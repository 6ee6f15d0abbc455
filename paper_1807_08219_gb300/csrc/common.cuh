// common.cuh -- device-side data layout and helpers shared by the libifem
// kernels (internal; not part of the C ABI).
//
// Data layout in device memory
//   node arrays   SoA: component a of node k at arr[a*N + k]
//   instances     InstDev[n_inst]: template, box, first node, first element,
//                 FP64 origin and its split origin*(n/L) = I0 + f0 (FP32 mode)
//   templates     TmplDev[n_tmpl]: element connectivity, reference data
//                 (FP64 and an FP32 copy), node->element incidence CSR
//   boxes         BoxDev[n_boxes]: cells per side, tiles, field offset
//   grid field    per box: 3 lattices of n^3 values, x fastest
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ifem {

constexpr int kMaxTileEdge = 20;   // tile edge t + 4 at most (t <= 16)
constexpr int kOwnSub = 5;         // own-list sub-blocks (4 cells) per tile axis (tile edge <= 20)
constexpr int kOwnSub3 = kOwnSub * kOwnSub * kOwnSub;
constexpr int kScanThreads = 512;  // tile-count scan: threads per block
constexpr int kScanPer = 4;        // and values per thread
constexpr int kScanBlock = kScanThreads * kScanPer;
constexpr int kTileClasses = 4;    // DevWork::active lists
constexpr int kFsumBins = 8;       // DevWork::tile_fbin entries per sum
constexpr int kCounters = 16;      // DevWork::counters entries
constexpr int kMaxCtaSmemBytes = 227 * 1024;   // opt-in dynamic shared memory of one CTA
// FP32 nodal force kernel: a float4 (position, mean curvature) of shared
// memory per template node, 16-bit node ids
constexpr int kNodalMaxNodes = kMaxCtaSmemBytes / 16;
constexpr int kNodBits = 14, kNodMask = (1 << kNodBits) - 1;   // node id bits in the first id of an incidence
static_assert(kNodalMaxNodes <= kNodMask + 1, "node ids of the nodal kernel");
constexpr double kObtuseSum = 2.5, kObtuseMost = 64.0;   // forces.cuh, nodal path
__host__ __device__ inline size_t nodal_smem_bytes(int n_nodes) { return (size_t)n_nodes * sizeof(float4); }
constexpr int kStatusWords = 8;
enum StatusWord {
    ST_INVERTED = 0,
    ST_DOMAIN = 1,
    ST_CAPACITY = 2,
    ST_TIMEOUT = 3,
    ST_PAIRS = 4,
    ST_ACTIVE = 5,
    ST_TOUCHED = 6,
};

struct TmplDev {
    int kind;        // 0 membrane (triangles), 1 solid (tetrahedra)
    int law;         // membrane law (0 neo-Hookean, 1 Skalak)
    int n_nodes;
    int n_elems;
    const int *elems;      // 3 or 4 node ids per element (template-local)
    const double *ref_d;   // membrane: [m00 m01 m10 m11 A0]; solid: [M (3x3 row-major), V0]
    const float *ref_f;    // FP32 copy of ref_d
    const int *inc_off;    // n_nodes + 1: incidence CSR offsets
    const int *inc_idx;    // element*4 + local vertex, ascending element id
    const int2 *ring;      // membranes: per incidence, the other two vertices (j, k) of the
                           // triangle in its orientation order starting at the vertex
    // FP32 nodal force kernel (templates of at most kNodalMaxNodes nodes, else null): incidences in
    // slices of 32 nodes, slot s of node k at nod_off[k / 32] + 32 s + k % 32
    const int *nod_off;
    const float4 *nod_ref;   // membranes: reference edge dots r_a, r_b, r_c and 1/(2 A0); solids: h of the
                             // corners, 1/(6 V0) in the node's own place
    const void *nod_idx;     // membranes: ushort2 (j, l); solids: ushort4, the corners; the node's corner
                             // number in the bits of the first id above kNodBits
    double mu, C, kb, c0, lam;
    float vol_scale;         // power of two near 1 over the template's extent
    float mu_f, half_muD_f, kb_f, kH0_f, half_lam_f;   // FP32 nodal kernel: mu, C mu/2, kb, -c0/2, lam/2
};

struct InstDev {
    int tmpl;
    int box;
    int node_off;
    int n_nodes;
    long long elem_off;    // first element of this instance in element buffers
    int n_elems;
    int pad;
    double origin[3];
    int I0[3];             // floor(origin * n/L)      (FP32 transfer)
    float f0[3];           // origin * n/L - I0        (FP32 transfer)
};

struct BoxDev {
    int n;           // cells per side
    int t;           // nominal tile edge
    int T;           // tiles per axis (last tile absorbs the remainder, edge <= t + 4)
    int pad;
    long long tile_base;
    long long grid_off;    // offset of this box's first value in a grid field
    double L;
    double inv_h;          // n / L
    double scale;          // (n/L)^3
    double h3;             // 1 / scale
    float inv_h_f;         // FP32 copies for the FP32 kernels (no FP64 pipe use), and
    float inv_h_lo;        // what inv_h_f rounds off
    float scale_f;
};

struct DevBatch {
    int n_inst;
    int n_tmpl;
    long long N;
    int max_nodes;
    int max_elems;
    long long n_elems_total;
    int any_bending;       // some membrane template has kb != 0
    int nodal_ok;          // every template fits the FP32 nodal force kernel
    int any_obtuse;        // and some need its OBTUSE form
    const InstDev *inst;
    const TmplDev *tmpl;
    const int *node_inst;
    const int *inst_order; // instances by decreasing force work (the force kernel's CTAs: small ones fill the tail)
};

struct DevGrid {
    int n_boxes;
    long long n_tiles;
    int max_edge;
    const BoxDev *boxes;
};

// FP64 Peskin stencil of a node: along each axis of the two offsets its
// lattices have there (0 for the lattice of that component, 1/2 for the other
// two), the wrapped first index and the four weights.
struct alignas(16) DetW {
    double ph[3][2][4];
    int base[3][2];
    int pad[2];
};
static_assert(sizeof(DetW) == 224, "DetW layout");

// A tile with own nodes (FP32), as the transfer needs it.
struct alignas(16) TileDesc {
    int tile, n, beg, end;   // tile number, cells per box side, own records [beg, end)
    int start[3], edge[3];   // first cell and cells per axis
    long long grid_off;      // the box's offset in a grid field
    double h3;               // (L/n)^3
    float scale_f;           // (n/L)^3
    int slot;                // its place in the list
};
static_assert(sizeof(TileDesc) == 64, "TileDesc layout");

// FP32 tile transfer: width of the shared boxes in y and z (4 more in x) for
// tiles of at most max_edge cells, and bytes of a box.
__host__ __device__ inline int tile_width(int max_edge) { return max_edge <= 8 ? 12 : (max_edge <= 12 ? 16 : 20); }
__host__ __device__ inline size_t tile_box_bytes(int max_edge)
{
    const size_t w = tile_width(max_edge);
    return 4 * (w + 4) * w * w;
}
struct DevWork {
    int *cand_count;    // n_tiles + 1
    int *cand_off;      // n_tiles + 1
    int *cand_cursor;   // n_tiles
    int *cand_nodes;    // pair list: node id per (tile, node) candidate pair
    long long cand_cap;
    int *own_count;     // FP32, per (tile, 4^3 sub-block): n_tiles * kOwnSub3 + 1; then own_flag and
                        // tile_fsum. One piece with red_tile and counters before it (FP64: cand_count
                        // and red_done follow those)
    int *own_flag;      // n_tiles (FP32): 1 where the tile owns a node
    float *tile_fsum;   // 3 per tile (FP32): sum of |F_d| over the tile's own nodes, from the
                        // placement when it is given the forces (the transfer's fixed-point scale)
    unsigned long long *tile_fbin;   // the same for the reproducible spread: kFsumBins integers each
    int *own_cursor;    // FP32: offsets of the own lists within their scan block
    float4 *own_rec;    // FP32, 2 per node, by tile and sub-block: fractional cell coordinates
                        // x, y, z of the node and, in w, its cell within the tile packed as 8-bit
                        // x | y << 8 | z << 16; its force and, in w, its id
    int2 *node_key;     // N entries, by node (FP32): own-list key (-1: not binned) and
                        // the node's rank among the nodes of that key
    float4 *node_rec;   // N entries, by node (FP32): the first float4 of its own_rec entry
    int *active;        // tiles with candidate pairs, kTileClasses lists of n_tiles entries
    TileDesc *tile_desc;  // tiles with own nodes (FP32), counters[3] of them
    int *tile_slot;     // n_tiles (FP32): a tile's place in that list, or -1
    int2 *near_tile;    // reproducible spread: tiles that a box reaches and their boxes, counters[9] of them
    float *box_buf;     // reproducible spread: a box per listed tile and, with box_lattices = 3, lattice;
    int box_lattices;   // with 1 the lattices take it in turn
    int *counters;      // kCounters: [2] work counter, [3] tiles with own nodes,
                        // [4] total pairs (FP64), [5] total own nodes (FP32), [1] [6] [7] work counters of
                        // one-lattice launches, [8] scan blocks finished, [9] near_tile entries,
                        // [10] to [13] active tiles per class
    int *scan_blocks;   // block partial sums for the tile scan
    void *elem_buf;     // per element nodal forces (12 reals per element)
    void *bend_buf;     // per node bending scratch (A, kH, n[3], lap) 6 reals
    double *red_part;   // FP64 Peskin: 8 octants' sums per long list and lattice, and
    int *red_done;      // how many of them are there
    double *red_tile;   // per tile: 3 FP64 sums of added spread values
    size_t zero_bytes;  // counters and what follows them (cleared by every binning)
    DetW *wtab;         // N entries (FP64 Peskin only, else null): written by the binning
    unsigned long long *status;  // kStatusWords
};

// ---------------------------------------------------------------- helpers
__host__ __device__ inline int wrapi(long long i, int n)
{
    long long m = i % n;
    return (int)(m < 0 ? m + n : m);
}

// Tile of a (wrapped) cell along one axis: tiles of edge t, the last one
// absorbing the remainder.
__host__ __device__ inline int tile_of(int c, int t, int T)
{
    int j = c / t;
    return j < T - 1 ? j : T - 1;
}
__host__ __device__ inline int tile_start(int j, int t) { return j * t; }
__host__ __device__ inline int tile_edge(int j, int t, int T, int n) { return j < T - 1 ? t : n - j * t; }

// Tiles per axis for a box of n cells and nominal tile edge t: every tile has
// at least 5 cells (so 5 consecutive cells meet at most 2 tiles) and at most
// t + 4.
__host__ __device__ inline int tiles_per_axis(int n, int t)
{
    int T = (n + t - 1) / t;
    int r = n - (T - 1) * t;
    if (T > 1 && r < 5)
        T -= 1;
    return T;
}

// Adams-Bashforth position update of one value (Eq. Bashforth_eqn),
// x + dt*(1.5*v - 0.5*vp) rounded operation by operation in this order (no
// contraction into FMAs), so every kernel that takes it gives the same bits.
__device__ __forceinline__ float ab2_value(float x, float v, float vp, float dt)
{
    return __fadd_rn(x, __fmul_rn(dt, __fsub_rn(__fmul_rn(1.5f, v), __fmul_rn(0.5f, vp))));
}
__device__ __forceinline__ double ab2_value(double x, double v, double vp, double dt)
{
    return __dadd_rn(x, __dmul_rn(dt, __dsub_rn(__dmul_rn(1.5, v), __dmul_rn(0.5, vp))));
}

// Reductions into shared memory addressed by 32-bit shared-window offsets
// (no generic-to-shared address check per access).
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void red_shared_add(unsigned a, int v)
{
    asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void red_shared_add(unsigned a, float v)
{
    asm volatile("red.shared.add.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

__device__ inline void status_add(unsigned long long *st, int w, unsigned long long v)
{
    if (v)
        atomicAdd(st + w, v);
}

// 4-point discrete delta (Peskin 2002), evaluation order fixed:
//   a = |r|, q = 4a; |r| <= 1: ((3 - 2a) + sqrt((1 + q) - q*a)) * 0.125
//   1 < |r| <= 2: ((5 - 2a) - sqrt(((12a) - 7) - q*a)) * 0.125
template <typename real>
__device__ __forceinline__ real phi4(real r)
{
    real a = r < real(0) ? -r : r;
    real q = real(4) * a;
    if (a <= real(1)) {
        real t = (real(1) + q) - q * a;
        return ((real(3) - real(2) * a) + sqrt(t)) * real(0.125);
    }
    if (a <= real(2)) {
        real t = ((real(12) * a) - real(7)) - q * a;
        return ((real(5) - real(2) * a) - sqrt(t)) * real(0.125);
    }
    return real(0);
}

// MLS cubic-spline weight W(r) (Sec. "Interpolation Scheme"; first branch
// read as 2/3 - 4r^2 + 4r^3, continuous at r = 1/2).
template <typename real>
__device__ __forceinline__ real mls_w(real r)
{
    if (r <= real(0.5))
        return real(2.0 / 3.0) - real(4) * r * r + real(4) * r * r * r;
    if (r <= real(1))
        return real(4.0 / 3.0) - real(4) * r + real(4) * r * r - real(4.0 / 3.0) * r * r * r;
    return real(0);
}

// Linear MLS weights at one point: s = lattice coordinates (3), support in
// cells. base = floor(s + 1/2) - 1 (unwrapped). w[27] in z-outer, x-inner
// order. Returns false if the 4x4 moment matrix is not positive definite.
template <typename real>
__device__ inline bool mls_weights(const real s[3], real support, int base[3], real w[27])
{
    real A[10];   // packed lower triangle of the symmetric 4x4 moment matrix
#pragma unroll
    for (int i = 0; i < 10; ++i)
        A[i] = real(0);
    for (int a = 0; a < 3; ++a)
        base[a] = (int)floor(s[a] + real(0.5)) - 1;
    int J = 0;
    for (int kz = 0; kz < 3; ++kz)
        for (int jy = 0; jy < 3; ++jy)
            for (int ix = 0; ix < 3; ++ix, ++J) {
                real y0 = real(base[0] + ix) - s[0];
                real y1 = real(base[1] + jy) - s[1];
                real y2 = real(base[2] + kz) - s[2];
                real Wj = mls_w(sqrt(y0 * y0 + y1 * y1 + y2 * y2) / support);
                w[J] = Wj;
                real p[4] = {real(1), y0, y1, y2};
                int q = 0;
                for (int r = 0; r < 4; ++r)
                    for (int c = 0; c <= r; ++c, ++q)
                        A[q] += Wj * p[r] * p[c];
            }
    // Cholesky of the packed matrix, then solve A z = e1.
    real Lm[10];
    int q = 0;
    for (int r = 0; r < 4; ++r)
        for (int c = 0; c <= r; ++c, ++q) {
            real acc = A[q];
            for (int k = 0; k < c; ++k)
                acc -= Lm[r * (r + 1) / 2 + k] * Lm[c * (c + 1) / 2 + k];
            if (r == c) {
                if (!(acc > real(0)))
                    return false;
                Lm[q] = sqrt(acc);
            } else {
                Lm[q] = acc / Lm[c * (c + 1) / 2 + c];
            }
        }
    real y[4], z[4];
    for (int r = 0; r < 4; ++r) {
        real acc = r == 0 ? real(1) : real(0);
        for (int k = 0; k < r; ++k)
            acc -= Lm[r * (r + 1) / 2 + k] * y[k];
        y[r] = acc / Lm[r * (r + 1) / 2 + r];
    }
    for (int r = 3; r >= 0; --r) {
        real acc = y[r];
        for (int k = r + 1; k < 4; ++k)
            acc -= Lm[k * (k + 1) / 2 + r] * z[k];
        z[r] = acc / Lm[r * (r + 1) / 2 + r];
    }
    J = 0;
    for (int kz = 0; kz < 3; ++kz)
        for (int jy = 0; jy < 3; ++jy)
            for (int ix = 0; ix < 3; ++ix, ++J) {
                real y0 = real(base[0] + ix) - s[0];
                real y1 = real(base[1] + jy) - s[1];
                real y2 = real(base[2] + kz) - s[2];
                w[J] = w[J] * (z[0] + z[1] * y0 + z[2] * y1 + z[3] * y2);
            }
    return true;
}

// Lattice coordinate of node k along axis a for MAC component d.
//   FP64: s = (origin + x) * (n/L) - o, I0 = 0  (exact order of the oracle)
//   FP32: s = (f0 - o) + x * (n/L) relative to the integer offset I0
template <typename real>
struct LatCoord;

template <>
struct LatCoord<double> {
    __device__ static inline double get(const InstDev &I, const BoxDev &B, int a, double x, double o, int &I0)
    {
        I0 = 0;
        double p = I.origin[a] + x;
        return p * B.inv_h - o;
    }
};

template <>
struct LatCoord<float> {
    __device__ static inline float get(const InstDev &I, const BoxDev &B, int a, float x, float o, int &I0)
    {
        I0 = I.I0[a];
        return (I.f0[a] - o) + x * B.inv_h_f;
    }
};

// x + y as a sum and its error
__device__ __forceinline__ float two_sum(float x, float y, float &err)
{
    const float s = x + y, b = s - x;
    err = (x - (s - b)) + (y - b);
    return s;
}

// ------------------------------------------------------------- launchers
// Launch parameters that depend on the device only, asked for once per context (0: not yet).
struct LaunchCache {
    int tile_ctas[2][3][2][2][2];   // transfer_tile_kernel<KER, W, SPREAD, INTERP, STORE>: resident CTAs per SM
    int wide_ctas[2][3];            // spread_wide_kernel<KER, W>
    int nodal[2][2], volume, vcorr, det_warp;   // forces_nodal_f32_kernel<CLUSTER, OBTUSE>, volume_f32_kernel,
                                    // vc_fused_f32_kernel, spread_det_warp_kernel: shared memory allowed
};

struct ForcesArgs {
    LaunchCache *cache;
    DevBatch b;
    DevWork w;
    const void *x;
    void *F;
    const void *wv;   // HVP direction (or null)
    int n_sm;
    int hvp;          // 1: compute Hw instead of F
    int inst0, inst_n;  // particle range [inst0, inst0 + inst_n) (inst_n = 0: all); the FP32
                        // nodal kernel only (forces_ranged_ok)
    cudaStream_t stream;
};

struct TransferArgs {
    LaunchCache *cache;
    DevBatch b;
    DevGrid g;
    DevWork w;
    const void *x;
    const void *F;
    const void *u;
    void *f;
    void *v;
    int kernel;       // 0 Peskin4, 1 MLS27
    int density;
    double support;
    int n_sm;
    int store;        // FP32: reproducible spread through the boxes of every tile
    int acc64;        // with 64-bit accumulators
    int cleared;      // f is zero before the spread (else the reproducible spread adds to it)
    int clear_f;      // the binning clears f too
    long long total;  // values of the grid
    int clear_sums;   // binning: a spread follows, clear its per-tile sums too
    int lattice;      // tile transfer: -1 all three lattices, else that lattice only
    int pdl;          // tile transfer: may start before the previous kernel in the stream ends
    int use_wtab;     // FP64 Peskin interpolation: read the stencils the binning of x tabulated
    const void *vp;   // fused position update (halo spread + interpolation only):
    void *xn;         //   xn = x + dt (3/2 v - 1/2 vp) when xn is not null
    double dt;
    cudaStream_t stream;
};

struct ReduceArgs {
    DevBatch b;
    DevGrid g;
    DevWork w;
    const void *x;
    const void *F;
    const void *v;
    double *red;
    int parts;        // 1: per-particle x/F sums; 2: per-particle sum v and the per-box sums; 3: all
    cudaStream_t stream;
};

// Defined once per precision in kernels_f32.cu / kernels_f64.cu.
cudaError_t launch_forces_f32(const ForcesArgs &a);
cudaError_t launch_forces_f64(const ForcesArgs &a);
// Binning in two parts: the clears, the count pass and the scan, then the
// placement (which also sums |F| per tile when TransferArgs::F is given).
// Only the FP32 binning takes them apart.
enum BinStage { BIN_COUNT = 1, BIN_PLACE = 2, BIN_ALL = 3 };
cudaError_t launch_bin_f32(const TransferArgs &a, int stages = BIN_ALL);
cudaError_t launch_bin_f64(const TransferArgs &a, int stages = BIN_ALL);
cudaError_t launch_spread_f32(const TransferArgs &a);
cudaError_t launch_spread_f64(const TransferArgs &a);
cudaError_t launch_interp_f32(const TransferArgs &a);
cudaError_t launch_interp_f64(const TransferArgs &a);
cudaError_t launch_reduce_f32(const ReduceArgs &a);
cudaError_t launch_reduce_f64(const ReduceArgs &a);

// Fluid-stress forces inside solids: F = (F +) sum of element contributions.
struct FluidArgs {
    DevBatch b;
    DevWork w;
    const void *x;
    const void *u;
    const void *C;    // 6 rows of N, or null
    double eta;
    double cp;        // eta (1 - beta) / lambda
    int add;          // 1: F = F + fluid forces
    void *F;
    cudaStream_t stream;
};
cudaError_t launch_fluid_f32(const FluidArgs &a);
cudaError_t launch_fluid_f64(const FluidArgs &a);
// Cell-centred multi-component interpolation (TransferArgs.u = field).
cudaError_t launch_interp_cc_f32(const TransferArgs &a, int ncomp);
cudaError_t launch_interp_cc_f64(const TransferArgs &a, int ncomp);

// Lagrangian update: AB2 positions, volumes, membrane volume correction.
struct LagrangeArgs {
    LaunchCache *cache;
    DevBatch b;
    void *x;
    void *x_out;      // AB2 result (null: in place)
    const void *v;
    const void *vp;
    double dt;
    const double *V0;
    double *out;      // volumes, or Lambda per instance (may be null for the correction)
    double *alpha;    // 3 doubles per node of scratch (correction)
    unsigned long long *status;
    cudaStream_t stream;
};
cudaError_t launch_ab2_f32(const LagrangeArgs &a);
cudaError_t launch_ab2_f64(const LagrangeArgs &a);
cudaError_t launch_volume_f32(const LagrangeArgs &a);
cudaError_t launch_volume_f64(const LagrangeArgs &a);
cudaError_t launch_vcorr_f32(const LagrangeArgs &a);
cudaError_t launch_vcorr_f64(const LagrangeArgs &a);
cudaError_t launch_area_normals_f32(const DevBatch &b, const void *x, void *nA, cudaStream_t s);
cudaError_t launch_area_normals_f64(const DevBatch &b, const void *x, void *nA, cudaStream_t s);

}  // namespace ifem
