// launch_impl.cuh -- host-side launch sequences, instantiated once per
// precision (kernels_f32.cu with FMA contraction, kernels_f64.cu without).
#pragma once
#include <type_traits>

#include "common.cuh"
#include "forces.cuh"
#include "transfer.cuh"
#include "lagrangian.cuh"

namespace ifem {

#define IFEM_LAUNCH_CHECK()                      \
    do {                                         \
        cudaError_t e_ = cudaGetLastError();     \
        if (e_ != cudaSuccess)                   \
            return e_;                           \
    } while (0)

// Allows a kernel its largest dynamic shared memory, once per context. The limit
// belongs to the function, which all contexts and threads share: set to what one
// launch needs, another thread's smaller batch could lower it before that launch.
template <typename Kernel>
static cudaError_t allow_smem(Kernel kern, size_t largest, int &done)
{
    if (done)
        return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)largest);
    done = e == cudaSuccess;
    return e;
}
// beside the kernels' own arrays (vol_totals)
constexpr size_t kVolSmemBytes = kMaxCtaSmemBytes - 8 * kVolThreadsF - 1024;
constexpr size_t kVcorrSmemBytes = kMaxCtaSmemBytes - 4 * 8 * kVolThreadsF - 1024;

// FP32 nodal forces of particles [inst0, inst0 + n): a cluster of S CTAs per
// particle. With few particles one CTA each leaves most SMs idle; with many,
// each doubling only stages the positions once more. Times in us, S = 1, 2, 4, 8:
//   one red cell (2562 nodes)     31  20  15  11
//   16 balls of 4096 nodes       107  57  31  26
//   64 balls of 4096 nodes       108  57  48  52
//   72 red cells and platelets    32  21  21  34
//   200 capsules of 2562 nodes    50  45  56  83
//   300 red cells                 51  55  82 121
//   600 red cells and platelets   92  97 138 226
// Nodes per thread: as few rounds as 512 threads allow, evenly filled (smaller
// blocks measured slower throughout: 600 particles 102 us with 192 threads).
template <typename real>   // float (a template so that kernels_f64.cu compiles no FP32 kernel)
static cudaError_t launch_nodal_forces(const DevBatch &b, const float *x, float *F, unsigned long long *status,
                                       int inst0, int n, int n_sm, LaunchCache *cache, cudaStream_t s)
{
    const int S = 16 * n <= n_sm ? 8 : (2 * n <= n_sm ? 4 : (2 * n <= 3 * n_sm ? 2 : 1));
    const int chunk = ((b.max_nodes + S - 1) / S + 31) & ~31;
    const int rounds = (chunk + 511) / 512;
    const int threads = ((chunk + rounds - 1) / rounds + 31) & ~31;
    const size_t sm = nodal_smem_bytes(b.max_nodes);
    auto kern = b.any_obtuse ? (S > 1 ? forces_nodal_f32_kernel<true, true> : forces_nodal_f32_kernel<false, true>)
                             : (S > 1 ? forces_nodal_f32_kernel<true, false> : forces_nodal_f32_kernel<false, false>);
    if (cudaError_t e = allow_smem(kern, nodal_smem_bytes(kNodalMaxNodes), cache->nodal[S > 1][b.any_obtuse != 0]))
        return e;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = S;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(n * S));
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = S > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, b, x, F, status, n == b.n_inst ? -1 : inst0, S);
}

template <typename real>
cudaError_t forces_impl(const ForcesArgs &a)
{
    const DevBatch &b = a.b;
    if (b.n_inst == 0)
        return cudaSuccess;
    const real *x = (const real *)a.x;
    real *F = (real *)a.F;
    cudaStream_t s = a.stream;
    if constexpr (std::is_same<real, float>::value) {
        if (!a.hvp && b.nodal_ok) {
            const int n = a.inst_n > 0 ? a.inst_n : b.n_inst;
            if (a.inst0 < 0 || a.inst0 + n > b.n_inst)
                return cudaErrorInvalidValue;
            return launch_nodal_forces<real>(b, x, F, a.w.status, a.inst0, n, a.n_sm, a.cache, s);
        }
    }
    if (a.inst0 != 0 || (a.inst_n != 0 && a.inst_n != b.n_inst))
        return cudaErrorInvalidValue;   // particle ranges: the nodal kernel only
    dim3 blk(256);
    dim3 ge((b.max_elems + 255) / 256, b.n_inst);
    dim3 gn((b.max_nodes + 255) / 256, b.n_inst);
    real *ebuf = (real *)a.w.elem_buf;
    if (a.hvp)
        elem_force_kernel<real, true><<<ge, blk, 0, s>>>(b, x, (const real *)a.wv, ebuf, a.w.status);
    else
        elem_force_kernel<real, false><<<ge, blk, 0, s>>>(b, x, nullptr, ebuf, a.w.status);
    IFEM_LAUNCH_CHECK();
    node_gather_kernel<real><<<gn, blk, 0, s>>>(b, ebuf, F);
    IFEM_LAUNCH_CHECK();
    if (!a.hvp && b.any_bending) {
        real *bb = (real *)a.w.bend_buf;
        bend_tri_kernel<real><<<ge, blk, 0, s>>>(b, x, ebuf);
        IFEM_LAUNCH_CHECK();
        bend_pass1_kernel<real><<<gn, blk, 0, s>>>(b, x, ebuf, bb);
        IFEM_LAUNCH_CHECK();
        bend_pass2_kernel<real><<<gn, blk, 0, s>>>(b, ebuf, bb, F);
        IFEM_LAUNCH_CHECK();
    }
    return cudaSuccess;
}

// Launch whose start overlaps the end of the kernel before it in the stream (the
// kernel itself waits, pdl_wait): of a small step's chain of short kernels the
// launches gaps, 1 to 3 us each, are a quarter (one capsule, 64^3: 42 us, 32
// with the whole chain launched so).
template <typename... P, typename... A>
cudaError_t launch_after(void (*kern)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t s, A... args)
{
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

// Binning. FP32: one-pass own lists (count, scan, placement; the stages can be
// launched apart). FP64: candidate lists, sorted, and the Peskin stencil table.
template <typename real>
cudaError_t bin_impl(const TransferArgs &a, int stages)
{
    const DevBatch &b = a.b;
    const DevWork &w = a.w;
    const long long nt = a.g.n_tiles;
    cudaStream_t s = a.stream;
    constexpr bool f32 = std::is_same<real, float>::value;
    if (!f32 && stages != BIN_ALL)
        return cudaErrorInvalidValue;
    const bool empty = b.n_inst == 0 || b.N == 0;
    dim3 gn((b.max_nodes + 255) / 256, b.n_inst);
    // one-pass binning: kBinPer nodes per thread
    dim3 g1((b.max_nodes + 256 * kBinPer - 1) / (256 * kBinPer), b.n_inst);
    if (stages & BIN_COUNT) {
        // one clear: the counters, counts and per-tile |F| sums, and before them
        // the spread's per-tile sums
        const size_t sums = a.clear_sums ? sizeof(double) * 3 * (size_t)nt : 0;
        const size_t words = (sums + w.zero_bytes) / sizeof(int);
        cudaError_t e = cudaSuccess;
        const size_t f_words = a.clear_f ? (size_t)a.total * sizeof(real) / sizeof(int) : 0;
        clear_kernel<<<(unsigned)std::min<size_t>((words + f_words + 255) / 256, 8 * a.n_sm), 256, 0, s>>>(
            w.counters - sums / sizeof(int), words, (int *)a.f, f_words);
        IFEM_LAUNCH_CHECK();
        if (empty)
            return cudaSuccess;
        if constexpr (f32) {
            if ((e = launch_after(own_count_kernel, g1, 256, 0, s, b, a.g, w, (const float *)a.x)) != cudaSuccess)
                return e;
        } else {
            bin_kernel<real, false><<<gn, 256, 0, s>>>(b, a.g, w, (const real *)a.x);
            IFEM_LAUNCH_CHECK();
        }
        // FP32: the local offsets go to the cursors (own_scatter_kernel adds the block offsets)
        const long long n = f32 ? nt * kOwnSub3 : nt;
        const unsigned nb = (unsigned)((n + kScanBlock - 1) / kScanBlock);
        if ((e = launch_after(scan_local_kernel, nb, kScanThreads, 0, s, n, f32 ? w.own_count : w.cand_count,
                              f32 ? w.own_cursor : w.cand_off, w.scan_blocks, w.counters + 8,
                              w.counters + (f32 ? 5 : 4))) != cudaSuccess)
            return e;
    }
    if (empty || !(stages & BIN_PLACE))
        return cudaSuccess;
    if constexpr (f32) {
        // enough threads for every tile as well as every node
        const long long per_inst = ((nt + 255) / 256 + b.n_inst - 1) / b.n_inst;
        dim3 gs((unsigned)std::max<long long>(g1.x, per_inst), b.n_inst);
        if (cudaError_t e = launch_after(own_scatter_kernel, gs, 256, 0, s, b, a.g, w, (const float *)a.F, a.store,
                                         (const float *)a.x, (const float *)a.v, (const float *)a.vp, (float *)a.xn,
                                         (float)a.dt))
            return e;
    } else {
        scan_finish_kernel<<<(unsigned)((nt + 1 + 255) / 256), 256, 0, s>>>(nt, w, a.n_sm);
        IFEM_LAUNCH_CHECK();
        bin_kernel<real, true><<<gn, 256, 0, s>>>(b, a.g, w, (const real *)a.x);
        IFEM_LAUNCH_CHECK();
        sort_segments_kernel<<<a.n_sm * 4, 512, 0, s>>>(a.g, w);
        IFEM_LAUNCH_CHECK();
        if (a.kernel == 0 && w.wtab) {
            det_weights_kernel<<<(unsigned)((3 * b.N + 255) / 256), 256, 0, s>>>(b, a.g, w.wtab, (const double *)a.x);
            IFEM_LAUNCH_CHECK();
        }
    }
    return cudaSuccess;
}

// The FP32 tile transfer over the own lists of the binning just before it:
// spreading (SPREAD), interpolation (INTERP) or both. One resident wave of CTAs
// takes the items.
template <int KER, int W, bool SPREAD, bool INTERP, bool STORE>
cudaError_t launch_tile_w(const TransferArgs &a)
{
    auto kern = transfer_tile_kernel<KER, W, SPREAD, INTERP, STORE>;
    constexpr int kKinds = (SPREAD ? 1 : 0) + (INTERP ? 1 : 0), T = TileShape<W>::kThreads;
    const size_t sm = (size_t)4 * TileShape<W>::kWords * 2 * kKinds;
    cudaError_t e = cudaSuccess;
    int &occ = a.cache->tile_ctas[KER][W / 4 - 3][SPREAD][INTERP][STORE];
    if (occ == 0) {
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)) != cudaSuccess)
            return e;
        int ctas = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, kern, T, sm);
        occ = ctas < 1 ? 1 : ctas;
    }
    float *f = (float *)a.f;
    const int add = !a.cleared;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    // programmatic dependent launch: the CTAs of this grid may start once
    // every CTA of the previous kernel in the stream has signalled
    // (griddepcontrol.launch_dependents, at its start); they read nothing it
    // writes
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(a.n_sm * occ);
    cfg.blockDim = dim3(T);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = a.stream;
    cfg.attrs = attr;
    cfg.numAttrs = a.pdl || a.lattice < 0 ? 1 : 0;
    auto transfer = [&](int lattice) {
        return cudaLaunchKernelEx(&cfg, kern, a.b, a.w, (const float *)a.x, f, a.density, (const float *)a.u,
                                  (float *)a.v, (const float *)a.vp, (float *)a.xn, (float)a.dt,
                                  (float)(1.0 / a.support), lattice, add);
    };
    if (!STORE)
        return transfer(a.lattice);
    const size_t wide = a.acc64 ? (size_t)8 * TileShape<W>::kWords : 0;
    auto kwide = spread_wide_kernel<KER, W>;
    int &wide_ctas = a.cache->wide_ctas[KER][W / 4 - 3];
    if (wide && wide_ctas == 0) {
        if ((e = cudaFuncSetAttribute(kwide, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wide)) != cudaSuccess ||
            (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&wide_ctas, kwide, TileShape<W>::kBoxThreads, wide)) !=
                cudaSuccess)
            return e;
        wide_ctas = std::max(wide_ctas, 1);
    }
    // one lattice after the other where the buffer holds the boxes of one: each waits
    // for the combination of the one before
    const bool apart = a.w.box_lattices == 1;
    if (apart)
        cfg.numAttrs = 0;
    const long long units = (apart ? 1 : 3) * std::min<long long>(a.g.n_tiles, 27 * a.b.N);
    const long long blocks = std::min(units, 8LL * a.n_sm);   // all resident
    auto combine = apart ? tile_combine_kernel<W, 1> : tile_combine_kernel<W, 3>;
    for (int d = apart ? 0 : -1; d < (apart ? 3 : 0); ++d)
        if ((e = !wide ? transfer(d)
                       : launch_after(kwide, a.n_sm * wide_ctas, TileShape<W>::kBoxThreads, wide, a.stream, a.w, f,
                                      a.density, (float)(1.0 / a.support), d, add)) != cudaSuccess ||
            (e = launch_after(combine, (unsigned)blocks, kCombineThreads, 0, a.stream, a.g, a.w, f, add,
                              d)) != cudaSuccess)
            return e;
    if constexpr (STORE && INTERP)
        if (wide)
            return launch_tile_w<KER, W, false, true, false>(a);
    return cudaSuccess;
}
template <int KER, bool SPREAD, bool INTERP, bool STORE>
cudaError_t launch_tile(const TransferArgs &a)
{
    switch (tile_width(a.g.max_edge)) {
    case 12:
        return launch_tile_w<KER, 12, SPREAD, INTERP, STORE>(a);
    case 16:
        return launch_tile_w<KER, 16, SPREAD, INTERP, STORE>(a);
    default:
        return launch_tile_w<KER, 20, SPREAD, INTERP, STORE>(a);
    }
}

template <typename real>
cudaError_t spread_impl(const TransferArgs &a)
{
    const DevBatch &b = a.b;
    cudaStream_t s = a.stream;
    if (b.n_inst == 0 || b.N == 0)
        return cudaSuccess;
    if constexpr (std::is_same<real, float>::value) {
        // with u and v given, interpolation is fused into the spread (the MLS
        // spread is reproducible in both scatter modes)
        const bool fused = a.u != nullptr && a.v != nullptr;
        if (a.kernel == 1)
            return fused ? launch_tile<1, true, true, true>(a) : launch_tile<1, true, false, true>(a);
        if (a.store)
            return fused ? launch_tile<0, true, true, true>(a) : launch_tile<0, true, false, true>(a);
        return fused ? launch_tile<0, true, true, false>(a) : launch_tile<0, true, false, false>(a);
    } else {
        if (a.kernel == 0) {
            // a warp per (tile, lattice) or octant of one, over the binning's stencil table
            if (!a.w.wtab)
                return cudaErrorInvalidValue;
            // as many warps per CTA (up to kDetWarps) as the largest tile's
            // accumulators fit in one CTA's shared memory
            const size_t per_warp = det_warp_bytes(a.g.max_edge);
            const int warps = (int)std::min<size_t>(kDetWarps, kMaxCtaSmemBytes / per_warp);
            if (warps < 1)
                return cudaErrorInvalidValue;
            const size_t sm = per_warp * warps;
            if (cudaError_t e = allow_smem(spread_det_warp_kernel, kMaxCtaSmemBytes, a.cache->det_warp))
                return e;
            int occ = 1;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, spread_det_warp_kernel, 32 * warps, sm);
            occ = occ < 1 ? 1 : occ;
            spread_det_warp_kernel<<<a.n_sm * occ, 32 * warps, sm, s>>>(b, a.g, a.w, (const double *)a.F,
                                                                      (double *)a.f, a.density);
            IFEM_LAUNCH_CHECK();
            return cudaSuccess;
        }
        auto kern = spread_det_mls_kernel;
        int occ = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kDetThreads, 0);
        occ = occ < 1 ? 1 : occ;
        kern<<<a.n_sm * occ, kDetThreads, 0, s>>>(b, a.g, a.w, (const double *)a.x, (const double *)a.F,
                                                  (double *)a.f, a.density, a.support);
    }
    IFEM_LAUNCH_CHECK();
    return cudaSuccess;
}

template <typename real>
cudaError_t interp_impl(const TransferArgs &a)
{
    const DevBatch &b = a.b;
    if (b.n_inst == 0 || b.N == 0)
        return cudaSuccess;
    if constexpr (std::is_same<real, float>::value) {
        return a.kernel == 0 ? launch_tile<0, false, true, false>(a) : launch_tile<1, false, true, false>(a);
    } else {
        unsigned grid = (unsigned)((b.N + kInterpThreads - 1) / kInterpThreads);
        if (a.kernel == 0)
            interp_kernel<real, 0><<<grid, kInterpThreads, 0, a.stream>>>(b, a.g, a.w, (const real *)a.u,
                                                                    (const real *)a.x, (real *)a.v, (real)a.support,
                                                                    a.use_wtab && a.w.wtab != nullptr);
        else
            interp_kernel<real, 1><<<grid, kInterpThreads, 0, a.stream>>>(b, a.g, a.w, (const real *)a.u,
                                                                    (const real *)a.x, (real *)a.v, (real)a.support, 0);
    }
    IFEM_LAUNCH_CHECK();
    return cudaSuccess;
}

template <typename real>
cudaError_t reduce_impl(const ReduceArgs &a)
{
    const int parts = a.parts ? a.parts : 3;
    const unsigned blocks = (unsigned)(a.b.n_inst + ((parts & 2) ? 3 * a.g.n_boxes : 0));
    if (blocks == 0)
        return cudaSuccess;
    reduce_kernel<real><<<blocks, kReduceThreads, 0, a.stream>>>(a.b, a.g, a.w.red_tile, (const real *)a.x,
                                                               (const real *)a.F, (const real *)a.v, a.red, parts);
    IFEM_LAUNCH_CHECK();
    return cudaSuccess;
}

template <typename real>
cudaError_t fluid_impl(const FluidArgs &a)
{
    const DevBatch &b = a.b;
    if (b.n_inst == 0)
        return cudaSuccess;
    dim3 blk(256);
    dim3 ge((b.max_elems + 255) / 256, b.n_inst);
    dim3 gn((b.max_nodes + 255) / 256, b.n_inst);
    real *ebuf = (real *)a.w.elem_buf;
    fluid_elem_kernel<real><<<ge, blk, 0, a.stream>>>(b, (const real *)a.x, (const real *)a.u, (const real *)a.C,
                                                      (real)a.eta, (real)a.cp, ebuf);
    IFEM_LAUNCH_CHECK();
    if (a.add)
        fluid_gather_kernel<real, true><<<gn, blk, 0, a.stream>>>(b, ebuf, (real *)a.F);
    else
        fluid_gather_kernel<real, false><<<gn, blk, 0, a.stream>>>(b, ebuf, (real *)a.F);
    IFEM_LAUNCH_CHECK();
    return cudaSuccess;
}

template <typename real>
cudaError_t interp_cc_impl(const TransferArgs &a, int ncomp)
{
    const DevBatch &b = a.b;
    if (b.n_inst == 0 || b.N == 0)
        return cudaSuccess;
    unsigned grid = (unsigned)((b.N * ncomp + 255) / 256);
    if (a.kernel == 0)
        interp_cc_kernel<real, 0><<<grid, 256, 0, a.stream>>>(b, a.g, a.w, (const real *)a.u, ncomp,
                                                              (const real *)a.x, (real *)a.v, (real)a.support);
    else
        interp_cc_kernel<real, 1><<<grid, 256, 0, a.stream>>>(b, a.g, a.w, (const real *)a.u, ncomp,
                                                              (const real *)a.x, (real *)a.v, (real)a.support);
    IFEM_LAUNCH_CHECK();
    return cudaSuccess;
}

template <typename real>
cudaError_t ab2_impl(const LagrangeArgs &a)
{
    const long long n3 = 3 * a.b.N;
    if (n3 == 0)
        return cudaSuccess;
    ab2_kernel<real><<<(unsigned)((n3 + 255) / 256), 256, 0, a.stream>>>(
        n3, (const real *)a.x, (real *)(a.x_out ? a.x_out : a.x), (const real *)a.v, (const real *)a.vp,
        (real)a.dt);
    IFEM_LAUNCH_CHECK();
    return cudaSuccess;
}

template <typename real>
cudaError_t volume_impl(const LagrangeArgs &a)
{
    if (a.b.n_inst == 0)
        return cudaSuccess;
    if constexpr (std::is_same<real, float>::value) {
        const size_t sm = sizeof(float4) * (size_t)a.b.max_nodes;
        // all in FP64: volume_kernel's smaller blocks (200 capsules of 162 nodes 8 us, 12)
        if (sm <= kVolSmemBytes && a.b.max_elems >= kPairElems) {
            if (cudaError_t e = allow_smem(volume_f32_kernel, kVolSmemBytes, a.cache->volume))
                return e;
            volume_f32_kernel<<<a.b.n_inst, kVolThreadsF, sm, a.stream>>>(a.b, (const float *)a.x, a.out);
            IFEM_LAUNCH_CHECK();
            return cudaSuccess;
        }
    }
    volume_kernel<real><<<a.b.n_inst, kVolThreads, 0, a.stream>>>(a.b, (const real *)a.x, a.out);
    IFEM_LAUNCH_CHECK();
    return cudaSuccess;
}

template <typename real>
cudaError_t vcorr_impl(const LagrangeArgs &a)
{
    if (a.b.n_inst == 0)
        return cudaSuccess;
    if constexpr (std::is_same<real, float>::value) {
        const size_t sm = 2 * sizeof(float4) * (size_t)a.b.max_nodes;
        if (sm <= kVcorrSmemBytes) {
            if (cudaError_t e = allow_smem(vc_fused_f32_kernel, kVcorrSmemBytes, a.cache->vcorr))
                return e;
            vc_fused_f32_kernel<<<a.b.n_inst, kVolThreadsF, sm, a.stream>>>(a.b, (float *)a.x, a.V0, a.out, a.status);
            IFEM_LAUNCH_CHECK();
            return cudaSuccess;
        }
    }
    dim3 gn((a.b.max_nodes + 255) / 256, a.b.n_inst);
    vc_alpha_kernel<real><<<gn, 256, 0, a.stream>>>(a.b, (const real *)a.x, a.alpha);
    IFEM_LAUNCH_CHECK();
    vc_correct_kernel<real><<<a.b.n_inst, kVolThreads, 0, a.stream>>>(a.b, (real *)a.x, a.alpha, a.V0, a.out,
                                                                       a.status);
    IFEM_LAUNCH_CHECK();
    return cudaSuccess;
}

template <typename real>
cudaError_t area_normals_impl(const DevBatch &b, const void *x, void *nA, cudaStream_t s)
{
    if (b.n_inst == 0)
        return cudaSuccess;
    dim3 gn((b.max_nodes + 255) / 256, b.n_inst);
    area_normal_kernel<real><<<gn, 256, 0, s>>>(b, (const real *)x, (real *)nA);
    IFEM_LAUNCH_CHECK();
    return cudaSuccess;
}

}  // namespace ifem
