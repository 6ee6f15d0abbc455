// lagrangian.cuh -- the Lagrangian update after a coupling step: the
// Adams-Bashforth position update (Eq. Bashforth_eqn), per-particle volumes
// and the membrane volume correction of Sec. "Conservation of Volume for
// Membranes" (after Mendez et al. 2014). Positions are the particles' local
// offsets; volumes and the correction's sums have FP64 accuracy in both precisions
// (for FP32 positions by float pairs, see below).
#pragma once
#include "forces.cuh"
#include "transfer.cuh"

namespace ifem {

// xo = x + dt*(1.5*v - 0.5*vp), componentwise over the 3N node values (in
// place when xo == x).
template <typename real>
__global__ void ab2_kernel(long long n3, const real *x, real *xo, const real *__restrict__ v,
                           const real *__restrict__ vp, real dt)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n3)
        xo[i] = ab2_value(x[i], v[i], vp[i], dt);
}

__device__ __forceinline__ void cross3d(const double a[3], const double b[3], double r[3])
{
    r[0] = a[1] * b[2] - a[2] * b[1];
    r[1] = a[2] * b[0] - a[0] * b[2];
    r[2] = a[0] * b[1] - a[1] * b[0];
}
__device__ __forceinline__ double dot3d(const double a[3], const double b[3])
{
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

template <typename real>
__device__ __forceinline__ void load_node_d(const real *x, long long N, long long node, double p[3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a)
        p[a] = (double)x[a * N + node];
}

constexpr int kVolThreads = 256;

// Block per instance: membranes V = (1/18) sum_faces [a.(b x c) + b.(c x a)
// + c.(a x b)] (the polyhedron formula; the three terms are equal, so
// V = 1/6 sum a.(b x c)), solids V = sum_tets det(Ds)/6.
template <typename real>
__global__ void __launch_bounds__(kVolThreads) volume_kernel(DevBatch b, const real *__restrict__ x,
                                                             double *__restrict__ vol)
{
    __shared__ double sh[kVolThreads];
    const InstDev I = b.inst[blockIdx.x];
    const TmplDev T = b.tmpl[I.tmpl];
    const long long N = b.N;
    double s = 0.0;
    for (int e = threadIdx.x; e < T.n_elems; e += blockDim.x) {
        if (T.kind == 0) {
            // the three cyclic triple products of the formula are equal: one
            // per face, V = 1/6 sum a.(b x c)
            double p[3][3], t[3];
            for (int c = 0; c < 3; ++c)
                load_node_d(x, N, I.node_off + T.elems[3 * e + c], p[c]);
            cross3d(p[1], p[2], t);
            s += dot3d(p[0], t);
        } else {
            double p[4][3], Ds[3][3];
            for (int c = 0; c < 4; ++c)
                load_node_d(x, N, I.node_off + T.elems[4 * e + c], p[c]);
            for (int c = 0; c < 3; ++c)
                for (int a = 0; a < 3; ++a)
                    Ds[a][c] = p[1 + c][a] - p[0][a];
            s += det3(Ds) / 6.0;
        }
    }
    const double r = block_sum<kVolThreads>(s, sh);
    if (threadIdx.x == 0)
        vol[blockIdx.x] = T.kind == 0 ? r / 6.0 : r;
}

// ------------------------------------------------ FP32 positions, float pairs
// Volumes and the correction's sums of FP32 positions to FP64 accuracy with little
// of the FP64 pipe (two lane operations a cycle and SM on this GPU, conversions
// included): a triple product of float vectors as an unevaluated float pair.
// Products are exact (by FMA), sums carry their error term. Inputs are scaled by
// powers of two (TmplDev::vol_scale) so that the error terms stay in range for
// particles of any unit.
// A pair holds 2^-48 of a term. What is left of that in a volume falls with the
// square root of the number of elements, to what FP64 leaves from kPairElems of them
// on, if the sums themselves are FP64 (each element's below kPairFew elements, four
// as a pair from there; vol_totals). Relative error of the volume, rms over random
// affine maps and noise, FP64 and pairs: 80 triangles 0.8 and 1.9e-16, 320 0.7 and
// 1.0e-16, 1280 0.7 and 0.9e-16 (red cells 0.8 and 0.8e-16), 2058 tets 0.7 and
// 0.8e-16, 5120 triangles 0.8 and 0.7e-16; pairs summed as pairs up to the block 3 to
// 5e-16 throughout. Below, volumes take the FP64 pipe.
constexpr int kPairElems = 1024, kPairFew = 4096;

__device__ __forceinline__ DF df_cross_comp(float a1, float b2, float a2, float b1)   // a1 b2 - a2 b1
{
    const float p = __fmul_rn(a1, b2), pe = fmaf(a1, b2, -p), q = __fmul_rn(a2, b1), qe = fmaf(a2, b1, -q);
    const float s = p - q, bv = s - p;
    const float e = ((p - (s - bv)) - (q + bv)) + (pe - qe);
    const float h = s + e;
    return DF{h, e - (h - s)};
}
// a . (b x c) + rest: the products' high parts are summed exactly, what is below
// them (eight terms and rest) with its error, so that half an ulp of the low part
// is nearly all that is lost
__device__ __forceinline__ DF df_triple(const float a[3], const float b[3], const float c[3], float rest)
{
    float h = 0.f, l = rest, m = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int j = (i + 1) % 3, k = (i + 2) % 3;
        const DF u = df_cross_comp(b[j], c[k], b[k], c[j]);
        const float p = __fmul_rn(u.hi, a[i]), pe = fmaf(u.hi, a[i], -p);
        float e, e1, e2;
        h = i ? two_sum(h, p, e) : p;
        l = two_sum(l, pe, e1);
        l = two_sum(l, __fmul_rn(u.lo, a[i]), e2);
        m += e1 + e2;
        if (i) {
            l = two_sum(l, e, e1);
            m += e1;
        }
    }
    float e;
    h = two_sum(h, l, e);
    return DF{h, e + m};
}
// y - x as an exact float pair h + l (l is mostly 0)
__device__ __forceinline__ void df_edge(const float x[3], const float y[3], float h[3], float l[3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float s = y[a] - x[a], bv = s - y[a];
        h[a] = s;
        l[a] = (y[a] - (s - bv)) - (x[a] + bv);
    }
}
__device__ __forceinline__ float dot_cross_f32(const float a[3], const float b[3], const float c[3])
{
    float n[3];
    cross_f32(b, c, n);
    return a[0] * n[0] + a[1] * n[1] + a[2] * n[2];
}
// a . (b x c) of a face = a . ((b - a) x (c - a)): the edges are about a cell
// long, so the products that cancel in the cross product are (h/R)^2 times those
// of b x c (the rounding that is left is below the FP64 evaluation of b x c). The
// l terms to first order: they are below 2^-24 of the h.
__device__ __forceinline__ DF df_face(const float p[3][3])
{
    float h1[3], l1[3], h2[3], l2[3];
    df_edge(p[0], p[1], h1, l1);
    df_edge(p[0], p[2], h2, l2);
    return df_triple(p[0], h1, h2, dot_cross_f32(p[0], l1, h2) + dot_cross_f32(p[0], h1, l2));
}
// det of a tet's edges x_i - x_0, the same way
__device__ __forceinline__ DF df_tet(const float x[4][3])
{
    float h[3][3], l[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
        df_edge(x[0], x[1 + c], h[c], l[c]);
    float rest = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c)
        rest += dot_cross_f32(l[c], h[(c + 1) % 3], h[(c + 2) % 3]);
    return df_triple(h[0], h[1], h[2], rest);
}

constexpr int kVolThreadsF = 512;

// A thread's sum of float pairs: so many as a pair, those in FP64.
struct PairSum {
    DF p{0.f, 0.f};
    double s = 0.0;
    int n = 0;
    __device__ __forceinline__ void add(DF t) { df_add_df(p, t); }
    __device__ __forceinline__ void add(DF t, int every)
    {
        df_add_df(p, t);
        if (++n == every)
            flush();
    }
    __device__ __forceinline__ void flush()
    {
        s += (double)p.hi;
        s += (double)p.lo;
        p = DF{0.f, 0.f};
        n = 0;
    }
};

// Fixed-order block totals of Q FP64 values per thread, a warp each (every thread
// gets them).
template <int Q>
__device__ __forceinline__ void vol_totals(const double (&v)[Q], double (*sh)[kVolThreadsF], double (&tot)[Q])
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < Q; ++q)
        sh[q][threadIdx.x] = v[q];
    __syncthreads();
    if (wid < Q) {
        double r = 0.0;
        for (int k = lane; k < kVolThreadsF; k += 32)
            r += sh[wid][k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            r += __shfl_down_sync(0xffffffffu, r, o);
        __syncwarp();   // the warp has read its row
        if (lane == 0)
            sh[wid][0] = r;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q; ++q)
        tot[q] = sh[q][0];
}

// Stages an instance's positions, scaled, in shared memory.
__device__ __forceinline__ void vol_stage(const InstDev &I, const float *x, long long N, float scale, float4 *xs)
{
    for (int k = threadIdx.x; k < I.n_nodes; k += kVolThreadsF) {
        const long long i = I.node_off + k;
        xs[k] = make_float4(x[i] * scale, x[N + i] * scale, x[2 * N + i] * scale, 0.f);
    }
    __syncthreads();
}
__device__ __forceinline__ void vol_get(const float4 *xs, int k, float p[3])
{
    const float4 v = xs[k];
    p[0] = v.x;
    p[1] = v.y;
    p[2] = v.z;
}
__device__ __forceinline__ double vol_unscale(float scale, int power)   // scale^-power, exact
{
    const double r = 1.0 / (double)scale;
    return power == 2 ? r * r : (power == 3 ? r * r * r : r);
}
// Adds an element's six-fold volume: p its corners, E its template's elements.
__device__ __forceinline__ void vol_add(PairSum &s, int kind, int E, const float p[4][3])
{
    if (E >= kPairElems) {
        s.add(kind == 0 ? df_face(p) : df_tet(p), E >= kPairFew ? 4 : 1);
        return;
    }
    double q[3][3], t[3];   // a face's corners, or a tet's edges
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int a = 0; a < 3; ++a)
            q[c][a] = kind == 0 ? (double)p[c][a] : (double)p[c + 1][a] - (double)p[0][a];
    cross3d(q[1], q[2], t);
    s.s += dot3d(q[0], t);
}

// Block per instance, FP32 positions (templates whose positions fit shared
// memory): the formulas of volume_kernel. 200 capsules of 2562 nodes: 18 us
// against 59 us in FP64; of 642 nodes 10 and 19.
static __global__ void __launch_bounds__(kVolThreadsF) volume_f32_kernel(DevBatch b, const float *__restrict__ x,
                                                                         double *__restrict__ vol)
{
    extern __shared__ __align__(16) float4 vol_xs[];
    __shared__ double sh[1][kVolThreadsF];
    const InstDev I = b.inst[blockIdx.x];
    const TmplDev &T = b.tmpl[I.tmpl];
    vol_stage(I, x, b.N, T.vol_scale, vol_xs);
    const int nv = T.kind == 0 ? 3 : 4;
    PairSum s;
    for (int e = threadIdx.x; e < T.n_elems; e += kVolThreadsF) {
        float p[4][3];
        for (int c = 0; c < nv; ++c)
            vol_get(vol_xs, T.elems[nv * e + c], p[c]);
        vol_add(s, T.kind, T.n_elems, p);
    }
    s.flush();
    const double v[1] = {s.s};
    double r[1];
    vol_totals(v, sh, r);
    if (threadIdx.x == 0)
        vol[blockIdx.x] = r[0] * vol_unscale(T.vol_scale, 3) / 6.0;
}

// Thread per (instance, node) of a membrane: alpha_I = -(1/12) sum over the
// incident faces, ascending, of x_{I2} x x_{I3} (the face's other two nodes
// in cyclic order); FP64 for FP64 positions, FP32 edge vectors for FP32
// positions (below). alpha: 3 doubles per node (batch node order).
template <typename real>
__global__ void vc_alpha_kernel(DevBatch b, const real *__restrict__ x, double *__restrict__ alpha)
{
    const InstDev I = b.inst[blockIdx.y];
    const TmplDev T = b.tmpl[I.tmpl];
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (T.kind != 0 || k >= T.n_nodes)
        return;
    const long long N = b.N;
    double *o = alpha + 3 * (I.node_off + k);
    if constexpr (std::is_same<real, float>::value) {
        // FP32: over the closed ring sum x_I2 x x_I3 = sum (x_I2 - x_I) x (x_I3 - x_I)
        // (the ring's edges x_I3 - x_I2 sum to zero), so the cross products
        // take edge vectors about one cell long, exact enough in FP32; the
        // correction's sums use this same alpha in FP64, so the corrected
        // volume still meets V0
        float pk[3], acc[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 0; a < 3; ++a)
            pk[a] = x[a * N + I.node_off + k];
        for (int q = T.inc_off[k]; q < T.inc_off[k + 1]; ++q) {
            const int code = T.inc_idx[q], e = code >> 2, v = code & 3;
            const long long n1 = I.node_off + T.elems[3 * e + (v + 1) % 3];
            const long long n2 = I.node_off + T.elems[3 * e + (v + 2) % 3];
            float e1[3], e2[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                e1[a] = x[a * N + n1] - pk[a];
                e2[a] = x[a * N + n2] - pk[a];
            }
            acc[0] += e1[1] * e2[2] - e1[2] * e2[1];
            acc[1] += e1[2] * e2[0] - e1[0] * e2[2];
            acc[2] += e1[0] * e2[1] - e1[1] * e2[0];
        }
#pragma unroll
        for (int a = 0; a < 3; ++a)
            o[a] = (double)acc[a] * (-1.0 / 12.0);
    } else {
        double acc[3] = {0.0, 0.0, 0.0};
        for (int q = T.inc_off[k]; q < T.inc_off[k + 1]; ++q) {
            const int code = T.inc_idx[q], e = code >> 2, v = code & 3;
            const int n1 = T.elems[3 * e + (v + 1) % 3], n2 = T.elems[3 * e + (v + 2) % 3];
            double p1[3], p2[3], t[3];
            load_node_d(x, N, I.node_off + n1, p1);
            load_node_d(x, N, I.node_off + n2, p2);
            cross3d(p1, p2, t);
#pragma unroll
            for (int a = 0; a < 3; ++a)
                acc[a] = acc[a] + t[a];
        }
#pragma unroll
        for (int a = 0; a < 3; ++a)
            o[a] = acc[a] * (-1.0 / 12.0);
    }
}

// Lambda of the cubic by Newton from 0; 0 and a count in ST_DOMAIN where it does
// not converge.
__device__ inline double vc_newton(double A, double B, double C, double D, unsigned long long *status)
{
    double L = 0.0;
    for (int it = 0; it < 100; ++it) {
        const double f = ((A * L + B) * L + C) * L + D;
        const double fp = (3.0 * A * L + 2.0 * B) * L + C;
        if (fp == 0.0)
            break;
        const double step = f / fp;
        L = L - step;
        if (fabs(step) <= 1e-15 * fmax(1.0, fabs(L)))
            return L;
    }
    status_add(status, ST_DOMAIN, 1);
    return 0.0;
}

// Block per instance of a membrane: the cubic A L^3 + B L^2 + C L + D = 0 of
// the volume correction with the paper's cyclic sums (A = (1/18) sum
// alpha.(alpha x alpha), B = (1/6) sum x.(alpha x alpha), C = (1/6) sum
// alpha.(x x x), D = V(x) - V0, FP64 block trees; for A and V the three
// cyclic terms are equal and one is taken, times 3, and C is evaluated as
// -2 sum |alpha_I|^2, equal to it since alpha_I = -(1/2) grad_I V), Lambda by Newton from 0
// (|step| <= 1e-15 max(1, |L|), at most 100 steps; the root the oracle
// takes), then x_I = x_I + Lambda alpha_I. Solids: lambda = 0, x unchanged.
// status ST_DOMAIN counts instances whose Newton failed (x left unchanged).
template <typename real>
__global__ void __launch_bounds__(kVolThreads) vc_correct_kernel(DevBatch b, real *__restrict__ x,
                                                                 const double *__restrict__ alpha,
                                                                 const double *__restrict__ V0,
                                                                 double *__restrict__ lambda,
                                                                 unsigned long long *status)
{
    __shared__ double sh[kVolThreads];
    __shared__ double sL;
    const InstDev I = b.inst[blockIdx.x];
    const TmplDev T = b.tmpl[I.tmpl];
    const long long N = b.N;
    if (T.kind != 0) {
        if (threadIdx.x == 0 && lambda)
            lambda[blockIdx.x] = 0.0;
        return;
    }
    double sA = 0.0, sB = 0.0, sC = 0.0, sV = 0.0;
    for (int e = threadIdx.x; e < T.n_elems; e += blockDim.x) {
        int nd[3];
        double p[3][3], q[3][3];
        for (int c = 0; c < 3; ++c) {
            nd[c] = T.elems[3 * e + c];
            load_node_d(x, N, I.node_off + nd[c], p[c]);
            const double *al = alpha + 3 * (I.node_off + nd[c]);
            q[c][0] = al[0];
            q[c][1] = al[1];
            q[c][2] = al[2];
        }
        // cyclic (a, b, c), (b, c, a), (c, a, b): B takes all three terms;
        // the three terms of A and of V are equal, so those take one (1/6)
        double xx[3], qq[3];
        cross3d(p[1], p[2], xx);
        sV += dot3d(p[0], xx);
        for (int c = 0; c < 3; ++c) {
            const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
            cross3d(q[c1], q[c2], qq);
            sB += dot3d(p[c], qq);
            if (c == 0)
                sA += dot3d(q[0], qq);
        }
    }
    // C = 1/6 sum alpha.(x x x) (cyclic) = sum_I alpha_I . grad_I V = -2 sum_I |alpha_I|^2,
    // since alpha_I = -(1/2) grad_I V exactly
    for (int k = threadIdx.x; k < T.n_nodes; k += blockDim.x) {
        const double *al = alpha + 3 * (I.node_off + k);
        sC += al[0] * al[0] + al[1] * al[1] + al[2] * al[2];
    }
    const double A = block_sum<kVolThreads>(sA, sh) / 6.0;
    const double B = block_sum<kVolThreads>(sB, sh) / 6.0;
    const double C = -2.0 * block_sum<kVolThreads>(sC, sh);
    const double D = block_sum<kVolThreads>(sV, sh) / 6.0 - V0[blockIdx.x];
    if (threadIdx.x == 0) {
        const double L = vc_newton(A, B, C, D, status);
        sL = L;
        if (lambda)
            lambda[blockIdx.x] = L;
    }
    __syncthreads();
    const double L = sL;
    for (int k = threadIdx.x; k < T.n_nodes; k += blockDim.x) {
        const double *al = alpha + 3 * (I.node_off + k);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            real *p = x + a * N + I.node_off + k;
            *p = (real)((double)*p + L * al[a]);
        }
    }
}

// The correction of FP32 positions in one launch, block per instance (templates
// whose positions and alphas fit shared memory): alpha_I as in vc_alpha_kernel
// (12 alpha = -acc, acc an FP32 sum of edge cross products, kept as it is), the
// cubic's sums in float pairs with the factors 1/12 taken out, Newton in FP64,
// x_I = x_I + Lambda alpha_I to one rounding. D is what Lambda's error comes from
// (a volume to 1e-16 less a close one), so A, B and C are kept as pairs up to the
// block. Lambda differs from the FP64 kernels' by what FP64 leaves (1e-13 for a
// volume off by 1e-3). 200 capsules of 2562 nodes: 61 us against 203 us for
// vc_alpha_kernel and vc_correct_kernel in FP64; of 642 nodes 29 and 64, 162 nodes
// 23 and 31.
static __global__ void __launch_bounds__(kVolThreadsF) vc_fused_f32_kernel(DevBatch b, float *__restrict__ x,
                                                                           const double *__restrict__ V0,
                                                                           double *__restrict__ lambda,
                                                                           unsigned long long *status)
{
    extern __shared__ __align__(16) float4 vol_xs[];
    __shared__ double sh[4][kVolThreadsF];
    __shared__ double sL;
    const InstDev I = b.inst[blockIdx.x];
    const TmplDev &T = b.tmpl[I.tmpl];
    const long long N = b.N;
    if (T.kind != 0) {
        if (threadIdx.x == 0 && lambda)
            lambda[blockIdx.x] = 0.0;
        return;
    }
    const int nn = T.n_nodes;
    const float sx = T.vol_scale, sa = sx * sx;
    float4 *xs = vol_xs, *as = vol_xs + nn;   // positions and the alphas' sums, scaled
    vol_stage(I, x, N, sx, xs);
    PairSum sA, sB, sC, sV;
    for (int k = threadIdx.x; k < nn; k += kVolThreadsF) {
        const float4 xk = xs[k];
        const float pk[3] = {xk.x, xk.y, xk.z};
        float acc[3] = {0.f, 0.f, 0.f};
        for (int q = T.inc_off[k]; q < T.inc_off[k + 1]; ++q) {
            const int2 jl = T.ring[q];
            float p1[3], p2[3], e1[3], e2[3];
            vol_get(xs, jl.x, p1);
            vol_get(xs, jl.y, p2);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                e1[a] = p1[a] - pk[a];
                e2[a] = p2[a] - pk[a];
            }
            acc[0] += e1[1] * e2[2] - e1[2] * e2[1];
            acc[1] += e1[2] * e2[0] - e1[0] * e2[2];
            acc[2] += e1[0] * e2[1] - e1[1] * e2[0];
        }
        as[k] = make_float4(acc[0], acc[1], acc[2], 0.f);   // scaled by sa
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float p = __fmul_rn(acc[a], acc[a]);
            sC.add(DF{p, fmaf(acc[a], acc[a], -p)});
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < T.n_elems; e += kVolThreadsF) {
        float p[4][3], q[3][3];
        for (int c = 0; c < 3; ++c) {
            const int v = T.elems[3 * e + c];
            vol_get(xs, v, p[c]);
            vol_get(as, v, q[c]);
        }
        // the cyclic terms: the three of A and of V are equal, B takes all
        vol_add(sV, 0, T.n_elems, p);
        sA.add(df_triple(q[0], q[1], q[2], 0.f));
        sB.add(df_triple(p[0], q[1], q[2], 0.f));
        sB.add(df_triple(p[1], q[2], q[0], 0.f));
        sB.add(df_triple(p[2], q[0], q[1], 0.f));
    }
    sA.flush();
    sB.flush();
    sC.flush();
    sV.flush();
    const double v[4] = {sA.s, sB.s, sC.s, sV.s};
    double tot[4];
    vol_totals(v, sh, tot);
    const double ux = vol_unscale(sx, 1), ua = vol_unscale(sa, 1), g = -1.0 / 12.0;
    const double A = tot[0] * (ua * ua * ua) * (g * g * g) / 6.0;
    const double B = tot[1] * (ux * ua * ua) * (g * g) / 6.0;
    const double C = -2.0 * tot[2] * (ua * ua) * (g * g);
    const double D = tot[3] * (ux * ux * ux) / 6.0 - V0[blockIdx.x];
    if (threadIdx.x == 0) {
        const double L = vc_newton(A, B, C, D, status);
        sL = L;
        if (lambda)
            lambda[blockIdx.x] = L;
    }
    __syncthreads();
    // Lambda alpha = acc * M in the scaled positions' unit, M a float pair
    if (sL == 0.0)
        return;
    const double M = sL * g * ua * (double)sx;
    const float mh = (float)M, ml = (float)(M - (double)mh);
    for (int k = threadIdx.x; k < nn; k += kVolThreadsF) {
        const float4 xk = xs[k], ak = as[k];
        const float xv[3] = {xk.x, xk.y, xk.z}, av[3] = {ak.x, ak.y, ak.z};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float p = __fmul_rn(av[a], mh), pe = fmaf(av[a], mh, -p) + av[a] * ml;
            DF s{xv[a], 0.f};
            df_add_df(s, DF{p, pe});
            x[a * N + I.node_off + k] = (s.hi + s.lo) * (float)ux;
        }
    }
}

}  // namespace ifem
