// forces.cuh -- Lagrangian internal-force kernels (Algorithm step 1).
//
//   membranes  Eq. FEM_Membrane: F_k = -A0 P^ grad N^_k with the tangent-plane
//              deformation gradient F^ = Ds Dm^-1 and S^ = 2 dW/dC^ for the
//              neo-Hookean (Eq. neo-Hookena) and Skalak (Eq. Skalak) laws;
//   solids     Eq. FEM: F_k = -V0 P grad N_k, F = sum_k x_k (x) grad N_k,
//              P = F S, S = lambda/2 (J^2 - 1) C^-1 + mu (I - C^-1);
//   bending    F_k = 2 kb [Lap(kH - kH0) + 2 (kH - kH0)(kH^2 - kG + kH0 kH)] n_k A_k
//              (force of the Canham-Helfrich energy, Eq. Bending_Energy) with
//              the discrete operators of Meyer, Desbrun, Schroeder & Barr.
//
// Every expression follows one fixed evaluation order (written out in the
// comments of the oracle-independent specification in each function), so
// that the FP64 build, compiled without FMA contraction, is bit-reproducible.
#pragma once
#include "common.cuh"

namespace ifem {

// ------------------------------------------------------------ membranes
// Per triangle (a, b, c) with m = Dm^-1 = [m00 m01; m10 m11] and area A0:
//   d1 = xb - xa, d2 = xc - xa
//   Fh[i][0] = d1[i]*m00 + d2[i]*m10,  Fh[i][1] = d1[i]*m01 + d2[i]*m11
//   C00 = (Fh00^2 + Fh10^2) + Fh20^2, C01 = (Fh00 Fh01 + Fh10 Fh11) + Fh20 Fh21, C11 likewise
//   I1 = C00 + C11, I2 = C00*C11 - C01*C01
//   NH:     q = mu/(I2*I2); S00 = mu - q*C11; S01 = q*C01; S11 = mu - q*C00
//   Skalak: a = mu*((I1-2)+1); b = (0.5*(C*mu))*(I2-1) - mu;
//           S00 = a + b*C11; S01 = -(b*C01); S11 = a + b*C00
//   P0 = Fh[i][0]*S00 + Fh[i][1]*S01, P1 = Fh[i][0]*S01 + Fh[i][1]*S11
//   fb[i] = -(A0*(P0*m00 + P1*m01)); fc[i] = -(A0*(P0*m10 + P1*m11)); fa[i] = -(fb[i] + fc[i])
template <typename real>
__device__ __forceinline__ void membrane_kin(const real xa[3], const real xb[3], const real xc[3],
                                             const real m[4], real Fh[3][2], real &C00, real &C01,
                                             real &C11)
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        real d1 = xb[i] - xa[i];
        real d2 = xc[i] - xa[i];
        Fh[i][0] = d1 * m[0] + d2 * m[2];
        Fh[i][1] = d1 * m[1] + d2 * m[3];
    }
    C00 = (Fh[0][0] * Fh[0][0] + Fh[1][0] * Fh[1][0]) + Fh[2][0] * Fh[2][0];
    C01 = (Fh[0][0] * Fh[0][1] + Fh[1][0] * Fh[1][1]) + Fh[2][0] * Fh[2][1];
    C11 = (Fh[0][1] * Fh[0][1] + Fh[1][1] * Fh[1][1]) + Fh[2][1] * Fh[2][1];
}

template <typename real>
__device__ __forceinline__ void membrane_S(int law, real mu, real C, real C00, real C01, real C11,
                                           real &S00, real &S01, real &S11)
{
    real I1 = C00 + C11;
    real I2 = C00 * C11 - C01 * C01;
    if (law == 0) {
        real q = mu / (I2 * I2);
        S00 = mu - q * C11;
        S01 = q * C01;
        S11 = mu - q * C00;
    } else {
        real a = mu * ((I1 - real(2)) + real(1));
        real b = (real(0.5) * (C * mu)) * (I2 - real(1)) - mu;
        S00 = a + b * C11;
        S01 = -(b * C01);
        S11 = a + b * C00;
    }
}

template <typename real>
__device__ __forceinline__ void membrane_force(int law, real mu, real C, const real m[4], real A0,
                                               const real xa[3], const real xb[3], const real xc[3],
                                               real f[3][3])
{
    real Fh[3][2], C00, C01, C11, S00, S01, S11;
    membrane_kin(xa, xb, xc, m, Fh, C00, C01, C11);
    membrane_S(law, mu, C, C00, C01, C11, S00, S01, S11);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        real P0 = Fh[i][0] * S00 + Fh[i][1] * S01;
        real P1 = Fh[i][0] * S01 + Fh[i][1] * S11;
        f[1][i] = -(A0 * (P0 * m[0] + P1 * m[1]));
        f[2][i] = -(A0 * (P0 * m[2] + P1 * m[3]));
        f[0][i] = -(f[1][i] + f[2][i]);
    }
}

// Directional derivative of the membrane element force along w (for the
// Hessian-vector product): dFh = dDs Dm^-1, dC = dFh^T Fh + Fh^T dFh,
//   NH:     dS = -mu (adj(dC)/I2^2 - 2 adj(C) dI2/I2^3)
//   Skalak: dS = mu dI1 I + (muD/2) dI2 adj(C) + (muD/2 (I2-1) - mu) adj(dC)
//   dP = dFh S + Fh dS,  df_k = -A0 dP grad N_k.
template <typename real>
__device__ __forceinline__ void membrane_dforce(int law, real mu, real C, const real m[4], real A0,
                                                const real xa[3], const real xb[3], const real xc[3],
                                                const real wa[3], const real wb[3], const real wc[3],
                                                real df[3][3])
{
    real Fh[3][2], C00, C01, C11, S00, S01, S11, dF[3][2];
    membrane_kin(xa, xb, xc, m, Fh, C00, C01, C11);
    membrane_S(law, mu, C, C00, C01, C11, S00, S01, S11);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        real d1 = wb[i] - wa[i], d2 = wc[i] - wa[i];
        dF[i][0] = d1 * m[0] + d2 * m[2];
        dF[i][1] = d1 * m[1] + d2 * m[3];
    }
    real dC00 = 0, dC01 = 0, dC11 = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        dC00 += real(2) * dF[i][0] * Fh[i][0];
        dC11 += real(2) * dF[i][1] * Fh[i][1];
        dC01 += dF[i][0] * Fh[i][1] + Fh[i][0] * dF[i][1];
    }
    real I2 = C00 * C11 - C01 * C01;
    real dI1 = dC00 + dC11, dI2 = dC00 * C11 + C00 * dC11 - real(2) * C01 * dC01;
    real dS00, dS01, dS11;
    if (law == 0) {
        real i2 = real(1) / (I2 * I2), i3 = real(2) * dI2 / (I2 * I2 * I2);
        dS00 = -mu * (dC11 * i2 - C11 * i3);
        dS11 = -mu * (dC00 * i2 - C00 * i3);
        dS01 = mu * (dC01 * i2 - C01 * i3);
    } else {
        real muD = C * mu;
        real b = real(0.5) * muD * (I2 - real(1)) - mu, db = real(0.5) * muD * dI2;
        dS00 = mu * dI1 + db * C11 + b * dC11;
        dS11 = mu * dI1 + db * C00 + b * dC00;
        dS01 = -(db * C01 + b * dC01);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        real P0 = dF[i][0] * S00 + dF[i][1] * S01 + Fh[i][0] * dS00 + Fh[i][1] * dS01;
        real P1 = dF[i][0] * S01 + dF[i][1] * S11 + Fh[i][0] * dS01 + Fh[i][1] * dS11;
        df[1][i] = -(A0 * (P0 * m[0] + P1 * m[1]));
        df[2][i] = -(A0 * (P0 * m[2] + P1 * m[3]));
        df[0][i] = -(df[1][i] + df[2][i]);
    }
}

// ------------------------------------------------------------ solids
// det3 = M00 (M11 M22 - M12 M21) - M01 (M10 M22 - M12 M20) + M02 (M10 M21 - M11 M20)
template <typename real>
__device__ __forceinline__ real det3(const real M[3][3])
{
    return M[0][0] * (M[1][1] * M[2][2] - M[1][2] * M[2][1])
         - M[0][1] * (M[1][0] * M[2][2] - M[1][2] * M[2][0])
         + M[0][2] * (M[1][0] * M[2][1] - M[1][1] * M[2][0]);
}

// inverse by the adjugate: R[i][j] = cofactor[j][i] / det
template <typename real>
__device__ __forceinline__ void inv3(const real M[3][3], real det, real R[3][3])
{
    R[0][0] = (M[1][1] * M[2][2] - M[1][2] * M[2][1]) / det;
    R[0][1] = (M[0][2] * M[2][1] - M[0][1] * M[2][2]) / det;
    R[0][2] = (M[0][1] * M[1][2] - M[0][2] * M[1][1]) / det;
    R[1][0] = (M[1][2] * M[2][0] - M[1][0] * M[2][2]) / det;
    R[1][1] = (M[0][0] * M[2][2] - M[0][2] * M[2][0]) / det;
    R[1][2] = (M[0][2] * M[1][0] - M[0][0] * M[1][2]) / det;
    R[2][0] = (M[1][0] * M[2][1] - M[1][1] * M[2][0]) / det;
    R[2][1] = (M[0][1] * M[2][0] - M[0][0] * M[2][1]) / det;
    R[2][2] = (M[0][0] * M[1][1] - M[0][1] * M[1][0]) / det;
}

// F = Ds M: F[i][j] = (Ds[i][0]*M[0][j] + Ds[i][1]*M[1][j]) + Ds[i][2]*M[2][j],
// Ds columns x1-x0, x2-x0, x3-x0.
template <typename real>
__device__ __forceinline__ void tet_F(const real x[4][3], const real *M, real F[3][3])
{
    real Ds[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int i = 0; i < 3; ++i)
            Ds[i][c] = x[1 + c][i] - x[0][i];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            F[i][j] = (Ds[i][0] * M[0 * 3 + j] + Ds[i][1] * M[1 * 3 + j]) + Ds[i][2] * M[2 * 3 + j];
}

// J = det F; Finv = adj(F)/J; Cinv[i][j] = (Finv[i][0] Finv[j][0] + Finv[i][1] Finv[j][1]) + Finv[i][2] Finv[j][2];
// a = (0.5*lam)*(J*J - 1); S[i][j] = a*Cinv[i][j] + mu*(delta_ij - Cinv[i][j]).
template <typename real>
__device__ __forceinline__ real tet_S(real lam, real mu, const real F[3][3], real S[3][3],
                                      real Ci[3][3], real Fi[3][3])
{
    real J = det3(F);
    inv3(F, J, Fi);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            Ci[i][j] = (Fi[i][0] * Fi[j][0] + Fi[i][1] * Fi[j][1]) + Fi[i][2] * Fi[j][2];
    real a = (real(0.5) * lam) * (J * J - real(1));
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            S[i][j] = a * Ci[i][j] + mu * ((i == j ? real(1) : real(0)) - Ci[i][j]);
    return J;
}

// P[i][j] = (F[i][0] S[0][j] + F[i][1] S[1][j]) + F[i][2] S[2][j];
// f_k[i] = -(V0*((P[i][0] M[k-1][0] + P[i][1] M[k-1][1]) + P[i][2] M[k-1][2])), k = 1..3;
// f_0[i] = -((f_1[i] + f_2[i]) + f_3[i]). Returns J.
template <typename real>
__device__ __forceinline__ real tet_force(real lam, real mu, const real *M, real V0, const real x[4][3],
                                          real f[4][3])
{
    real F[3][3], S[3][3], Ci[3][3], Fi[3][3], P[3][3];
    tet_F(x, M, F);
    real J = tet_S(lam, mu, F, S, Ci, Fi);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            P[i][j] = (F[i][0] * S[0][j] + F[i][1] * S[1][j]) + F[i][2] * S[2][j];
#pragma unroll
    for (int k = 1; k <= 3; ++k)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const real *g = M + 3 * (k - 1);
            f[k][i] = -(V0 * ((P[i][0] * g[0] + P[i][1] * g[1]) + P[i][2] * g[2]));
        }
#pragma unroll
    for (int i = 0; i < 3; ++i)
        f[0][i] = -((f[1][i] + f[2][i]) + f[3][i]);
    return J;
}

// dF = dDs M, dJ = J tr(F^-1 dF), dC = dF^T F + F^T dF, dC^-1 = -C^-1 dC C^-1,
// dS = lam J dJ C^-1 + (lam/2 (J^2 - 1) - mu) dC^-1, dP = dF S + F dS.
template <typename real>
__device__ __forceinline__ void tet_dforce(real lam, real mu, const real *M, real V0, const real x[4][3],
                                           const real w[4][3], real df[4][3])
{
    real F[3][3], S[3][3], Ci[3][3], Fi[3][3], dF[3][3];
    tet_F(x, M, F);
    tet_F(w, M, dF);
    real J = tet_S(lam, mu, F, S, Ci, Fi);
    real tr = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k)
            tr += Fi[i][k] * dF[k][i];
    real dJ = J * tr;
    real dC[3][3], T[3][3], dS[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            real s = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k)
                s += dF[k][i] * F[k][j] + F[k][i] * dF[k][j];
            dC[i][j] = s;
        }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            real s = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k)
                s += Ci[i][k] * dC[k][j];
            T[i][j] = s;
        }
    real a = real(0.5) * lam * (J * J - real(1)) - mu;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            real s = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k)
                s += T[i][k] * Ci[k][j];
            dS[i][j] = lam * J * dJ * Ci[i][j] - a * s;
        }
    real dP[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            real s = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k)
                s += dF[i][k] * S[k][j] + F[i][k] * dS[k][j];
            dP[i][j] = s;
        }
#pragma unroll
    for (int k = 1; k <= 3; ++k)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const real *g = M + 3 * (k - 1);
            df[k][i] = -(V0 * (dP[i][0] * g[0] + dP[i][1] * g[1] + dP[i][2] * g[2]));
        }
#pragma unroll
    for (int i = 0; i < 3; ++i)
        df[0][i] = -(df[1][i] + df[2][i] + df[3][i]);
}

template <typename real>
__device__ __forceinline__ const real *ref_ptr(const TmplDev &T);
template <>
__device__ __forceinline__ const double *ref_ptr<double>(const TmplDev &T) { return T.ref_d; }
template <>
__device__ __forceinline__ const float *ref_ptr<float>(const TmplDev &T) { return T.ref_f; }

// ------------------------------------------------------------ element pass
// Thread per (instance, element). Writes the element's nodal forces (or
// force derivatives along w, negated: the Hessian-vector contribution) to
// elem_buf[(elem_off + e)*12 + 3*v + i].
template <typename real, bool HVP>
__global__ void elem_force_kernel(DevBatch b, const real *__restrict__ x, const real *__restrict__ w,
                                  real *__restrict__ ebuf, unsigned long long *status)
{
    const int i = blockIdx.y;
    const InstDev I = b.inst[i];
    const TmplDev T = b.tmpl[I.tmpl];
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long inverted = 0;
    if (e < T.n_elems) {
        const long long N = b.N;
        const real *ref = ref_ptr<real>(T);
        real *out = ebuf + (I.elem_off + e) * 12;
        if (T.kind == 0) {
            int v[3] = {T.elems[3 * e], T.elems[3 * e + 1], T.elems[3 * e + 2]};
            real xs[3][3], ws[3][3], f[3][3];
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    xs[c][a] = x[a * N + I.node_off + v[c]];
                    if (HVP)
                        ws[c][a] = w[a * N + I.node_off + v[c]];
                }
            const real *r = ref + 5 * e;
            real m[4] = {r[0], r[1], r[2], r[3]};
            if (HVP) {
                membrane_dforce<real>(T.law, (real)T.mu, (real)T.C, m, r[4], xs[0], xs[1], xs[2], ws[0],
                                      ws[1], ws[2], f);
            } else {
                membrane_force<real>(T.law, (real)T.mu, (real)T.C, m, r[4], xs[0], xs[1], xs[2], f);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    out[3 * c + a] = HVP ? -f[c][a] : f[c][a];
        } else {
            real xs[4][3], ws[4][3], f[4][3];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                int v = T.elems[4 * e + c];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    xs[c][a] = x[a * N + I.node_off + v];
                    if (HVP)
                        ws[c][a] = w[a * N + I.node_off + v];
                }
            }
            const real *r = ref + 10 * e;
            if (HVP) {
                tet_dforce<real>((real)T.lam, (real)T.mu, r, r[9], xs, ws, f);
            } else {
                real J = tet_force<real>((real)T.lam, (real)T.mu, r, r[9], xs, f);
                inverted = !(J > real(0));
            }
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    out[3 * c + a] = HVP ? -f[c][a] : f[c][a];
        }
    }
    if (!HVP) {
        // one status update per warp
        unsigned long long tot = inverted;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            tot += __shfl_down_sync(0xffffffffu, tot, o);
        if ((threadIdx.x & 31) == 0)
            status_add(status, ST_INVERTED, tot);
    }
}

// Thread per (instance, node): F = sum over incident (element, vertex) in
// ascending element order, starting from 0: acc = acc + f.
template <typename real>
__global__ void node_gather_kernel(DevBatch b, const real *__restrict__ ebuf, real *__restrict__ F)
{
    const int i = blockIdx.y;
    const InstDev I = b.inst[i];
    const TmplDev T = b.tmpl[I.tmpl];
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= T.n_nodes)
        return;
    real acc[3] = {real(0), real(0), real(0)};
    for (int q = T.inc_off[k]; q < T.inc_off[k + 1]; ++q) {
        int code = T.inc_idx[q];
        const real *src = ebuf + (I.elem_off + (code >> 2)) * 12 + 3 * (code & 3);
#pragma unroll
        for (int a = 0; a < 3; ++a)
            acc[a] = acc[a] + src[a];
    }
    const long long N = b.N;
#pragma unroll
    for (int a = 0; a < 3; ++a)
        F[a * N + I.node_off + k] = acc[a];
}

// ------------------------------------------------------------ fluid stress
// Newtonian and polymer fluid-stress parts of Eq. FEM inside a solid (Sec.
// "Governing Equations"; they enter F^IB with a plus sign), per tet on the
// reference configuration, in this order:
//   F = Ds M, J = det F, Fi = F^-1; G = Du M = sum_k u_k (x) grad N_k;
//   Lv[i][j] = (G[i][0] Fi[0][j] + G[i][1] Fi[1][j]) + G[i][2] Fi[2][j];
//   E[i][j] = Lv[i][j] + Lv[j][i];
//   P[i][j] = (eta J) ((E[i][0] Fi[j][0] + E[i][1] Fi[j][1]) + E[i][2] Fi[j][2]);
//   polymer: Cb[i][j] = (((c_0 + c_1) + c_2) + c_3) * 0.25, c_k = C_k[i][j] - d_ij,
//   P[i][j] = P[i][j] + (J cp) ((Cb[i][0] Fi[j][0] + Cb[i][1] Fi[j][1]) + Cb[i][2] Fi[j][2]),
//   cp = eta (1 - beta) / lambda;
//   f_k[i] = V0 ((P[i][0] M[k-1][0] + P[i][1] M[k-1][1]) + P[i][2] M[k-1][2]), k = 1..3;
//   f_0[i] = -((f_1[i] + f_2[i]) + f_3[i]).
// C per node: (xx, yy, zz, xy, xz, yz).
template <typename real>
__device__ __forceinline__ void tet_fluid_force(real eta, real cp, const real *M, real V0, const real x[4][3],
                                                const real u[4][3], const real C[4][6], bool polymer,
                                                real f[4][3])
{
    real F[3][3], G[3][3], Fi[3][3], Lv[3][3], E[3][3], P[3][3];
    tet_F(x, M, F);
    tet_F(u, M, G);
    const real J = det3(F);
    inv3(F, J, Fi);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            Lv[i][j] = (G[i][0] * Fi[0][j] + G[i][1] * Fi[1][j]) + G[i][2] * Fi[2][j];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            E[i][j] = Lv[i][j] + Lv[j][i];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            P[i][j] = (eta * J) * ((E[i][0] * Fi[j][0] + E[i][1] * Fi[j][1]) + E[i][2] * Fi[j][2]);
    if (polymer) {
        const int sym[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};
        real Cb[3][3];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const real dij = i == j ? real(1) : real(0);
                real acc = C[0][sym[i][j]] - dij;
#pragma unroll
                for (int k = 1; k < 4; ++k)
                    acc = acc + (C[k][sym[i][j]] - dij);
                Cb[i][j] = acc * real(0.25);
            }
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j)
                P[i][j] = P[i][j] + (J * cp) * ((Cb[i][0] * Fi[j][0] + Cb[i][1] * Fi[j][1]) + Cb[i][2] * Fi[j][2]);
    }
#pragma unroll
    for (int k = 1; k <= 3; ++k)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const real *g = M + 3 * (k - 1);
            f[k][i] = V0 * ((P[i][0] * g[0] + P[i][1] * g[1]) + P[i][2] * g[2]);
        }
#pragma unroll
    for (int i = 0; i < 3; ++i)
        f[0][i] = -((f[1][i] + f[2][i]) + f[3][i]);
}

// Thread per (instance, element) of a solid: the element's fluid-stress
// nodal forces into elem_buf; fluid_gather_kernel then sums them per node.
// Membranes carry no fluid stress in the paper's thin-shell model.
template <typename real>
__global__ void fluid_elem_kernel(DevBatch b, const real *__restrict__ x, const real *__restrict__ u,
                                  const real *__restrict__ C, real eta, real cp, real *__restrict__ ebuf)
{
    const InstDev I = b.inst[blockIdx.y];
    const TmplDev T = b.tmpl[I.tmpl];
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= T.n_elems)
        return;
    if (T.kind == 0)
        return;   // membranes: no fluid stress (fluid_gather_kernel writes their zeros)
    real *out = ebuf + (I.elem_off + e) * 12;
    const long long N = b.N;
    real xs[4][3], us[4][3], Cs[4][6], f[4][3];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const long long v = I.node_off + T.elems[4 * e + c];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            xs[c][a] = x[a * N + v];
            us[c][a] = u[a * N + v];
        }
#pragma unroll
        for (int q = 0; q < 6; ++q)
            Cs[c][q] = C ? C[q * N + v] : real(0);
    }
    const real *r = ref_ptr<real>(T) + 10 * e;
    tet_fluid_force<real>(eta, cp, r, r[9], xs, us, Cs, C != nullptr, f);
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int a = 0; a < 3; ++a)
            out[3 * c + a] = f[c][a];
}

// ------------------------------------------------------------ bending
// Geometry of one incident triangle (p[c] is the vertex itself, corners
// c1 = c+1, c2 = c+2): edge dots at every corner, twice the area
// (|u x w| is the same from every corner), the unnormalised face normal.
// cot at a corner = dot / (2 area); the corner is obtuse iff its dot < 0.
template <typename real>
struct TriGeom {
    real dot[3];
    real twoA;
    real fn[3];
};

template <typename real>
__device__ __forceinline__ void tri_geom(const real p[3][3], TriGeom<real> &t)
{
    real e1[3], e2[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        e1[a] = p[1][a] - p[0][a];
        e2[a] = p[2][a] - p[0][a];
    }
    t.fn[0] = e1[1] * e2[2] - e1[2] * e2[1];
    t.fn[1] = e1[2] * e2[0] - e1[0] * e2[2];
    t.fn[2] = e1[0] * e2[1] - e1[1] * e2[0];
    t.twoA = sqrt(t.fn[0] * t.fn[0] + t.fn[1] * t.fn[1] + t.fn[2] * t.fn[2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        real u0 = p[(c + 1) % 3][0] - p[c][0], u1 = p[(c + 1) % 3][1] - p[c][1], u2 = p[(c + 1) % 3][2] - p[c][2];
        real w0 = p[(c + 2) % 3][0] - p[c][0], w1 = p[(c + 2) % 3][1] - p[c][1], w2 = p[(c + 2) % 3][2] - p[c][2];
        t.dot[c] = u0 * w0 + u1 * w1 + u2 * w2;
    }
}

// Pass 1 at vertex i (template-local id k), over its incident triangles in
// ascending order: K += cot_k (x_i - x_j) + cot_j (x_i - x_k); mixed Voronoi
// area (Voronoi region if no corner is obtuse, area/2 at an obtuse corner,
// area/4 at the others); corner angles; area-weighted normal. Outputs A,
// kH = K.n/2 (K /= 2A), kG = (2 pi - angles)/A and the unit normal n.
// The cotangents share one reciprocal of 2A per triangle. The angle deficit
// 2 pi - sum theta is minus the argument of prod (dot + i 2A) over the corners
// (each factor has argument theta), one atan2 per vertex instead of one per
// corner; it equals the angle sum's deficit while that lies in (-pi, pi), and
// the product is rescaled by an exact power of two if it grows small.
template <typename real, typename Load>
__device__ inline void bend_vertex_pass1(const TmplDev &T, int k, Load ld, real &A_out, real &kH_out,
                                         real &kG_out, real n_out[3])
{
    real K[3] = {0, 0, 0}, nrm[3] = {0, 0, 0}, A = 0;
    real zr = 1, zi = 0;   // running product of (dot + i 2A) over the corners
    for (int q = T.inc_off[k]; q < T.inc_off[k + 1]; ++q) {
        // incident triangle rotated to start at this vertex: (k, j, l)
        const int2 jk = T.ring[q];
        const int c = 0, c1 = 1, c2 = 2;
        real p[3][3];
        ld(k, p[0]);
        ld(jk.x, p[1]);
        ld(jk.y, p[2]);
        TriGeom<real> t;
        tri_geom(p, t);
        const real inv2A = real(1) / t.twoA;
        real cj = t.dot[c1] * inv2A, ck = t.dot[c2] * inv2A;
        real eij[3], eik[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            eij[a] = p[c][a] - p[c1][a];
            eik[a] = p[c][a] - p[c2][a];
        }
#pragma unroll
        for (int a = 0; a < 3; ++a)
            K[a] += ck * eij[a] + cj * eik[a];
        bool obtuse = t.dot[0] < real(0) || t.dot[1] < real(0) || t.dot[2] < real(0);
        real Ai;
        if (!obtuse)
            Ai = (ck * (eij[0] * eij[0] + eij[1] * eij[1] + eij[2] * eij[2])
                  + cj * (eik[0] * eik[0] + eik[1] * eik[1] + eik[2] * eik[2])) / real(8);
        else if (t.dot[c] < real(0))
            Ai = t.twoA / real(4);
        else
            Ai = t.twoA / real(8);
        A += Ai;
        const real pr = zr * t.dot[c] - zi * t.twoA, pi = zr * t.twoA + zi * t.dot[c];
        zr = pr;
        zi = pi;
        if (fabs(zr) + fabs(zi) < real(1e-30)) {
            zr *= real(1099511627776.0);   // 2^40, exact
            zi *= real(1099511627776.0);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a)
            nrm[a] += t.fn[a];
    }
    real nl = sqrt(nrm[0] * nrm[0] + nrm[1] * nrm[1] + nrm[2] * nrm[2]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        n_out[a] = nrm[a] / nl;
        K[a] /= real(2) * A;
    }
    A_out = A;
    kH_out = real(0.5) * (K[0] * n_out[0] + K[1] * n_out[1] + K[2] * n_out[2]);
    kG_out = -atan2(zi, zr) / A;
}

// Bending in global memory: what a triangle gives its corners once per triangle
// (the element buffer, free after the gather: unnormalised normal, cotangents,
// the corners' areas), then two passes over the nodes. The FP64 pipe bounds it;
// a pass that evaluates a node's triangles itself does each one three times, in
// both passes (133 k nodes in all: 396 us, 231 now).
// bend_buf per global node: [A, kH, kG, n0, n1, n2].
template <typename real>
__global__ void bend_tri_kernel(DevBatch b, const real *__restrict__ x, real *__restrict__ ebuf)
{
    const InstDev I = b.inst[blockIdx.y];
    const TmplDev &T = b.tmpl[I.tmpl];
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (T.kind != 0 || T.kb == 0.0 || e >= T.n_elems)
        return;
    const long long N = b.N;
    real p[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int v = T.elems[3 * e + c];
#pragma unroll
        for (int a = 0; a < 3; ++a)
            p[c][a] = x[a * N + I.node_off + v];
    }
    TriGeom<real> t;
    tri_geom(p, t);
    const real inv2A = real(1) / t.twoA;
    real cot[3], len2[3];   // len2[c]: of the edge from corner c to the next
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        cot[c] = t.dot[c] * inv2A;
        real d[3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
            d[a] = p[c][a] - p[(c + 1) % 3][a];
        len2[c] = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    }
    const bool obtuse = t.dot[0] < real(0) || t.dot[1] < real(0) || t.dot[2] < real(0);
    real *o = ebuf + (I.elem_off + e) * 12;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        o[c] = t.fn[c];
        o[3 + c] = cot[c];
        o[6 + c] = !obtuse ? (cot[(c + 2) % 3] * len2[c] + cot[(c + 1) % 3] * len2[(c + 2) % 3]) / real(8)
                           : t.twoA / (t.dot[c] < real(0) ? real(4) : real(8));
    }
}

// Thread per (instance, node): bend_vertex_pass1 from the triangles' values. The
// angle deficit comes from the product of (cot + i), whose factors have the same
// arguments as (dot + i 2A); it grows, and is scaled down by an exact power of two.
template <typename real>
__global__ void bend_pass1_kernel(DevBatch b, const real *__restrict__ x, const real *__restrict__ ebuf,
                                  real *__restrict__ bb)
{
    const InstDev I = b.inst[blockIdx.y];
    const TmplDev &T = b.tmpl[I.tmpl];
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (T.kind != 0 || T.kb == 0.0 || k >= T.n_nodes)
        return;
    const long long N = b.N;
    real me[3], K[3] = {0, 0, 0}, nrm[3] = {0, 0, 0}, A = 0, zr = 1, zi = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a)
        me[a] = x[a * N + I.node_off + k];
    for (int q = T.inc_off[k]; q < T.inc_off[k + 1]; ++q) {
        const int code = T.inc_idx[q], c = code & 3, c1 = c == 2 ? 0 : c + 1, c2 = c == 0 ? 2 : c - 1;
        const int2 jk = T.ring[q];   // the corners c1 and c2
        const real *o = ebuf + (I.elem_off + (code >> 2)) * 12;
        const real cot = o[3 + c], cj = o[3 + c1], ck = o[3 + c2];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const real *xa = x + a * N + I.node_off;
            K[a] += ck * (me[a] - xa[jk.x]) + cj * (me[a] - xa[jk.y]);
            nrm[a] += o[a];
        }
        A += o[6 + c];
        const real pr = zr * cot - zi, pi = zr + zi * cot;
        zr = pr;
        zi = pi;
        if (fabs(zr) + fabs(zi) > real(1e12)) {
            zr *= real(9.094947017729282379150390625e-13);   // 2^-40, exact
            zi *= real(9.094947017729282379150390625e-13);
        }
    }
    const real nl = sqrt(nrm[0] * nrm[0] + nrm[1] * nrm[1] + nrm[2] * nrm[2]);
    real n[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        n[a] = nrm[a] / nl;
        K[a] /= real(2) * A;
    }
    real *o = bb + 6LL * (I.node_off + k);
    o[0] = A;
    o[1] = real(0.5) * (K[0] * n[0] + K[1] * n[1] + K[2] * n[2]);
    o[2] = -atan2(zi, zr) / A;
    o[3] = n[0];
    o[4] = n[1];
    o[5] = n[2];
}

// Thread per (instance, node): cotangent Laplacian of (kH - kH0) and the force,
// F = F_el + F_be (one add per component).
template <typename real>
__global__ void bend_pass2_kernel(DevBatch b, const real *__restrict__ ebuf, const real *__restrict__ bb,
                                  real *__restrict__ F)
{
    const InstDev I = b.inst[blockIdx.y];
    const TmplDev &T = b.tmpl[I.tmpl];
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (T.kind != 0 || T.kb == 0.0 || k >= T.n_nodes)
        return;
    const long long N = b.N;
    const real *all = bb + 6LL * I.node_off, *me = all + 6LL * k;
    const real A = me[0], kH = me[1], kG = me[2], kH0 = real(-0.5) * (real)T.c0;
    real lap = 0;
    for (int q = T.inc_off[k]; q < T.inc_off[k + 1]; ++q) {
        const int code = T.inc_idx[q], c = code & 3, c1 = c == 2 ? 0 : c + 1, c2 = c == 0 ? 2 : c - 1;
        const int2 jk = T.ring[q];
        const real *cot = ebuf + (I.elem_off + (code >> 2)) * 12 + 3;
        lap += cot[c2] * ((all[6LL * jk.x + 1] - kH0) - (kH - kH0)) + cot[c1] * ((all[6LL * jk.y + 1] - kH0) - (kH - kH0));
    }
    const real L = lap / (real(2) * A), dh = kH - kH0;
    const real mag = real(2) * (real)T.kb * (L + real(2) * dh * (kH * kH - kG + kH0 * kH)) * A;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        real *p = F + a * N + I.node_off + k;
        *p = *p + mag * me[3 + a];
    }
}

// Node sums of the fluid-stress element buffer for solids (ascending element
// order from 0, as node_gather_kernel); membrane nodes get 0 (ADD: unchanged).
template <typename real, bool ADD>
__global__ void fluid_gather_kernel(DevBatch b, const real *__restrict__ ebuf, real *__restrict__ F)
{
    const InstDev I = b.inst[blockIdx.y];
    const TmplDev T = b.tmpl[I.tmpl];
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= T.n_nodes || (ADD && T.kind == 0))
        return;
    real acc[3] = {real(0), real(0), real(0)};
    if (T.kind != 0) {
        for (int q = T.inc_off[k]; q < T.inc_off[k + 1]; ++q) {
            const int code = T.inc_idx[q];
            const real *src = ebuf + (I.elem_off + (code >> 2)) * 12 + 3 * (code & 3);
#pragma unroll
            for (int a = 0; a < 3; ++a)
                acc[a] = acc[a] + src[a];
        }
    }
    const long long N = b.N;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        real *p = F + a * N + I.node_off + k;
        *p = ADD ? *p + acc[a] : acc[a];
    }
}

// n_k A_k of every membrane node (unit normal times mixed area, from the
// bending pass-1 operators) as a node array; solid nodes get 0. Source of
// the indicator-function equation (Sec. "Variable Viscosity Implementation").
template <typename real>
__global__ void area_normal_kernel(DevBatch b, const real *__restrict__ x, real *__restrict__ nA)
{
    const int i = blockIdx.y;
    const InstDev I = b.inst[i];
    const TmplDev T = b.tmpl[I.tmpl];
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= T.n_nodes)
        return;
    const long long N = b.N;
    const long long node = I.node_off + k;
    if (T.kind != 0) {
#pragma unroll
        for (int a = 0; a < 3; ++a)
            nA[a * N + node] = real(0);
        return;
    }
    auto ld = [&](int v, real p[3]) {
#pragma unroll
        for (int a = 0; a < 3; ++a)
            p[a] = x[a * N + I.node_off + v];
    };
    real A, kH, kG, n[3];
    bend_vertex_pass1<real>(T, k, ld, A, kH, kG, n);
#pragma unroll
    for (int a = 0; a < 3; ++a)
        nA[a * N + node] = n[a] * A;
}

// ------------------------------------------------------------ FP32 nodal path
// Thread per node: the node's force is gathered over its incident elements in
// a fixed order, so there are no atomics, no element buffer and no second
// pass over the elements, and the result is the same from run to run. Each
// element is evaluated once per corner (3 or 4 times), in forms that need only
// the corner's own row. What an element gives its corners adds up to zero in
// exact arithmetic; the forms below keep that under rounding (every corner
// computes the same bits of what it shares with another, and takes them with
// the opposite sign), as an element evaluated once does: errors that do not
// cancel between neighbours show up in the spread field, where the forces
// themselves mostly do (one red cell: error of the field 2.1e-6 without, 1.1e-6
// with, relative L2).
//
// Membranes, triangle (a, b, c), the node k one of its corners, (k, j, l) in
// orientation order: the laws depend on the metric alone. With d_i the edge dot
// at corner i (d_k = (x_j - x_k).(x_l - x_k)) and r_i the same of the reference
// triangle, w = 1/(2 A0), 4 A^2 = |e x e'|^2:
//   I1 = w^2 (d_a (r_b + r_c) + d_b (r_c + r_a) + d_c (r_a + r_b)), I2 = 4 A^2 w^2,
//   F_k = s_l (x_j - x_k) + s_j (x_l - x_k), s_i = (w/2) (a r_i + b d_i),
// S^ = a I + b adj C^: NH a = mu, b = -mu/I2^2; Skalak a = mu (I1 - 1), b = (C
// mu/2)(I2 - 1) - mu. s_i belongs to the edge opposite corner i: both of its
// ends take the same s_i (the dots do not depend on the corner they are computed
// from, I1 and 4 A^2 are evaluated in the triangle's own order), times edge
// vectors of opposite sign (a fused multiply-add: exact up to the sum).
//
// Solids, tet (0, 1, 2, 3), y_i = x_i - x_0: with P = mu F + beta cof F, beta =
// (lam/2 (J^2 - 1) - mu)/J, J = y_1 . (y_2 x y_3)/(6 V0),
//   F_k = sum_m mu h_km (x_m - x_k) + (beta/6) n_k,  h_km = -V0 grad N_k . grad N_m,
//   n_1, n_2, n_3 = -y_2 x y_3, -y_3 x y_1, -y_1 x y_2, n_0 = -(n_1 + n_2 + n_3):
// h_km is the same number at both ends, y, J, beta and the n are evaluated in
// the tet's own order by every corner.
//
// 4 A^2 comes from the dots, d_a d_b + d_b d_c + d_c d_a, whose error grows with the
// square of 1/sin of an obtuse angle, where that of the cross product grows with
// 1/sin. Batches with templates whose reference triangles have it above
// kObtuseSum times the result (105 degrees) take OBTUSE, which takes the cross
// product there (error of single triangles' forces at 150 degrees, 15% deformed: 6e-6
// with the dots, 1.1e-6; in the reference triangle's plane, as the general path, 0.9
// to 1.4e-6); it costs 8% (600 particles 92 us, 99), so others do without (at 100
// degrees, 1.84, the errors are equal). Beyond kObtuseMost (160 degrees) I1
// cancels too: the general path.
//
// Layout: incidences in slices of 32 nodes (a warp), slot by slot, so that a
// warp's reads are consecutive: reference values and 16-bit node ids, the
// node's corner number in the top bits. Membranes: r_a, r_b, r_c, w and (j, l);
// a closed surface's incidences are ordered as a fan around the node (l of one
// triangle is j of the next), so a triangle takes one new position instead of
// two. Solids: the h of the four corners with 1/(6 V0) in the node's own place
// (where x_m - x_k is 0) and the four corners.
//
// Bending (Meyer et al. 2003) per incident triangle: 2A = |e1 x e2| from one
// rsqrt, cotangents d/2A. The corner-angle sum enters only through 2 pi -
// sum(theta); it is taken as -arg(prod_t (cos theta_t + i sin theta_t)), one
// atan2 per node, which equals the deficit while it lies in (-pi, pi) (any
// vertex of a closed mesh that is not folded onto itself).
struct RingF {
    float fn[3], q, inv2A, dk, dj, dl;   // q = |e1 x e2|^2
};
__device__ __forceinline__ float dot3f(const float a[3], const float b[3])
{
    return fmaf(a[2], b[2], fmaf(a[1], b[1], __fmul_rn(a[0], b[0])));
}
__device__ __forceinline__ void edge_f32(const float4 p, const float4 q, float e[3])   // q - p
{
    e[0] = q.x - p.x;
    e[1] = q.y - p.y;
    e[2] = q.z - p.z;
}
// e1 = x_j - x_k, e2 = x_l - x_k and e3 = x_l - x_j. Each component of a dot is
// a product of the same two coordinate differences from whichever corner it is
// computed, up to two signs that cancel: the dots are the same bits at all three.
__device__ __forceinline__ void ring_tri_f32(const float e1[3], const float e2[3], const float e3[3], RingF &t)
{
    t.fn[0] = e1[1] * e2[2] - e1[2] * e2[1];
    t.fn[1] = e1[2] * e2[0] - e1[0] * e2[2];
    t.fn[2] = e1[0] * e2[1] - e1[1] * e2[0];
    t.q = t.fn[0] * t.fn[0] + t.fn[1] * t.fn[1] + t.fn[2] * t.fn[2];
    t.inv2A = rsqrtf(t.q);
    t.dk = dot3f(e1, e2);
    t.dj = -dot3f(e1, e3);
    t.dl = dot3f(e2, e3);
}

// |p x q|^2, every operation's rounding stated: the same bits for p, q of either sign
__device__ __forceinline__ float cross2_f32(const float p[3], const float q[3])
{
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int j = (i + 1) % 3, k = (i + 2) % 3;
        const float n = fmaf(p[j], q[k], -__fmul_rn(p[k], q[j]));
        s = fmaf(n, n, s);
    }
    return s;
}

// Pass 1 of a membrane node: elastic force and, with BEND, the part of the
// bending force that needs no neighbour's curvature, 2 kb * 2 (kH - kH0)
// (kH^2 - kG + kH0 kH) A n; kH receives the mean curvature. Along a fan the
// second edge of a triangle is the first of the next: its vector is kept.
template <bool BEND, bool OBTUSE>
__device__ __forceinline__ void nodal_membrane(const TmplDev &T, int k, const float4 *xs, float F[3], float &kH)
{
    const float mu = T.mu_f, half_muD = T.half_muD_f;
    const int deg = T.inc_off[k + 1] - T.inc_off[k];
    const long long at = T.nod_off[k >> 5] + (k & 31);
    const float4 *ref = T.nod_ref + at;
    const ushort2 *idx = reinterpret_cast<const ushort2 *>(T.nod_idx) + at;
    const float4 xk = xs[k];
    float K[3] = {0.f, 0.f, 0.f}, nrm[3] = {0.f, 0.f, 0.f}, A8 = 0.f, zr = 1.f, zi = 0.f;
    F[0] = F[1] = F[2] = 0.f;
    float4 rn = make_float4(0.f, 0.f, 0.f, 0.f);
    ushort2 in = make_ushort2(0, 0);
    int prev = -1;
    float4 xj = xk;
    float e1[3] = {0.f, 0.f, 0.f};   // x_j - x_k
    if (deg > 0) {
        rn = ref[0];
        in = idx[0];
    }
    for (int q = 0; q < deg; ++q) {
        const float4 r = rn;
        const int j = in.x & kNodMask, c = in.x >> kNodBits, l = in.y;
        if (q + 1 < deg) {
            rn = ref[32 * (q + 1)];
            in = idx[32 * (q + 1)];
        }
        if (j != prev) {   // a new fan
            xj = xs[j];
            edge_f32(xk, xj, e1);
        }
        prev = l;
        const float4 xl = xs[l];
        float e2[3], e3[3];
        edge_f32(xk, xl, e2);
        edge_f32(xj, xl, e3);
        xj = xl;
        RingF t;
        ring_tri_f32(e1, e2, e3, t);
        // the triangle's own order: k is its corner c, so (a, b, c) = (k, j, l), (l, k, j) or (j, l, k)
        const float da = c == 0 ? t.dk : (c == 1 ? t.dl : t.dj), db = c == 0 ? t.dj : (c == 1 ? t.dk : t.dl),
                    dc = c == 0 ? t.dl : (c == 1 ? t.dj : t.dk);
        const float rj = c == 0 ? r.y : (c == 1 ? r.z : r.x), rl = c == 0 ? r.z : (c == 1 ? r.x : r.y);
        const float w = r.w, w2 = __fmul_rn(w, w);
        float S = fmaf(dc, da, fmaf(db, dc, __fmul_rn(da, db)));   // 4 A^2
        if constexpr (OBTUSE) {
            // the products cancel in a triangle with an obtuse corner: there from the
            // edges of its first corner, whose cross product every corner computes
            // alike, up to its sign
            const float least = fminf(da, fminf(db, dc));
            if (least < 0.f && 16.f * __fmul_rn(least, least) > S) {
                float p[3], q2[3];
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    p[i] = c == 0 ? e1[i] : (c == 1 ? e2[i] : e3[i]);
                    q2[i] = c == 0 ? e2[i] : (c == 1 ? e3[i] : e1[i]);
                }
                S = cross2_f32(p, q2);
            }
        }
        const float I2 = __fmul_rn(S, w2);
        float a, b;
        if (T.law == 0) {
            a = mu;
            b = __fdiv_rn(-mu, __fmul_rn(I2, I2));
        } else {
            const float I1 = __fmul_rn(fmaf(dc, r.x + r.y, fmaf(db, r.z + r.x, __fmul_rn(da, r.y + r.z))), w2);
            a = __fmul_rn(mu, I1 - 1.f);
            b = fmaf(half_muD, I2 - 1.f, -mu);
        }
        const float hw = 0.5f * w;
        const float sl = __fmul_rn(hw, fmaf(a, rl, __fmul_rn(b, t.dl)));   // edge (k, j)
        const float sj = __fmul_rn(hw, fmaf(a, rj, __fmul_rn(b, t.dj)));   // edge (k, l)
#pragma unroll
        for (int i = 0; i < 3; ++i)
            F[i] = fmaf(sj, e2[i], fmaf(sl, e1[i], F[i]));
        if constexpr (BEND) {
            const float cj = t.dj * t.inv2A, cl = t.dl * t.inv2A;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                K[i] += cl * e1[i] + cj * e2[i];   // cot_l (x_j - x_k) + cot_j (x_l - x_k), sign taken below
                nrm[i] += t.fn[i];
            }
            const float l1 = t.dk + t.dj, l2 = t.dk + t.dl, twoA = t.q * t.inv2A;
            // 8 x mixed area: Voronoi, or 2A / 4 at an obtuse corner and 2A / 8 beside one
            const float obt = t.dk < 0.f ? twoA + twoA : twoA;
            A8 += fminf(t.dk, fminf(t.dj, t.dl)) >= 0.f ? cl * l1 + cj * l2 : obt;
            // unit (cos, sin) of the corner angle at k, |e1||e2| = sqrt(l1 l2)
            const float rr = rsqrtf(l1 * l2);
            const float cr = t.dk * rr, ci = twoA * rr;
            const float nr = zr * cr - zi * ci;
            zi = zr * ci + zi * cr;
            zr = nr;
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
            e1[i] = e2[i];
    }
    if constexpr (BEND) {
        const float kb = T.kb_f, kH0 = T.kH0_f;
        const float rnl = rsqrtf(nrm[0] * nrm[0] + nrm[1] * nrm[1] + nrm[2] * nrm[2]);
        const float A = 0.125f * A8;
        const float h = -0.5f / A;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            nrm[i] *= rnl;
            K[i] *= h;
        }
        kH = 0.5f * (K[0] * nrm[0] + K[1] * nrm[1] + K[2] * nrm[2]);
        const float kG = -atan2f(zi, zr) / A;
        const float dh = kH - kH0;
        const float mag = 2.f * kb * (2.f * dh * (kH * kH - kG + kH0 * kH)) * A;
#pragma unroll
        for (int i = 0; i < 3; ++i)
            F[i] += mag * nrm[i];
    }
}

// Pass 2 of a membrane node: 2 kb Lap(kH - kH0) A n = kb lap n, lap = sum over
// the ring of cot_l (kH_j - kH_k) + cot_j (kH_l - kH_k) (kH beside the
// positions; A cancels), n recomputed in the order of pass 1.
__device__ __forceinline__ void nodal_bend2(const TmplDev &T, int k, const float4 *xs, float Fb[3])
{
    const int deg = T.inc_off[k + 1] - T.inc_off[k];
    const ushort2 *idx = reinterpret_cast<const ushort2 *>(T.nod_idx) + T.nod_off[k >> 5] + (k & 31);
    const float4 xk = xs[k];
    float lap = 0.f, nrm[3] = {0.f, 0.f, 0.f};
    float4 xj = xk;
    float e1[3] = {0.f, 0.f, 0.f};
    int prev = -1;
    ushort2 in = deg > 0 ? idx[0] : make_ushort2(0, 0);
    for (int q = 0; q < deg; ++q) {
        const int j = in.x & kNodMask, l = in.y;
        if (q + 1 < deg)
            in = idx[32 * (q + 1)];
        if (j != prev) {
            xj = xs[j];
            edge_f32(xk, xj, e1);
        }
        prev = l;
        const float4 xl = xs[l];
        float e2[3], e3[3];
        edge_f32(xk, xl, e2);
        edge_f32(xj, xl, e3);
        RingF t;
        ring_tri_f32(e1, e2, e3, t);
        lap += (t.dl * (xj.w - xk.w) + t.dj * (xl.w - xk.w)) * t.inv2A;
        xj = xl;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            nrm[i] += t.fn[i];
            e1[i] = e2[i];
        }
    }
    const float s = T.kb_f * lap * rsqrtf(nrm[0] * nrm[0] + nrm[1] * nrm[1] + nrm[2] * nrm[2]);
#pragma unroll
    for (int i = 0; i < 3; ++i)
        Fb[i] = s * nrm[i];
}

__device__ __forceinline__ void cross_f32(const float a[3], const float b[3], float r[3])
{
    r[0] = a[1] * b[2] - a[2] * b[1];
    r[1] = a[2] * b[0] - a[0] * b[2];
    r[2] = a[0] * b[1] - a[1] * b[0];
}

// A solid node; returns the number of incident tets with J <= 0 among those
// that count here (each tet is counted at its first corner).
__device__ __forceinline__ int nodal_solid(const TmplDev &T, int k, const float4 *xs, float F[3])
{
    const float mu = T.mu_f, half_lam = T.half_lam_f;
    const int deg = T.inc_off[k + 1] - T.inc_off[k];
    const long long at = T.nod_off[k >> 5] + (k & 31);
    const float4 *ref = T.nod_ref + at;
    const ushort4 *idx = reinterpret_cast<const ushort4 *>(T.nod_idx) + at;
    const float4 xk = xs[k];
    int inverted = 0;
    F[0] = F[1] = F[2] = 0.f;
    float4 rn = make_float4(0.f, 0.f, 0.f, 0.f);
    ushort4 in = make_ushort4(0, 0, 0, 0);
    if (deg > 0) {
        rn = ref[0];
        in = idx[0];
    }
    for (int q = 0; q < deg; ++q) {
        const float4 h = rn;
        const ushort4 v = in;
        if (q + 1 < deg) {
            rn = ref[32 * (q + 1)];
            in = idx[32 * (q + 1)];
        }
        const int c = v.x >> kNodBits;
        const float4 p0 = xs[v.x & kNodMask], p1 = xs[v.y], p2 = xs[v.z], p3 = xs[v.w];
        float y1[3], y2[3], y3[3], n1[3], n2[3], n3[3];
        edge_f32(p0, p1, y1);
        edge_f32(p0, p2, y2);
        edge_f32(p0, p3, y3);
        cross_f32(y2, y3, n1);
        cross_f32(y3, y1, n2);
        cross_f32(y1, y2, n3);
        const float inv6V = c == 0 ? h.x : (c == 1 ? h.y : (c == 2 ? h.z : h.w));
        const float J = dot3f(y1, n1) * inv6V;
        inverted += c == 0 && !(J > 0.f);
        const float beta = __fdiv_rn(fmaf(half_lam, fmaf(J, J, -1.f), -mu), 6.f * J);
        const float m0 = mu * h.x, m1 = mu * h.y, m2 = mu * h.z, m3 = mu * h.w;
        const float x0[3] = {p0.x - xk.x, p0.y - xk.y, p0.z - xk.z}, x1[3] = {p1.x - xk.x, p1.y - xk.y, p1.z - xk.z};
        const float x2[3] = {p2.x - xk.x, p2.y - xk.y, p2.z - xk.z}, x3[3] = {p3.x - xk.x, p3.y - xk.y, p3.z - xk.z};
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float n = c == 0 ? (n1[i] + n2[i]) + n3[i] : -(c == 1 ? n1[i] : (c == 2 ? n2[i] : n3[i]));
            float acc = fmaf(m0, x0[i], F[i]);
            acc = fmaf(m1, x1[i], acc);
            acc = fmaf(m2, x2[i], acc);
            acc = fmaf(m3, x3[i], acc);
            F[i] = fmaf(beta, n, acc);
        }
    }
    return inverted;
}

// What bounds it: latency and instruction issue, at the 28 warps per SM that 64
// registers allow (fewer registers spill: 110 against 85 us on the 600-particle
// suspension with 40), shared memory at a third of its rate. 600 particles (1.33 M
// nodes): 92 us against 129 us for the kernel before it (per-element forces
// added with float atomics in shared memory, 60 % of that pipe), one red cell
// 11 against 47 us, the element-buffer path of the deterministic mode (four
// launches) 51 -> 20 us on 72 particles, 64 balls of 4096 nodes 93 -> 48 us.
// One cluster of S CTAs per particle (S = 1: one CTA), each holding every
// position of the particle in shared memory (float4, kH in w) and taking a
// chunk of its nodes (inst0 < 0: all particles, the largest first; else
// particles inst0, inst0 + 1, ...); kH goes to every CTA of the cluster between the passes.
// The row of F is kept in global memory between the passes (read back by the
// thread that wrote it).
template <bool CLUSTER, bool OBTUSE>
static __global__ void __launch_bounds__(512, 2) forces_nodal_f32_kernel(DevBatch b, const float *__restrict__ x,
                                                                      float *__restrict__ F,
                                                                      unsigned long long *status, int inst0, int S)
{
    extern __shared__ __align__(16) float4 nodal_xs[];
    float4 *xs = nodal_xs;
    const int rank = CLUSTER ? (int)(blockIdx.x % S) : 0;
    const int which = CLUSTER ? (int)(blockIdx.x / S) : (int)blockIdx.x;
    const InstDev I = b.inst[inst0 < 0 ? b.inst_order[which] : inst0 + which];
    const TmplDev &T = b.tmpl[I.tmpl];
    const int nn = I.n_nodes;
    const long long N = b.N;
    const float *xp = x + I.node_off;
    for (int k = threadIdx.x; k < nn; k += blockDim.x)
        xs[k] = make_float4(xp[k], xp[N + k], xp[2 * N + k], 0.f);
    if constexpr (CLUSTER)   // every CTA of the cluster holds its positions (and runs) before kH arrives
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else
        __syncthreads();
    const int chunk = CLUSTER ? ((nn + S - 1) / S + 31) & ~31 : nn;
    const int k0 = rank * chunk, k1 = min(nn, k0 + chunk);
    float *Fp = F + I.node_off;
    if (T.kind != 0) {
        int inverted = 0;
        for (int k = k0 + (int)threadIdx.x; k < k1; k += blockDim.x) {
            float f[3];
            inverted += nodal_solid(T, k, xs, f);
#pragma unroll
            for (int a = 0; a < 3; ++a)
                Fp[a * N + k] = f[a];
        }
        inverted = __reduce_add_sync(0xffffffffu, inverted);
        if ((threadIdx.x & 31) == 0)
            status_add(status, ST_INVERTED, (unsigned long long)inverted);
        return;   // every CTA of the cluster alike
    }
    if (T.kb_f == 0.f) {
        for (int k = k0 + (int)threadIdx.x; k < k1; k += blockDim.x) {
            float f[3], kH;
            nodal_membrane<false, OBTUSE>(T, k, xs, f, kH);
#pragma unroll
            for (int a = 0; a < 3; ++a)
                Fp[a * N + k] = f[a];
        }
        return;
    }
    for (int k = k0 + (int)threadIdx.x; k < k1; k += blockDim.x) {
        float f[3], kH;
        nodal_membrane<true, OBTUSE>(T, k, xs, f, kH);
#pragma unroll
        for (int a = 0; a < 3; ++a)
            Fp[a * N + k] = f[a];
        if constexpr (CLUSTER) {
            const unsigned at = smem_u32(&xs[k].w);
            for (int r = 0; r < S; ++r) {
                unsigned there;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(at), "r"(r));
                asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(there), "f"(kH) : "memory");
            }
        } else {
            xs[k].w = kH;
        }
    }
    if constexpr (CLUSTER)
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else
        __syncthreads();
    for (int k = k0 + (int)threadIdx.x; k < k1; k += blockDim.x) {
        float f[3];
        nodal_bend2(T, k, xs, f);
#pragma unroll
        for (int a = 0; a < 3; ++a)
            Fp[a * N + k] += f[a];
    }
}

}  // namespace ifem
