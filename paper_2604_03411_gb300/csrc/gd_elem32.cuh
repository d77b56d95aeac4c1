// gd_elem32.cuh -- FP32 element math shared by the two mixed-precision element
// kernels (CUDA-core networks in gd_asm_mixed.cu, tensor-core networks in
// gd_asm_tc.cu): per-point kinematics and invariants, the network input map, the
// energy derivatives with respect to (I1-3, I2-3, J-1) (qp mode, lane = quadrature
// point), and the local damage update on the CUDA cores.  The per-point records of
// stress and tangent and the element rows are those of gd_rows.cuh.
//
// Paper passages: Sec. 3.1f (F, phi_q, grad phi_q, element residual, Table
// kernel_inputs), Sec. 2.1f (P, Y vector, Y), Sec. 3.2f (monolithic tangent),
// Sec. 4.1f (degradation, gradient and penalty energies, Eq. (ostwald_potential)),
// Sec. 4.2f Eqs. (dd_0), (dd_1).
#pragma once

#include <cuda_runtime.h>

#include "gd_internal.cuh"
#include "gd_rows.cuh"

namespace gd {
namespace e32 {

constexpr float kGauss = 0.57735026918962576f;   // 1/sqrt(3)
constexpr float kEpsF = 1.1920929e-7f;

struct MatF {
    float mu_e, lambda_e, eta_d, kappa_d, beta_d, c_d, gamma_d, qcoef;
    int energy, local_max;
};
struct NcF {
    float psi_N0, psi_n, y_N0, y_s;
};
__device__ __forceinline__ NcF ncf(const NetConst &n)
{
    NcF r = {(float)n.psi_N0, (float)n.psi_n, (float)n.y_N0, (float)n.y_s};
    return r;
}
template <class Args>
__device__ __forceinline__ int spec_of(const Args &A, int64_t e) { return A.elem_spec ? __ldg(A.elem_spec + e) : 0; }
template <class Args>
__device__ __forceinline__ const DevNet &psi_of(const Args &A, int s) { return A.psi_tab ? A.psi_tab[s] : A.psi; }
template <class Args>
__device__ __forceinline__ const DevNet &yld_of(const Args &A, int s) { return A.yld_tab ? A.yld_tab[s] : A.yld; }

__device__ __forceinline__ MatF to_f(const MatConst &m)
{
    MatF r;
    r.mu_e = (float)m.mu_e; r.lambda_e = (float)m.lambda_e; r.eta_d = (float)m.eta_d; r.kappa_d = (float)m.kappa_d;
    r.beta_d = (float)m.beta_d; r.c_d = (float)m.c_d; r.gamma_d = (float)m.gamma_d; r.qcoef = (float)m.qcoef;
    r.energy = m.energy; r.local_max = m.local_max;
    return r;
}

// softplus(v) and its derivative sigmoid(v) from one exponential
__device__ __forceinline__ void sp_sig(float v, float &sp, float &sg)
{
    const float e = expf(-fabsf(v));
    sp = fmaxf(v, 0.0f) + log1pf(e);
    const float r = 1.0f / (1.0f + e);
    sg = v >= 0.0f ? r : e * r;
}
template <int DIM>
struct Geo {
    static constexpr int NEN = DIM == 2 ? 4 : 8;
    static constexpr int NQ = NEN;
    static constexpr int NDOF = DIM + 1;
    static constexpr int EPW = 32 / NQ;         // elements per batch
};

// sign of node a along reference axis k (HEX8 ordering; Q4 uses the first four)
__device__ __forceinline__ float node_sgn(int a, int k)
{
    int b = (k == 0) ? ((a & 3) == 1 || (a & 3) == 2) : (k == 1 ? ((a & 3) >= 2) : (a >= 4));
    return b ? 1.0f : -1.0f;
}

// N_a and dN_a/dxi at reference point xi
template <int DIM>
__device__ __forceinline__ void ref_shape(int a, const float *xi, float &N, float *dN)
{
    float f[3], s[3];
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        s[k] = node_sgn(a, k);
        f[k] = 0.5f * (1.0f + s[k] * xi[k]);
    }
    N = 1.0f;
#pragma unroll
    for (int k = 0; k < DIM; ++k) N *= f[k];
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        float v = 0.5f * s[k];
#pragma unroll
        for (int l = 0; l < DIM; ++l)
            if (l != k) v *= f[l];
        dN[k] = v;
    }
}

__device__ __forceinline__ int sym6(int i, int j)
{
    // (0,0)0 (0,1)1 (0,2)2 (1,1)3 (1,2)4 (2,2)5
    int a = i < j ? i : j, b = i < j ? j : i;
    return a == 0 ? b : (a == 1 ? 2 + b : 5);
}

// Unit mode evaluates the networks of kNP points of one element at once (lane = network unit,
// up to two units per lane), so that a weight load serves four points and four independent
// chains hide each other's latency.  (Two groups of 16 lanes for narrow networks were slower:
// the second copy of the code cost more in instruction fetches than half-empty warps, 2.23
// against 1.84 ms on 96 specimens of widths 16 to 32.)
constexpr int kNP = 4;
constexpr int kUnits = 2;                     // units per lane
struct alignas(16) PVec {
    float v[kNP];
};
// floats of a warp's unit-mode buffer
__host__ __device__ constexpr int unit_floats(int wmax) { return 24 * wmax; }

// Yield network value and slope of four points in unit mode: G(q) = s (N_k(q) - N_k(0)),
// G' = s N_k'(q) (Eq. (Gq_NN)).  Lane l holds the argument of point l / 8 and receives
// its G and G'.  Every lane calls it.
static __device__ __forceinline__ void yield_unit4(const DevNet &net, const NcF &nc, float q, float &G, float &Gp,
                                                   float *buf, int lane)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int w = net.width;
    const float *V1 = net.pf, *c1 = V1 + w, *V2 = c1 + w, *B2 = V2 + w * w, *c2 = B2 + w, *v3 = c2 + w,
                 *b3 = v3 + w;
    PVec *sS = reinterpret_cast<PVec *>(buf), *sT = sS + w;
    float qp[kNP];
#pragma unroll
    for (int p = 0; p < kNP; ++p) qp[p] = __shfl_sync(kAll, q, 8 * p);
#pragma unroll 1
    for (int t = 0; t < kUnits; ++t) {
        const int j = lane + 32 * t;
        if (j < w) {
            const float a = __ldg(V1 + j), b = __ldg(c1 + j);
            PVec s, d;
#pragma unroll
            for (int p = 0; p < kNP; ++p) {
                float sg;
                sp_sig(b + a * qp[p], s.v[p], sg);
                d.v[p] = sg * a;
            }
            sS[j] = s;
            sT[j] = d;
        }
    }
    __syncwarp();
    float n0[kNP], n1[kNP];
#pragma unroll
    for (int p = 0; p < kNP; ++p) n0[p] = n1[p] = 0.0f;
#pragma unroll 1
    for (int t = 0; t < kUnits; ++t) {
        const int k = lane + 32 * t;
        if (k < w) {
            const float bk = __ldg(B2 + k), ck = __ldg(c2 + k), vk = __ldg(v3 + k);
            float h[kNP], d[kNP];
#pragma unroll
            for (int p = 0; p < kNP; ++p) {
                h[p] = ck + bk * qp[p];
                d[p] = bk;
            }
            const float *col = net.W2Tf + k;
#pragma unroll 2
            for (int j = 0; j < w; ++j) {
                const float wkj = __ldg(col + j * w);
                const PVec s = sS[j], e = sT[j];
#pragma unroll
                for (int p = 0; p < kNP; ++p) {
                    h[p] += wkj * s.v[p];
                    d[p] += wkj * e.v[p];
                }
            }
#pragma unroll
            for (int p = 0; p < kNP; ++p) {
                float spv, sg;
                sp_sig(h[p], spv, sg);
                n0[p] += vk * spv;
                n1[p] += vk * sg * d[p];
            }
        }
    }
    // the eight lanes of a point end with its two sums
    float a2[2], d2[2];
    const bool h4 = lane & 16, h3 = lane & 8;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        a2[i] = (h4 ? n0[2 + i] : n0[i]) + __shfl_xor_sync(kAll, h4 ? n0[i] : n0[2 + i], 16);
        d2[i] = (h4 ? n1[2 + i] : n1[i]) + __shfl_xor_sync(kAll, h4 ? n1[i] : n1[2 + i], 16);
    }
    float a = (h3 ? a2[1] : a2[0]) + __shfl_xor_sync(kAll, h3 ? a2[0] : a2[1], 8);
    float d = (h3 ? d2[1] : d2[0]) + __shfl_xor_sync(kAll, h3 ? d2[0] : d2[1], 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        a += __shfl_xor_sync(kAll, a, o);
        d += __shfl_xor_sync(kAll, d, o);
    }
    const float b = __ldg(b3);
    G = nc.y_s * (a + b * q - nc.y_N0);
    Gp = nc.y_s * (d + b);
    __syncwarp();
}

// r(kappa) = G(q(kappa)) - kappa and dr/dkappa (Eq. (potential_function)) of four points,
// q = psi_e + qcoef (phi - kappa) / f_d(kappa) (Eq. (ostwald_potential)); lane l holds
// point l / 8.  Width 0 is the identity G(q) = q.
__device__ __forceinline__ void r_slope4(const DevNet &yld, const MatF &m, const NcF &nc, float pe, float phi,
                                         float kappa, float &r, float &dr, float &Gp, float *buf, int lane)
{
    const bool dmg = kappa > m.kappa_d;
    const float f = dmg ? expf(-m.eta_d * (kappa - m.kappa_d)) : 1.0f;
    const float q = pe + m.qcoef * (phi - kappa) / f;
    const float dq = m.qcoef * (-1.0f / f + (dmg ? (phi - kappa) * m.eta_d / f : 0.0f));
    float G;
    if (yld.width == 0) {
        G = q;
        Gp = 1.0f;
    } else {
        yield_unit4(yld, nc, q, G, Gp, buf, lane);
    }
    r = G - kappa;
    dr = Gp * dq - 1.0f;
}

// Local damage update of four points in unit mode (Eq. (dd_7_no_nn)), lane l holding point
// l / 8.  The trial value decides loading in FP64 (Phi_d(kappa_n) = G(q(kappa_n)) - kappa_n >
// 0 with the FP64 kappa_n kn_d); a loading point's kappa is the smallest root above kappa_n of
// r(kappa) = G(q(kappa)) - kappa, searched from the warm start kg when that lies above
// kappa_n, to |r| <= 2e-6 max(1, kappa) (or a bracket of 4 FP32 ulps).  On return r' = dr and
// G' = Gp are those at kappa, n_eval counts the point's evaluations; false when local_max
// iterations did not reach the root.  The points iterate together until the last one is
// done, a finished point keeps its values; trial, warm start and iterations share one
// evaluation in the code (three inlined copies cost instruction fetches).
__device__ __forceinline__ bool local_update4(const DevNet &yn, const MatF &m, const NcF &ncp, float pe, float phi,
                                              float kn, double kn_d, float kg, float &kappa, bool &loading,
                                              float &dr, float &Gp, int &n_eval, float *buf, int lane)
{
    // Newton iteration on r(kappa) = G(q(kappa)) - kappa from kappa_n (r > 0 there)
    // or from the warm-start guess, bracketing lazily: lo keeps the last point with
    // r > 0; once a point with r <= 0 is met it becomes hi and the iteration turns
    // into the safeguarded Newton-bisection on [lo, hi].  Before that, a step that
    // is not a forward Newton step (slope >= 0) probes ahead geometrically.
    constexpr unsigned kAll = 0xffffffffu;
    float r = 0.0f, lo = kn, hi = kn, dx_prev = 1.0e30f, dx = 1.0e30f;
    bool have_hi = false, ok = true, todo = true;
    kappa = kn;
    loading = false;
    dr = -1.0f;
    Gp = 0.0f;
    n_eval = 0;
    int it = -2;                      // -2 trial, -1 warm start, then the iterations done
#pragma unroll 1
    while (__any_sync(kAll, todo)) {
        float r1, dr1, G1;
        r_slope4(yn, m, ncp, pe, phi, kappa, r1, dr1, G1, buf, lane);
        if (!todo) continue;
        r = r1;
        dr = dr1;
        Gp = G1;
        ++n_eval;
        if (it == -2) {
            loading = (double)(r + kn) - kn_d > 0.0;
            if (!loading) {
                todo = false;
                continue;
            }
            it = -1;
            if (kg > kn && isfinite(kg)) {
                kappa = kg;
                continue;             // evaluate the warm start
            }
        }
        if (r > 0.0f) {
            lo = kappa;
        } else {
            hi = kappa;
            have_hi = true;
            if (it == -1) dx_prev = dx = hi - lo;
        }
        ++it;
        const float scale = fabsf(kappa) > 1.0f ? fabsf(kappa) : 1.0f;
        if (it >= m.local_max) {
            ok = false;
            todo = false;
            continue;
        }
        if (fabsf(r) <= 2e-6f * scale || (have_hi && (hi - lo) <= 4.0f * kEpsF * scale)) {
            todo = false;
            continue;
        }
        const float newton = kappa - r / dr;
        bool take;
        if (have_hi) {
            take = (newton > lo) && (newton < hi) && (fabsf(2.0f * r) <= fabsf(dx_prev * dr));
        } else {
            // forward Newton step, at most a few times the distance covered so far
            const float cap = 4.0f * ((float)(r > 1e-12f ? r : 1e-12f) + (kappa - kn));
            take = dr < 0.0f && newton > lo && (newton - kappa) <= cap;
        }
        dx_prev = dx;
        if (take) {
            dx = kappa - newton;
            kappa = newton;
        } else if (have_hi) {
            dx = 0.5f * (hi - lo);
            kappa = lo + dx;
        } else {
            const float step = 2.0f * ((kappa - kn) > (r > 1e-12f ? r : 1e-12f) ? (kappa - kn) : (r > 1e-12f ? r : 1e-12f));
            dx = step;
            kappa = lo + step;
        }
    }
    return ok;
}

// element nodes of a warp's batch into shared memory (lane = (element, node)).
// Coordinates and displacements are taken relative to the element's first node,
// the differences formed in FP64: the FP32 kinematics use only their differences
// (sum_a grad N_a = 0), and on a fine mesh far from the origin the absolute FP32
// values would lose the element-size digits.  phi stays absolute (its value enters
// the penalty).  Elements past the end get placeholder nodes and zero dofs.
template <int DIM, class Args>
__device__ __forceinline__ void load_nodes(const Args &A, int64_t e0, float *sX, float *sD, int lane)
{
    using G_ = Geo<DIM>;
    constexpr int NEN = G_::NEN, NDOF = G_::NDOF, EPW = G_::EPW;
    for (int t = lane; t < EPW * NEN; t += 32) {
        int el = t / NEN, a = t % NEN;
        int64_t e = e0 + el;
        if (e < A.n_elems) {
            int32_t n = __ldg(A.conn + e * NEN + a), n0 = __ldg(A.conn + e * NEN);
#pragma unroll
            for (int J = 0; J < DIM; ++J)
                sX[t * DIM + J] = (float)(__ldg(A.X + (int64_t)n * DIM + J) - __ldg(A.X + (int64_t)n0 * DIM + J));
#pragma unroll
            for (int c = 0; c < DIM; ++c)
                sD[t * NDOF + c] =
                    (float)(__ldg(A.dofs + (int64_t)n * NDOF + c) - __ldg(A.dofs + (int64_t)n0 * NDOF + c));
            sD[t * NDOF + DIM] = (float)__ldg(A.dofs + (int64_t)n * NDOF + DIM);
        } else {
#pragma unroll
            for (int J = 0; J < DIM; ++J) sX[t * DIM + J] = (a & 1) ? 1.0f : 0.0f;
#pragma unroll
            for (int c = 0; c < NDOF; ++c) sD[t * NDOF + c] = 0.0f;
        }
    }
}

// dN/dxi and N of every node at every point, [NQ][NEN][4] (threads t0, t0 + n, ...)
template <int DIM>
__device__ __forceinline__ void ref_table(float *ref, int t0, int n)
{
    using G_ = Geo<DIM>;
    for (int t = t0; t < G_::NQ * G_::NEN; t += n) {
        const int q = t / G_::NEN;
        const float xi[3] = {(q & 1) ? kGauss : -kGauss, (q & 2) ? kGauss : -kGauss, (q & 4) ? kGauss : -kGauss};
        float N, dN[3] = {0.0f, 0.0f, 0.0f};
        ref_shape<DIM>(t % G_::NEN, xi, N, dN);
#pragma unroll
        for (int k = 0; k < 3; ++k) ref[t * 4 + k] = dN[k];
        ref[t * 4 + 3] = N;
    }
}

// qp mode: Ji = dxi/dX and the Jacobian determinant, F, phi_q, the reference gradient of
// phi, and x = (I1-3, I2-3, J-1) from C - I = H + H^T + H^T H without cancellation
// (Sec. 3.1f; Eq. (dd_0) inputs); ref: the point's rows of ref_table
template <int DIM>
__device__ __forceinline__ void qp_kinematics(const float *sX, const float *sD, const float *ref, int el,
                                              float (&F)[DIM][DIM], float (&Ji)[DIM][DIM], float (&gx)[DIM],
                                              float &phi, float (&x)[3], float &det)
{
    using G_ = Geo<DIM>;
    constexpr int NEN = G_::NEN, NDOF = G_::NDOF;
    const float *Xe = sX + el * NEN * DIM, *De = sD + el * NEN * NDOF;
    float Jm[DIM][DIM], Gr[DIM][DIM];
    phi = 0.0f;
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
        gx[i] = 0.0f;
#pragma unroll
        for (int k = 0; k < DIM; ++k) Jm[i][k] = Gr[i][k] = 0.0f;
    }
#pragma unroll
    for (int a = 0; a < NEN; ++a) {
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
            const float dN = ref[a * 4 + k];
#pragma unroll
            for (int J = 0; J < DIM; ++J) {
                Jm[J][k] += Xe[a * DIM + J] * dN;
                Gr[J][k] += De[a * NDOF + J] * dN;
            }
            gx[k] += De[a * NDOF + DIM] * dN;
        }
        phi += De[a * NDOF + DIM] * ref[a * 4 + 3];
    }
    if constexpr (DIM == 2) {
        det = Jm[0][0] * Jm[1][1] - Jm[0][1] * Jm[1][0];
        Ji[0][0] = Jm[1][1] / det; Ji[0][1] = -Jm[0][1] / det;
        Ji[1][0] = -Jm[1][0] / det; Ji[1][1] = Jm[0][0] / det;
    } else {
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int i1 = (j + 1) % 3, i2 = (j + 2) % 3, j1 = (i + 1) % 3, j2 = (i + 2) % 3;
                Ji[i][j] = Jm[i1][j1] * Jm[i2][j2] - Jm[i1][j2] * Jm[i2][j1];
            }
        det = Jm[0][0] * Ji[0][0] + Jm[0][1] * Ji[1][0] + Jm[0][2] * Ji[2][0];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) Ji[i][j] /= det;
    }
    float H[DIM][DIM];
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
        for (int J = 0; J < DIM; ++J) {
            float t = 0.0f;
#pragma unroll
            for (int k = 0; k < DIM; ++k) t += Gr[i][k] * Ji[k][J];
            H[i][J] = t;
            F[i][J] = i == J ? t + 1.0f : t;
        }
    float tA = 0.0f, AA = 0.0f, tH = 0.0f, HH = 0.0f;
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
        tH += H[i][i];
#pragma unroll
        for (int j = i; j < DIM; ++j) {
            float t = H[i][j] + H[j][i];
#pragma unroll
            for (int k = 0; k < DIM; ++k) t += H[k][i] * H[k][j];
            if (i == j) {
                tA += t;
                AA += t * t;
                HH += H[i][i] * H[i][i];
            } else {
                AA += 2.0f * t * t;
                HH += 2.0f * H[i][j] * H[j][i];
            }
        }
    }
    x[0] = tA;
    x[1] = 2.0f * tA + 0.5f * (tA * tA - AA);
    x[2] = tH + 0.5f * (tH * tH - HH);
    if constexpr (DIM == 3)
        x[2] += H[0][0] * (H[1][1] * H[2][2] - H[1][2] * H[2][1]) - H[0][1] * (H[1][0] * H[2][2] - H[1][2] * H[2][0]) +
                H[0][2] * (H[1][0] * H[2][1] - H[1][1] * H[2][0]);
}

// network input y (raw: y = x; isochoric: (I1G-3, I2G-3, J-1), Eq. (dd_0)) with
// Tm = dy/dx and T2 = d2y/dx2 (symmetric pairs in sym6 order)
__device__ __forceinline__ void input_map(const MatF &m, const float (&x)[3], float Jdet, float (&Tm)[3][3],
                                          float (&T2)[3][6], float (&yo)[3])
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int j = 0; j < 3; ++j) Tm[i][j] = (i == j) ? 1.0f : 0.0f;
#pragma unroll
        for (int j = 0; j < 6; ++j) T2[i][j] = 0.0f;
    }
    float y[3] = {x[0], x[1], x[2]};
    if (m.energy == GD_ENERGY_ICNN_ISO) {
        // I1G = J^-2/3 I1, I2G = I2^3 / (9 J^4) (Eq. (dd_0)); derivatives wrt (I1-3, I2-3, J-1)
        float L = log1pf(x[2]), E = expf(-2.0f / 3.0f * L), I1 = 3.0f + x[0], I2 = 3.0f + x[1], J = Jdet;
        y[0] = 3.0f * expm1f(-2.0f / 3.0f * L) + x[0] * E;
        y[1] = 3.0f * expm1f(3.0f * log1pf(x[1] / 3.0f) - 4.0f * L);
        float J4 = J * J * J * J;
        Tm[0][0] = E;
        Tm[0][2] = -2.0f / 3.0f * I1 * E / J;
        Tm[1][1] = I2 * I2 / (3.0f * J4);
        Tm[1][2] = -4.0f * I2 * I2 * I2 / (9.0f * J4 * J);
        T2[0][2] = -2.0f / 3.0f * E / J;                       // d2 y1 / dx1 dx3
        T2[0][5] = 10.0f / 9.0f * I1 * E / (J * J);            // d2 y1 / dx3^2
        T2[1][3] = 2.0f * I2 / (3.0f * J4);                    // d2 y2 / dx2^2
        T2[1][4] = -4.0f * I2 * I2 / (3.0f * J4 * J);          // d2 y2 / dx2 dx3
        T2[1][5] = 20.0f * I2 * I2 * I2 / (9.0f * J4 * J * J); // d2 y2 / dx3^2
    }
    yo[0] = y[0];
    yo[1] = y[1];
    yo[2] = y[2];
}

// energy psi_e and its first (ps) and second (ph, sym6) derivatives with respect to
// x = (I1-3, I2-3, J-1), from the network's value, gradient and Hessian o[10] with
// respect to y (or the closed-form Neo-Hookean energy, Sec. 4.1); psi_e = mu_e (N -
// N0 - n x3) + lambda_e ((J-1)^2/J)^2 (Eq. (dd_0))
__device__ __forceinline__ void energy_derivs(const MatF &m, const NcF &nc, const float (&x)[3], float Jdet,
                                              const float *o, const float (&Tm)[3][3], const float (&T2)[3][6],
                                              float (&ps)[3], float (&ph)[6], float &pe)
{
    const float J = Jdet, x3 = x[2];
    if (m.energy == GD_ENERGY_NEO_HOOKE) {
        float L = log1pf(x3);
        pe = 0.5f * m.mu_e * x[0] - m.mu_e * L + 0.5f * m.lambda_e * L * L;
        ps[0] = 0.5f * m.mu_e;
        ps[1] = 0.0f;
        ps[2] = (-m.mu_e + m.lambda_e * L) / J;
#pragma unroll
        for (int c = 0; c < 6; ++c) ph[c] = 0.0f;
        ph[5] = (m.lambda_e + m.mu_e - m.lambda_e * L) / (J * J);
    } else {
        float gy[3] = {o[1], o[2], o[3]};
        float hy[6] = {o[4], o[5], o[6], o[7], o[8], o[9]};
        // chain through the input map: dN/dx = T^T dN/dy, d2N/dx2 = T^T H T + sum_m dN/dy_m d2y_m/dx2
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            float s = 0.0f;
#pragma unroll
            for (int mm = 0; mm < 3; ++mm) s += Tm[mm][i] * gy[mm];
            ps[i] = s;
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = i; j < 3; ++j) {
                float s = 0.0f;
#pragma unroll
                for (int a = 0; a < 3; ++a)
#pragma unroll
                    for (int b = 0; b < 3; ++b) s += Tm[a][i] * hy[sym6(a, b)] * Tm[b][j];
#pragma unroll
                for (int mm = 0; mm < 3; ++mm) s += gy[mm] * T2[mm][sym6(i, j)];
                ph[sym6(i, j)] = s;
            }
        // psi_e = mu_e (N - N0 - n x3) + lambda_e t^2, t = (J-1)^2 / J
        float t = x3 * x3 / J, dt = 1.0f - 1.0f / (J * J), d2t = 2.0f / (J * J * J);
        pe = m.mu_e * (o[0] - nc.psi_N0 - nc.psi_n * x3) + m.lambda_e * t * t;
#pragma unroll
        for (int i = 0; i < 3; ++i) ps[i] *= m.mu_e;
#pragma unroll
        for (int c = 0; c < 6; ++c) ph[c] *= m.mu_e;
        ps[2] += -m.mu_e * nc.psi_n + m.lambda_e * 2.0f * t * dt;
        ph[5] += m.lambda_e * 2.0f * (dt * dt + t * d2t);
    }
}

}  // namespace e32
}  // namespace gd
