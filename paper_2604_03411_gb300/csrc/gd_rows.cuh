// gd_rows.cuh -- a quadrature point's stress and tangent in reference coordinates, and the
// element rows of the residual and of the consistent tangent built from them (shared by the
// FP64 and the mixed-precision element kernels).
//
// D = d(P, Y vector, -Y) / d(grad u, grad phi, phi) is formed once per point, both gradients
// pulled back to the reference element and weighted by J w; a row of the element matrix is
//   K_(a,i),(b,k) = sum_q sum_jl dN_a/dxi_j D_(ij),(kl) dN_b/dxi_l:
// three multiply-adds per entry of D and row, and the sum over the points with dN_b/dxi_l
// factorised over the axes (their values are products of (1 +- 1/sqrt 3) / 2): 20 instead of
// 64 operations per derivative and column.  About 100 operations per row and point, against
// 700 for the closed form of every (a, b) pair.
//
// Paper passages: Sec. 3.1f (element residual), Sec. 2.1f (P, Y vector, Y), Sec. 3.2f (monolithic
// tangent), Sec. 4.1f, Sec. 4.2f Eqs. (dd_0), (dd_1).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gd {
namespace rows {

// Record of a quadrature point for the row mode: every quantity pulled back to the reference
// element and times J w.
template <int DIM>
struct Rec {
    static constexpr int N2 = DIM * DIM, NS = DIM * (DIM + 1) / 2;
    static constexpr int A = 0;                      // d P_ij / d H_kl, symmetric, packed upper triangle of (ij) x (kl)
    static constexpr int B = A + N2 * (N2 + 1) / 2;  // d P_ij / d g_l [ij][l]
    static constexpr int CV = B + N2 * DIM;          // c_d C^-1, packed symmetric
    static constexpr int PE = CV + NS;               // dpsi_e/dF (undamaged, without J w) [ij]
    static constexpr int P = PE + N2;                // stress [ij]
    static constexpr int Y = P + N2;                 // flux [j]
    static constexpr int FDK = Y + DIM;              // f_d' dkappa/dphi
    static constexpr int BCK = FDK + 1;              // beta_d c_kappa
    static constexpr int PP = BCK + 1;               // beta_d (1 - dkappa/dphi)
    static constexpr int PEN = PP + 1;               // beta_d (phi - kappa)
    static constexpr int PENM = PEN + 1;             // beta_d (|phi| + |kappa|): what the penalty's rounding scales with
    static constexpr int SIZE = (PENM + 1) | 1;      // odd stride: one bank (FP64: bank pair) per point
};
// position of (r, c) in a packed symmetric N x N matrix (upper triangle by rows)
template <int N>
__device__ __forceinline__ int sym_pos(int r, int c)
{
    const int lo = r < c ? r : c, hi = r < c ? c : r;
    return lo * N - lo * (lo - 1) / 2 + hi - lo;
}

// 1D shape functions (1 +- 1/sqrt 3) / 2 at the Gauss points
template <class T>
__device__ __forceinline__ constexpr T np() { return (T)0.78867513459481288225; }
template <class T>
__device__ __forceinline__ constexpr T nm() { return (T)0.21132486540518711775; }

// out[b] = sum_q sum_l T[l][q] dN_b/dxi_l(q) (+ sum_q TN[q] N_b(q)), b and q numbered by
// their axis bits (x lowest).  One axis at a time: the derivative's axis sums its two points,
// the others mix them with (1 +- 1/sqrt 3) / 2.
template <bool NPART, class R>
__device__ __forceinline__ void expand_rows(const R (&T)[2][4], const R *TN, R (&out)[4])
{
    const R kNp = np<R>(), kNm = nm<R>();
    // x derivative: S(y), then the y axis; y derivative: S(x), then the x axis
    const R sx0 = T[0][0] + T[0][1], sx1 = T[0][2] + T[0][3];
    const R sy0 = T[1][0] + T[1][2], sy1 = T[1][1] + T[1][3];
    const R hp = R(0.5) * kNp, hm = R(0.5) * kNm;
    const R qx0 = hp * sx0 + hm * sx1, qx1 = hm * sx0 + hp * sx1;       // by = 0, 1
    const R qy0 = hp * sy0 + hm * sy1, qy1 = hm * sy0 + hp * sy1;       // bx = 0, 1
    out[0] = -qx0 - qy0;
    out[1] = qx0 - qy1;
    out[2] = qy0 - qx1;
    out[3] = qx1 + qy1;
    if (NPART) {
        const R a0 = kNp * TN[0] + kNm * TN[1], a1 = kNm * TN[0] + kNp * TN[1];
        const R b0 = kNp * TN[2] + kNm * TN[3], b1 = kNm * TN[2] + kNp * TN[3];
        out[0] += kNp * a0 + kNm * b0;
        out[1] += kNp * a1 + kNm * b1;
        out[2] += kNm * a0 + kNp * b0;
        out[3] += kNm * a1 + kNp * b1;
    }
}
template <bool NPART, class R>
__device__ __forceinline__ void expand_rows(const R (&T)[3][8], const R *TN, R (&out)[8])
{
    const R kNp = np<R>(), kNm = nm<R>();
    const R hp = R(0.5) * kNp, hm = R(0.5) * kNm;
    R Q[3][4];                      // derivative along axis l; the other two axes (lower first)
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        const int u = l == 0 ? 1 : 0, v = l == 2 ? 1 : 2;
        R s[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int q0 = ((m & 1) << u) | ((m >> 1) << v);
            s[m] = T[l][q0] + T[l][q0 | (1 << l)];
        }
        const R a0 = hp * s[0] + hm * s[1], a1 = hm * s[0] + hp * s[1];
        const R b0 = hp * s[2] + hm * s[3], b1 = hm * s[2] + hp * s[3];
        Q[l][0] = kNp * a0 + kNm * b0;
        Q[l][1] = kNp * a1 + kNm * b1;
        Q[l][2] = kNm * a0 + kNp * b0;
        Q[l][3] = kNm * a1 + kNp * b1;
    }
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const int bx = b & 1, by = (b >> 1) & 1, bz = b >> 2;
        const R x = Q[0][by | (bz << 1)], y = Q[1][bx | (bz << 1)], z = Q[2][bx | (by << 1)];
        const R xy = (bx == by) ? x + y : x - y;        // sign of x times the sum
        out[b] = (bx ? xy : -xy) + (bz ? z : -z);
    }
    if (NPART) {
        R a[8], c[8];
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
            a[q] = kNp * TN[q] + kNm * TN[q + 1];
            a[q + 1] = kNm * TN[q] + kNp * TN[q + 1];
        }
#pragma unroll
        for (int z = 0; z < 8; z += 4)
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                c[z + x] = kNp * a[z + x] + kNm * a[z + x + 2];
                c[z + x + 2] = kNm * a[z + x] + kNp * a[z + x + 2];
            }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            out[b] += kNp * c[b] + kNm * c[b + 4];
            out[b + 4] += kNm * c[b] + kNp * c[b + 4];
        }
    }
}
// node with the axis bits l (x lowest): counter-clockwise numbering of each layer
__device__ __forceinline__ int node_of_bits(int l) { return l ^ ((l >> 1) & 1); }

// Record of one point: F, Ji = dxi/dX, gx = the reference gradient of phi, x = (I1-3, I2-3, J-1),
// Jw (0 for a point past the end), ps and ph (sym6) = derivatives of psi_e by x, fd = f_d(kappa);
// Gp = G'(q) and dr = dPhi_d/dkappa of the local solve on loading points.
template <class T, int DIM, class Mat>
__device__ __forceinline__ void point_record(const Mat &m, const T (&F)[DIM][DIM], const T (&Ji)[DIM][DIM],
                                             const T (&gx)[DIM], const T *x, T phi, T Jw, const T *ps, const T *ph,
                                             T kappa, T fd, bool loading, T Gp, T dr, bool tangent, T *rec)
{
    using R_ = Rec<DIM>;
    constexpr int N2 = DIM * DIM;
    const T fdp = kappa > m.kappa_d ? -m.eta_d * fd : T(0);
    const T ck = loading ? -Gp / dr : T(0.0);          // G' / (1 - G' dq/dkappa)
    const T dkdphi = ck * m.qcoef / fd;                  // dq/dphi = qcoef / f_d
    const T J = T(1.0) + x[2], I1 = T(3.0) + x[0], ij = T(1.0) / J;
    // F^-1 = cof(F)^T / J; pulled back to the reference element: F' = F Ji^T (F_iJ Ji_jJ),
    // Fi'_ji = Ji_jJ F^-1_Ji
    T Fp[DIM][DIM], Fi[DIM][DIM], G2[DIM][DIM], h[DIM], mv[DIM], b[DIM][DIM], Mj[DIM][DIM];
    {
        T Fv[DIM][DIM];
        if constexpr (DIM == 2) {
            Fv[0][0] = F[1][1] * ij; Fv[0][1] = -F[0][1] * ij;
            Fv[1][0] = -F[1][0] * ij; Fv[1][1] = F[0][0] * ij;
        } else {
#pragma unroll
            for (int i = 0; i < DIM; ++i)
#pragma unroll
                for (int j = 0; j < DIM; ++j) {
                    const int i1 = (j + 1) % DIM, i2 = (j + 2) % DIM, j1 = (i + 1) % DIM, j2 = (i + 2) % DIM;
                    Fv[i][j] = (F[i1][j1] * F[i2][j2] - F[i1][j2] * F[i2][j1]) * ij;
                }
        }
#pragma unroll
        for (int i = 0; i < DIM; ++i)
#pragma unroll
            for (int j = 0; j < DIM; ++j) {
                T s = T(0.0), t = T(0.0);
#pragma unroll
                for (int K = 0; K < DIM; ++K) {
                    s += F[i][K] * Ji[j][K];
                    t += Ji[j][K] * Fv[K][i];
                }
                Fp[i][j] = s;
                Fi[j][i] = t;
            }
        // F F^T and the metric (delta_JL pulled back)
#pragma unroll
        for (int i = 0; i < DIM; ++i)
#pragma unroll
            for (int k = i; k < DIM; ++k) {
                T s = T(0.0), t = T(0.0);
#pragma unroll
                for (int K = 0; K < DIM; ++K) {
                    s += F[i][K] * F[k][K];
                    t += Ji[i][K] * Ji[k][K];
                }
                b[i][k] = b[k][i] = s;
                Mj[i][k] = Mj[k][i] = t;
            }
    }
    // h = F^-T grad phi (= Fi'^T of the reference gradient), C^-1 grad phi pulled back
#pragma unroll
    for (int i = 0; i < DIM; ++i) {
        T s = T(0.0);
#pragma unroll
        for (int k = 0; k < DIM; ++k) s += Fi[k][i] * gx[k];
        h[i] = s;
    }
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
        T s = T(0.0);
#pragma unroll
        for (int i = 0; i < DIM; ++i) s += Fi[j][i] * h[i];
        mv[j] = s;
    }
    // G^2 = dI2/dF pulled back; P = f_d dpsi_e/dF - c_d h (x) m
    const T ps3J = ps[2] * J, cdw = m.c_d * Jw, fdw = fd * Jw;
#pragma unroll
    for (int i = 0; i < DIM; ++i)
#pragma unroll
        for (int j = 0; j < DIM; ++j) {
            T s = I1 * Fp[i][j];
#pragma unroll
            for (int k = 0; k < DIM; ++k) s -= b[i][k] * Fp[k][j];
            G2[i][j] = T(2.0) * s;
            const T Pe = T(2.0) * ps[0] * Fp[i][j] + ps[1] * G2[i][j] + ps3J * Fi[j][i];
            rec[R_::PE + i * DIM + j] = Pe;
            rec[R_::P + i * DIM + j] = fdw * Pe - cdw * h[i] * mv[j];
        }
#pragma unroll
    for (int j = 0; j < DIM; ++j) rec[R_::Y + j] = cdw * mv[j];
    rec[R_::PEN] = m.beta_d * (phi - kappa) * Jw;
    if (sizeof(T) == 4) rec[R_::PENM] = m.beta_d * (fabs(phi) + fabs(kappa)) * Jw;
    if (tangent) {
        rec[R_::FDK] = fdp * dkdphi * Jw;
        rec[R_::BCK] = m.beta_d * ck * Jw;
        rec[R_::PP] = m.beta_d * (T(1.0) - dkdphi) * Jw;
        T hw[DIM];                                    // c_d J w h
#pragma unroll
        for (int i = 0; i < DIM; ++i) hw[i] = cdw * h[i];
        T Cv[DIM][DIM], Sj[DIM][DIM];
        const T g2w = T(2.0) * fdw * ps[1], g1w = T(2.0) * fdw * ps[0] + g2w * I1;
#pragma unroll
        for (int j = 0; j < DIM; ++j)
#pragma unroll
            for (int l = j; l < DIM; ++l) {
                T ci = T(0.0), c = T(0.0);
                const T mm = Mj[j][l];
#pragma unroll
                for (int i = 0; i < DIM; ++i) {
                    ci += Fi[j][i] * Fi[l][i];             // C^-1
                    c += Fp[i][j] * Fp[i][l];              // C
                }
                Cv[j][l] = Cv[l][j] = cdw * ci;
                rec[R_::CV + sym_pos<DIM>(j, l)] = cdw * ci;
                Mj[j][l] = Mj[l][j] = g2w * mm;
                Sj[j][l] = Sj[l][j] = g1w * mm - g2w * c;
            }
        // d2 psi_e/dF2 with the kappa coupling, times f_d and J w:
        //   sum_mn (f_d psi_mn + f_d' c_kappa psi_m psi_n) G^m G^n + f_d (psi_1 D2(I1) + psi_2 D2(I2) + psi_3 D2(J)),
        //   G^1 = 2 F, G^2 = 2 (I1 F - F F^T F), G^3 = J F^-T,
        //   D2(I1) = 2 d_ik d_JL,  D2(J) = J (F^-1_Ji F^-1_Lk - F^-1_Jk F^-1_Li),
        //   D2(I2) = 2 [2 F_iJ F_kL - F_iL F_kJ + (I1 d_JL - C_JL) d_ik - d_JL b_ik];
        // their products of first derivatives join the G^m G^n sum
        const T ckw = fdp * ck * Jw, g3w = fdw * ps3J;
        const T h11 = T(4.0) * (fdw * ph[0] + ckw * ps[0] * ps[0]) + T(2.0) * g2w;
        const T h12 = T(2.0) * (fdw * ph[1] + ckw * ps[0] * ps[1]);
        const T h13 = T(2.0) * (fdw * ph[2] + ckw * ps[0] * ps[2]) * J;
        const T h22 = fdw * ph[3] + ckw * ps[1] * ps[1];
        const T h23 = (fdw * ph[4] + ckw * ps[1] * ps[2]) * J;
        const T h33 = (fdw * ph[5] + ckw * ps[2] * ps[2]) * J * J + g3w;
        T V[DIM][DIM];                                // c_d J w h_k m_j - f_d psi_3 J J w F^-1_jk
#pragma unroll
        for (int k = 0; k < DIM; ++k)
#pragma unroll
            for (int j = 0; j < DIM; ++j) V[k][j] = hw[k] * mv[j] - g3w * Fi[j][k];
#pragma unroll
        for (int i = 0; i < DIM; ++i)
#pragma unroll
            for (int j = 0; j < DIM; ++j) {
                const int r = DIM * i + j;
                const T t1 = h11 * Fp[i][j] + h12 * G2[i][j] + h13 * Fi[j][i];
                const T t2 = h12 * Fp[i][j] + h22 * G2[i][j] + h23 * Fi[j][i];
                const T t3 = h13 * Fp[i][j] + h23 * G2[i][j] + h33 * Fi[j][i];
#pragma unroll
                for (int c = r; c < N2; ++c) {
                    const int k = c / DIM, l = c % DIM;
                    T v = t1 * Fp[k][l] + t2 * G2[k][l] + t3 * Fi[l][k];
                    if (i == k) v += Sj[j][l];
                    v -= Mj[j][l] * b[i][k];
                    v -= g2w * Fp[i][l] * Fp[k][j];
                    v += Fi[l][i] * V[k][j];
                    v += hw[i] * mv[l] * Fi[j][k];
                    v += Cv[j][l] * (h[i] * h[k]);
                    rec[R_::A + sym_pos<N2>(r, c)] = v;
                }
#pragma unroll
                for (int l = 0; l < DIM; ++l)
                    rec[R_::B + r * DIM + l] = -(cdw * mv[j] * Fi[l][i] + h[i] * Cv[j][l]);
            }
    }
}

// Residual (FP64 atomics) and tangent rows of the elements of eight points (HEX8: one element,
// Q4: two) from element e_first on, lane = element row (node a, dof i); rec: the points' records,
// ref: [NQ][NEN][4] dN/dxi and N at the points.  A.Rabs (may be null): the magnitudes of the
// residual terms.
template <class T, int DIM, class Args>
__device__ __forceinline__ void add_rows(const Args &A, const T *rec, const T *ref, int64_t e_first, int lane)
{
    using R_ = Rec<DIM>;
    constexpr int NEN = DIM == 2 ? 4 : 8, NQ = NEN, NDOF = DIM + 1, ND = NEN * NDOF, N2 = DIM * DIM, EP = 8 / NQ;
    const int ee = lane / ND, row = lane % ND, a = row / NDOF, i = row % NDOF;
    const int64_t e = e_first + ee;
    if (lane >= EP * ND || e >= A.n_elems) return;
    const T *R0 = rec + ee * NQ * R_::SIZE;
    const bool pr = i == DIM;                        // a phi row
    T Rr = T(0), Mr = T(0);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const T *rq = R0 + q * R_::SIZE, *c = ref + (q * NEN + a) * 4;
        const T *pj = rq + (pr ? R_::Y : R_::P + i * DIM);
#pragma unroll
        for (int j = 0; j < DIM; ++j) {
            Rr += c[j] * pj[j];
            if (sizeof(T) == 4) Mr += fabs(c[j] * pj[j]);
        }
        if (pr) {
            Rr += c[3] * rq[R_::PEN];
            if (sizeof(T) == 4) Mr += fabs(c[3]) * rq[R_::PENM];
        }
    }
    const int32_t na = __ldg(A.conn + e * NEN + a);
    if (A.R) atomicAdd(A.R + (int64_t)na * NDOF + i, (double)Rr);
    if (sizeof(T) == 4 && A.Rabs) atomicAdd(A.Rabs + (int64_t)na * NDOF + i, (double)Mr);
    if (!A.tangent) return;
    const int32_t rb = __ldg(A.rowptr + (int64_t)na * NDOF);
    const int64_t off = (int64_t)i * (__ldg(A.rowptr + (int64_t)na * NDOF + 1) - rb);
    const int32_t *sl = A.slot + (e * NEN + a) * NEN;
    // FP32 rows of 4 dofs per node are added four columns at a time (16-byte aligned values)
    const bool vec = sizeof(T) == 4 && NDOF == 4 && A.vals32 && (reinterpret_cast<uintptr_t>(A.vals32) & 15) == 0;
    T X[DIM][NQ], K[NEN];
    float Kv[NEN][4];
    auto put = [&](int k) {
#pragma unroll
        for (int l = 0; l < NEN; ++l) {
            if (vec) {
                Kv[l][k & 3] = (float)K[l];
                continue;
            }
            const int64_t pos = (int64_t)__ldg(sl + node_of_bits(l)) + off + k;
            if (A.vals) atomicAdd(A.vals + pos, (double)K[l]);
            else atomicAdd(A.vals32 + pos, (float)K[l]);
        }
    };
    constexpr int UNR = sizeof(T) == 4 ? DIM : 1;
#pragma unroll UNR
    for (int k = 0; k < DIM; ++k) {
        // columns (b, u_k)
        int at[DIM][DIM];
#pragma unroll
        for (int j = 0; j < DIM; ++j)
#pragma unroll
            for (int l = 0; l < DIM; ++l)
                at[j][l] = pr ? R_::B + (DIM * k + l) * DIM + j : R_::A + sym_pos<N2>(DIM * i + j, DIM * k + l);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const T *rq = R0 + q * R_::SIZE, *c = ref + (q * NEN + a) * 4;
#pragma unroll
            for (int l = 0; l < DIM; ++l) {
                T t = T(0);
#pragma unroll
                for (int j = 0; j < DIM; ++j) t += c[j] * rq[at[j][l]];
                X[l][q] = t;
            }
            if (pr) {
                const T nb = c[3] * rq[R_::BCK];
#pragma unroll
                for (int l = 0; l < DIM; ++l) X[l][q] -= nb * rq[R_::PE + DIM * k + l];
            }
        }
        expand_rows<false>(X, (const T *)nullptr, K);
        put(k);
    }
    // columns (b, phi)
    T XN[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const T *rq = R0 + q * R_::SIZE, *c = ref + (q * NEN + a) * 4;
        T t = T(0);
#pragma unroll
        for (int l = 0; l < DIM; ++l) {
            T s = T(0);
#pragma unroll
            for (int j = 0; j < DIM; ++j)
                s += c[j] * rq[pr ? R_::CV + sym_pos<DIM>(j, l) : R_::B + (DIM * i + j) * DIM + l];
            X[l][q] = s;
            t += c[l] * rq[R_::PE + (pr ? 0 : i) * DIM + l];
        }
        XN[q] = pr ? c[3] * rq[R_::PP] : rq[R_::FDK] * t;
    }
    expand_rows<true>(X, XN, K);
    put(DIM);
    if (vec)
#pragma unroll
        for (int l = 0; l < NEN; ++l) {
            float *p = A.vals32 + (int64_t)__ldg(sl + node_of_bits(l)) + off;
            asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(Kv[l][0]),
                         "f"(Kv[l][1]), "f"(Kv[l][2]), "f"(Kv[l][3])
                         : "memory");
        }
}

}  // namespace rows
}  // namespace gd
