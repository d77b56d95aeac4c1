// gd_asm_fp64.cu -- FP64 element kernel of the gradient-enhanced damage model.
//
// A CTA of KW warps owns NP quadrature points (NP / 8 HEX8 or NP / 4 Q4 elements) and switches
// between three lane mappings:
//   qp mode    thread = quadrature point (NP threads in an order that rotates with the
//              batch): kinematics, invariants, energy chain, stress and the point's tangent
//              in reference coordinates;
//   net mode   warp = four points at a time, eight lanes each: both ICNN layers of the
//              energy network (value, gradient by forward tangents, Hessian by one reverse
//              sweep through layer 2) and every yield-network evaluation of the local damage
//              solve, whose points iterate in lockstep (gd_net_fp64.cuh);
//   row mode   warp = the elements of eight points, lane = element row (node a, dof i): the
//              rows of the residual and of the consistent tangent, scattered into CSR
//              through the slot map.
//
// The FP64 pipe bounds the kernel (1.7 lanes per clock and SM), so the design spends as few
// FP64 operations as it can:
//  - The point's tangent is formed once per point as the derivative D of (P, Y vector, -Y)
//    with respect to (grad u, grad phi, phi) in reference coordinates, and the element rows
//    are built from it (gd_rows.cuh): about 100 operations per row and point, against 700 for
//    the closed form of every (a, b) pair.
//  - The networks run in 64-bit fixed point (gd_fixed.cuh).
// Measured (GB300, gd_assemble with tangent; before: FP64 networks one point at a time with
// a lane per unit, closed-form rows): 140,400 points of HEX8, both widths 64, 33.6 -> 5.75 ms;
// 159,744 of Q4, widths 32, 10.2 -> 2.55 ms; 256 of Q4, widths 16 and 8, 1.21 -> 0.087 ms;
// residual alone of 32,640 HEX8 points, widths 24 and 40, 3.53 -> 0.52 ms.  (Without the
// trust in the fixed-point sums being checked and with one scale for all first-layer and
// one for all output weights: 2 to 3 % less.)  Built for 16 warps per SM: 128
// registers, with 180-340 bytes of spills in 2D and 560-990 in 3D, the points' state in shared
// memory.  Width-64 HEX8 networks need 64 KB per CTA of four warps, so that 12 warps are
// resident there (8 with 255 registers: 7.5 ms where 12 took 5.75).  Instruction latency is the
// leading stall, the FP64 pipe 30 % busy.
//
// Paper passages: Sec. 3.1 (F, phi_q, grad phi_q, element residual, Table
// kernel_inputs), Sec. 2.1 (P, Y vector, Y), Sec. 2.2 and Sec. 3.2 Eq. (dd_7_no_nn)
// (local update, KKT), Sec. 3.2 (monolithic scheme), Sec. 4.1 (degradation,
// gradient and penalty energies, Eq. (ostwald_potential)), Sec. 4.2 Eqs. (dd_0),
// (dd_1), (Gq_NN), (dd_7).
#include <cuda_runtime.h>

#include "gd_elem32.cuh"
#include "gd_internal.cuh"
#include "gd_net_fp64.cuh"
#include "gd_rows.cuh"

namespace gd {
namespace {

// Trial yield values farther than this (relative to max(1, kappa_n)), and than what FP32 may be
// off by, from zero are decided by the FP32 evaluation; closer ones by an FP64 evaluation.  The
// FP32 network's relative error is a few 1e-7 (two sums of up to 64 positive terms) and __expf's, up to
// 1.4e-7 |h| (8e-6 at h = -57), of N(0) / N'(0) where the network hardly depends on q, and of q's
// terms near full damage.
constexpr double kTrialMargin = 1e-4, kTrialRel = 8e-6;

// the normalising constants of this kernel's own evaluation
__device__ __forceinline__ NetConst own_consts(const NetConst &c)
{
    NetConst r = c;
    r.psi_N0 = c.psi_N0_own;
    r.psi_n = c.psi_n_own;
    r.y_N0 = c.y_N0_own;
    r.y_s = c.y_s_own;
    return r;
}

// What a point keeps between its qp phases, in doubles (registers would halve the resident
// warps)
template <int DIM>
struct State {
    static constexpr int F = 0, JI = F + DIM * DIM, GX = JI + DIM * DIM, X = GX + DIM, PHI = X + 3, DET = PHI + 1;
    static constexpr int PS = DET + 1, PH = PS + 3;
    static constexpr int SIZE = (PH + 6) | 1;
};

// shared-memory layout of a CTA of KW warps with NP points, in doubles
template <int DIM, int NP, int KW>
struct Smem {
    using G_ = Geo<DIM>;
    static constexpr int EL = NP / G_::NQ;
    static constexpr int X = 0;                                      // [EL][NEN][DIM]
    static constexpr int D = X + EL * G_::NEN * DIM;                 // [EL][NEN][NDOF]
    static constexpr int REF = D + EL * G_::NEN * G_::NDOF;          // [NQ][NEN][4] dN/dxi, N
    static constexpr int IN = REF + G_::NQ * G_::NEN * 4;            // [NP][4] network input / psi_e, phi, kappa_n
    static constexpr int OUT = IN + NP * 4;                          // [NP][10] network output / local update
    static constexpr int ST = OUT + NP * 10;                         // [NP] State
    static constexpr int U = (ST + NP * State<DIM>::SIZE + 1) / 2 * 2;   // network buffers, then the points' records
    __host__ __device__ static int net(int wmax) { return (int)(grp::buf_bytes(wmax) / 8); }
    __host__ __device__ static int total(int wmax)
    {
        const int n = KW * net(wmax), r = NP * rows::Rec<DIM>::SIZE;
        return U + ((n > r ? n : r) + 1) / 2 * 2;
    }
};

// Local damage update (Eq. (dd_7_no_nn)) of the CTA's points p0 .. p0 + 3 that
// belong to specimen sn: psi_e, phi, kappa_n at sIn[p 4 ..], results (kappa, loading, G',
// dPhi/dkappa, failed) to sOut[p 10 ..].  A point's lanes hold its state alike; the points step
// together, every evaluation running for the points that still need it.  Returns the
// lane's share of the FP64 evaluations.
template <int DIM>
__device__ __forceinline__ int local_update(const AsmArgs &A, const e32::MatF &mf, int64_t e0, int p0, int sn,
                                            const double *sIn, double *sOut, unsigned char *nbuf, int lane)
{
    constexpr int NQ = Geo<DIM>::NQ;
    constexpr unsigned kAll = 0xffffffffu;
    const int p = p0 + lane / grp::kLanes;
    const int64_t e_p = e0 + p / NQ;
    const bool need = e_p < A.n_elems && spec_of(A, e_p < A.n_elems ? e_p : A.n_elems - 1) == sn;
    const DevNet &yn = yld_of(A, sn);
    const int yp = grp::path_of(yn);
    const NetConst nc = own_consts(A.netc[sn]);
    const e32::NcF nf = e32::ncf(nc);
    const int local_max = A.mat.local_max;
    const double pe = sIn[p * 4], phi = sIn[p * 4 + 1], kn = sIn[p * 4 + 2];
    const float pef = (float)pe, phf = (float)phi, knf = (float)kn;
    double kappa = kn, r = 0.0, dr = -1.0, Gp = 0.0;
    bool fail = false;
    int n_eval = 0;
    // Trial Phi_d(kappa_n): the FP32 network decides points clearly off the yield
    // surface, an FP64 evaluation the others.
    float r32, dr32, Gp32, mag;
    grp::residual32(mf, yn, nf, pef, phf, knf, r32, dr32, Gp32, mag, nbuf, lane);
    const double scale_n = fabs(kn) > 1.0 ? fabs(kn) : 1.0;
    bool load = need && r32 > 0.0f;
    const bool close = need && !(fabs((double)r32) > kTrialMargin * scale_n + kTrialRel * (double)mag);
    if (__any_sync(kAll, close)) {
        double rt, drt, gt;
        grp::residual<true>(A.mat, yn, yp, nc, pe, phi, kn, rt, drt, gt, nbuf, lane, close);
        if (close) {
            ++n_eval;
            r = rt;
            dr = drt;
            Gp = gt;
            load = rt > 0.0;
            r32 = (float)rt;
            dr32 = (float)drt;
        }
    }
    // The root in FP32 (the lazily bracketed Newton iteration of the mixed kernels, from the
    // warm start), then FP64: one value-only evaluation and a Newton step with the FP32 slope
    // (its relative error, ~1e-6, times a correction of ~1e-6 leaves ~1e-12), then one full
    // evaluation and a last Newton step; the slope and G' of that evaluation feed the tangent
    // (they change by ~1e-12 relative over the last step).  Where the FP32 root is not close
    // enough, the FP64 bracketed iteration takes over from it.  Both iterations also stop on
    // the next Newton correction |r / r'| (the step test of the safeguarded Newton-bisection;
    // FP32: 2e-6 relative, FP64: 4 ulp) once the root is bracketed within 1e-2 relative or the
    // iteration converges from one side: near full damage r' grows like 1 / f_d, and r itself
    // cannot get below its rounding.  (A wide bracket does not qualify: far past the root,
    // where f_d underflows, r' is huge and the correction meaningless.)
    float k32 = knf;
    bool ok32 = false;
    if (__any_sync(kAll, load)) {
        const float kg = load && A.kappa_guess ? (float)__ldg(A.kappa_guess + e0 * NQ + p) : knf;
        bool run = load, warm = load && kg > knf && isfinite(kg);
        float lo = knf, hi = knf, dx = 1.0e30f, dx_prev = 1.0e30f;
        bool have_hi = false, took_newton = false;
        int it = 0;
        if (warm) k32 = kg;
        else if (r32 > 0.0f) lo = k32;
        else {
            hi = k32;
            have_hi = true;
            dx = dx_prev = hi - lo;
        }
        while (__any_sync(kAll, run)) {
            if (run && !warm) {
                const float scale = fabsf(k32) > 1.0f ? fabsf(k32) : 1.0f;
                if (it >= local_max) {
                    run = false;
                } else if (fabsf(r32) <= 2e-6f * scale || (have_hi && (hi - lo) <= 4.0f * e32::kEpsF * scale) ||
                           (fabsf(r32) <= 2e-6f * scale * fabsf(dr32) &&
                            (have_hi ? (hi - lo) <= 1e-2f * scale
                                     : (took_newton && fabsf(2.0f * r32) <= fabsf(dx * dr32))))) {
                    run = false;
                    ok32 = true;
                } else {
                    const float newton = k32 - r32 / dr32;
                    const float rr = r32 > 1e-12f ? r32 : 1e-12f;
                    bool take;
                    if (have_hi) take = newton > lo && newton < hi && fabsf(2.0f * r32) <= fabsf(dx_prev * dr32);
                    else take = dr32 < 0.0f && newton > lo && (newton - k32) <= 4.0f * (rr + (k32 - knf));
                    dx_prev = dx;
                    took_newton = take;
                    if (take) {
                        dx = k32 - newton;
                        k32 = newton;
                    } else if (have_hi) {
                        dx = 0.5f * (hi - lo);
                        k32 = lo + dx;
                    } else {
                        dx = 2.0f * ((k32 - knf) > rr ? (k32 - knf) : rr);
                        k32 = lo + dx;
                    }
                }
            }
            if (!__any_sync(kAll, run)) break;
            float re, dre, ge;
            grp::residual32(mf, yn, nf, pef, phf, k32, re, dre, ge, mag, nbuf, lane);
            if (run) {
                r32 = re;
                dr32 = dre;
                if (r32 > 0.0f) lo = k32;
                else {
                    hi = k32;
                    have_hi = true;
                }
                if (warm) {
                    warm = false;
                    dx = dx_prev = have_hi ? hi - lo : 1.0e30f;
                } else {
                    ++it;
                }
            }
        }
    }
    bool polish = load && ok32 && isfinite(k32) && (double)k32 >= kn && dr32 < 0.0f;
    bool done = !load;
    if (__any_sync(kAll, polish)) {
        const double sc = fabs((double)k32) > 1.0 ? fabs((double)k32) : 1.0;
        double r0, d0, g0;
        grp::residual<false>(A.mat, yn, yp, nc, pe, phi, (double)k32, r0, d0, g0, nbuf, lane, polish);
        if (polish) ++n_eval;
        polish = polish && fabs(r0) <= 1e-4 * sc;
        const double k1 = polish ? (double)k32 - r0 / (double)dr32 : kn;
        grp::residual<true>(A.mat, yn, yp, nc, pe, phi, k1, r0, d0, g0, nbuf, lane, polish);
        if (polish) {
            ++n_eval;
            r = r0;
            dr = d0;
            Gp = g0;
            if (k1 >= kn && fabs(r) <= 1e-9 * sc && dr < 0.0) {
                const double k2 = fabs(r) <= 1e-13 * sc ? k1 : k1 - r / dr;
                kappa = k2 >= kn ? k2 : kn;
                done = true;
            }
        }
    }
    if (__any_sync(kAll, !done)) {
        // FP64 lazily bracketed Newton iteration from kappa_n, then the FP32 result (the
        // iteration of the FP64 reference path)
        const double kgd = isfinite(k32) ? (double)k32 : kn;
        bool run = !done, ok = done;
        int stage = kgd > kn ? 0 : 1;        // 0: at kappa_n, a guess follows; 1: first point; 2: iterating
        double lo = kn, hi = kn, dx = 1.0e30, dx_prev = 1.0e30;
        bool have_hi = false, took_newton = false;
        int it = 0;
        while (__any_sync(kAll, run)) {
            double re, dre, ge;
            grp::residual<true>(A.mat, yn, yp, nc, pe, phi, kappa, re, dre, ge, nbuf, lane, run);
            if (run) {
                ++n_eval;
                r = re;
                dr = dre;
                Gp = ge;
                if (stage == 0) {
                    kappa = kgd;
                    stage = 1;
                    continue;
                }
                if (r > 0.0) lo = kappa;
                else {
                    hi = kappa;
                    have_hi = true;
                }
                if (stage == 1) {
                    dx = dx_prev = have_hi ? hi - lo : 1.0e30;
                    stage = 2;
                } else {
                    ++it;
                }
                const double scale = fabs(kappa) > 1.0 ? fabs(kappa) : 1.0;
                const double ulp4 = 4.0 * 2.220446049250313e-16 * scale;
                if (it >= local_max) {
                    run = false;
                } else if (fabs(r) <= 1e-13 * scale || (have_hi && (hi - lo) <= ulp4) ||
                           (fabs(r) <= ulp4 * fabs(dr) &&
                            (have_hi ? (hi - lo) <= 1e-2 * scale : (took_newton && fabs(2.0 * r) <= fabs(dx * dr))))) {
                    run = false;
                    ok = true;
                } else {
                    const double newton = kappa - r / dr;
                    const double rr = r > 1e-12 ? r : 1e-12;
                    bool take;
                    if (have_hi) take = newton > lo && newton < hi && fabs(2.0 * r) <= fabs(dx_prev * dr);
                    // forward Newton step, at most a few times the distance covered so far
                    else take = dr < 0.0 && newton > lo && (newton - kappa) <= 4.0 * (rr + (kappa - kn));
                    dx_prev = dx;
                    took_newton = take;
                    if (take) {
                        dx = kappa - newton;
                        kappa = newton;
                    } else if (have_hi) {
                        dx = 0.5 * (hi - lo);
                        kappa = lo + dx;
                    } else {
                        dx = 2.0 * ((kappa - kn) > rr ? (kappa - kn) : rr);
                        kappa = lo + dx;
                    }
                }
            }
        }
        if (!ok) fail = true;
    }
    if (need && lane % grp::kLanes == 0) {
        double *o = sOut + p * 10;
        o[0] = kappa;
        o[1] = load ? 1.0 : 0.0;
        o[2] = Gp;
        o[3] = dr;
        o[4] = fail ? 1.0 : 0.0;
    }
    return lane % grp::kLanes == 0 ? n_eval : 0;
}

// NP points and KW warps per CTA (a launch-shape choice: see launch_dim); built for 16 warps
// per SM
template <int DIM, int NP, int KW>
__global__ void __launch_bounds__(32 * KW, 16 / KW) asm_fp64_kernel(AsmArgs A)
{
    using G_ = Geo<DIM>;
    using S_ = Smem<DIM, NP, KW>;
    using R_ = rows::Rec<DIM>;
    using P_ = State<DIM>;
    constexpr int NEN = G_::NEN, NQ = G_::NQ, NDOF = G_::NDOF, EL = S_::EL;
    extern __shared__ __align__(16) double smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double *sX = smem + S_::X, *sD = smem + S_::D, *sRef = smem + S_::REF, *sIn = smem + S_::IN, *sOut = smem + S_::OUT;
    double *sRec = smem + S_::U;
    unsigned char *nbuf = reinterpret_cast<unsigned char *>(smem + S_::U + warp * S_::net(A.wmax));
    const MatConst &m = A.mat;
    for (int t = threadIdx.x; t < NQ * NEN; t += 32 * KW) {
        const int qq = t / NEN, a = t % NEN;
        const double xi[3] = {(qq & 1) ? kGauss : -kGauss, (qq & 2) ? kGauss : -kGauss, (qq & 4) ? kGauss : -kGauss};
        double N, dN[3] = {0.0, 0.0, 0.0};
        ref_shape<DIM>(a, xi, N, dN);
#pragma unroll
        for (int k = 0; k < 3; ++k) sRef[t * 4 + k] = dN[k];
        sRef[t * 4 + 3] = N;
    }
    const int64_t e_last = A.n_elems - 1;
    const int psi_path = m.energy != GD_ENERGY_NEO_HOOKE && !A.psi_tab ? grp::path_of(A.psi) : 0;

    const int64_t n_batches = (A.n_elems + EL - 1) / EL;
    for (int64_t batch = blockIdx.x; batch < n_batches; batch += gridDim.x) {
        const int64_t e0 = batch * EL;
        __syncthreads();
        for (int t = threadIdx.x; t < EL * NEN; t += 32 * KW) {
            const int64_t e = e0 + t / NEN;
            if (e < A.n_elems) {
                const int32_t n = __ldg(A.conn + e * NEN + t % NEN);
#pragma unroll
                for (int J = 0; J < DIM; ++J) sX[t * DIM + J] = __ldg(A.X + (int64_t)n * DIM + J);
#pragma unroll
                for (int c = 0; c < NDOF; ++c) sD[t * NDOF + c] = __ldg(A.dofs + (int64_t)n * NDOF + c);
            } else {
                // a unit element without displacement
                const int a = t % NEN;
#pragma unroll
                for (int J = 0; J < DIM; ++J) sX[t * DIM + J] = node_sgn(a, J) > 0.0 ? 1.0 : 0.0;
#pragma unroll
                for (int c = 0; c < NDOF; ++c) sD[t * NDOF + c] = 0.0;
            }
        }
        __syncthreads();

        // ================= qp mode: kinematics and invariants =================
        // the threads that hold the points move on by one warp per batch, so that the SM's
        // four quarters share this mode's FP64 work
        const int pt = (threadIdx.x + 32 * (int)((batch / gridDim.x + blockIdx.x) % KW)) % (32 * KW);
        const bool qp = pt < NP;
        const int el = pt / NQ, q = pt % NQ;
        const int64_t e_me = e0 + el;
        const bool valid = qp && e_me < A.n_elems;
        const double *ref = sRef + q * NEN * 4;
        double *st = smem + S_::ST + pt * P_::SIZE;
        if (qp) {
            double Ji[DIM][DIM], gx[DIM], x[3], phi = 0.0, det;
            const double *Xe = sX + el * NEN * DIM, *De = sD + el * NEN * NDOF;
            double Jm[DIM][DIM], Gr[DIM][DIM];
#pragma unroll
            for (int i = 0; i < DIM; ++i) {
                gx[i] = 0.0;
#pragma unroll
                for (int k = 0; k < DIM; ++k) Jm[i][k] = Gr[i][k] = 0.0;
            }
#pragma unroll
            for (int a = 0; a < NEN; ++a) {
#pragma unroll
                for (int k = 0; k < DIM; ++k) {
                    const double dN = ref[a * 4 + k];
#pragma unroll
                    for (int J = 0; J < DIM; ++J) {
                        Jm[J][k] += Xe[a * DIM + J] * dN;
                        Gr[J][k] += De[a * NDOF + J] * dN;
                    }
                    gx[k] += De[a * NDOF + DIM] * dN;
                }
                phi += De[a * NDOF + DIM] * ref[a * 4 + 3];
            }
            if (DIM == 2) {
                det = Jm[0][0] * Jm[1][1] - Jm[0][1] * Jm[1][0];
                const double di = 1.0 / det;
                Ji[0][0] = Jm[1][1] * di; Ji[0][1] = -Jm[0][1] * di;
                Ji[1][0] = -Jm[1][0] * di; Ji[1][1] = Jm[0][0] * di;
            } else {
#pragma unroll
                for (int i = 0; i < DIM; ++i)
#pragma unroll
                    for (int j = 0; j < DIM; ++j) {
                        const int i1 = (j + 1) % DIM, i2 = (j + 2) % DIM, j1 = (i + 1) % DIM, j2 = (i + 2) % DIM;
                        Ji[i][j] = Jm[i1][j1] * Jm[i2][j2] - Jm[i1][j2] * Jm[i2][j1];
                    }
                det = 0.0;
#pragma unroll
                for (int k = 0; k < DIM; ++k) det += Jm[0][k] * Ji[k][0];
                const double di = 1.0 / det;
#pragma unroll
                for (int i = 0; i < DIM; ++i)
#pragma unroll
                    for (int j = 0; j < DIM; ++j) Ji[i][j] *= di;
            }
            // H = grad u; C - I = H + H^T + H^T H; invariants without cancellation
            double H[DIM][DIM];
#pragma unroll
            for (int i = 0; i < DIM; ++i)
#pragma unroll
                for (int J = 0; J < DIM; ++J) {
                    double s = 0.0;
#pragma unroll
                    for (int k = 0; k < DIM; ++k) s += Gr[i][k] * Ji[k][J];
                    H[i][J] = s;
                    st[P_::F + i * DIM + J] = i == J ? s + 1.0 : s;
                    st[P_::JI + i * DIM + J] = Ji[i][J];
                }
            double tA = 0.0, AA = 0.0, tH = 0.0, HH = 0.0;
#pragma unroll
            for (int i = 0; i < DIM; ++i) {
                tH += H[i][i];
#pragma unroll
                for (int j = i; j < DIM; ++j) {
                    double s = H[i][j] + H[j][i];
#pragma unroll
                    for (int k = 0; k < DIM; ++k) s += H[k][i] * H[k][j];
                    if (i == j) {
                        tA += s;
                        AA += s * s;
                        HH += H[i][i] * H[i][i];
                    } else {
                        AA += 2.0 * s * s;
                        HH += 2.0 * H[i][j] * H[j][i];
                    }
                }
            }
            x[0] = tA;
            x[1] = 2.0 * tA + 0.5 * (tA * tA - AA);
            x[2] = tH + 0.5 * (tH * tH - HH);
            if constexpr (DIM == 3)
                x[2] += H[0][0] * (H[1][1] * H[2][2] - H[1][2] * H[2][1]) -
                        H[0][1] * (H[1][0] * H[2][2] - H[1][2] * H[2][0]) +
                        H[0][2] * (H[1][0] * H[2][1] - H[1][1] * H[2][0]);
#pragma unroll
            for (int k = 0; k < DIM; ++k) st[P_::GX + k] = gx[k];
#pragma unroll
            for (int k = 0; k < 3; ++k) st[P_::X + k] = x[k];
            st[P_::PHI] = phi;
            st[P_::DET] = det;
            // network input (raw or isochoric map: I1G = J^-2/3 I1, I2G = I2^3 / (9 J^4), Eq. (dd_0))
            double y[3] = {x[0], x[1], x[2]};
            if (m.energy == GD_ENERGY_ICNN_ISO) {
                const double L = log1p(x[2]);
                y[0] = 3.0 * expm1(-2.0 / 3.0 * L) + x[0] * exp(-2.0 / 3.0 * L);
                y[1] = 3.0 * expm1(3.0 * log1p(x[1] / 3.0) - 4.0 * L);
            }
            sIn[pt * 4 + 0] = y[0];
            sIn[pt * 4 + 1] = y[1];
            sIn[pt * 4 + 2] = y[2];
        }
        __syncthreads();

        // ================= net mode: energy network =================
        // (points of different specimens take turns: a round's networks are uniform)
        // specimens of the points p0 .. p0 + 3: s0 .. s1 (none past the last element)
        auto specimens = [&](int p0, int &s0, int &s1) {
            const int64_t ea = e0 + p0 / NQ, eb = e0 + (p0 + grp::kPts - 1) / NQ;
            s0 = 0;
            s1 = -1;
            if (ea < A.n_elems) {
                s0 = spec_of(A, ea);
                s1 = spec_of(A, eb < e_last ? eb : e_last);
            }
        };
        if (m.energy != GD_ENERGY_NEO_HOOKE) {
#pragma unroll 1
            for (int p0 = warp * grp::kPts; p0 < NP; p0 += KW * grp::kPts) {
                int s0, s1;
                specimens(p0, s0, s1);
                const int64_t e_p = e0 + (p0 + lane / grp::kLanes) / NQ;
                const int sp = e_p <= e_last ? spec_of(A, e_p) : -1;
                for (int sn = s0; sn <= s1; ++sn) {
                    const DevNet &net = psi_of(A, sn);
                    grp::energy(net, A.psi_tab ? grp::path_of(net) : psi_path, sIn + p0 * 4, sOut + p0 * 10, nbuf, lane,
                                sp == sn, A.tangent != 0);
                }
            }
        }
        __syncthreads();

        // ================= qp mode: energy derivatives wrt (I1-3, I2-3, J-1) =================
        if (qp) {
            const double x3 = st[P_::X + 2], J = 1.0 + x3;
            double ps[3], ph[6], pe;
            if (m.energy == GD_ENERGY_NEO_HOOKE) {
                double L = log1p(x3);
                pe = 0.5 * m.mu_e * st[P_::X] - m.mu_e * L + 0.5 * m.lambda_e * L * L;
                ps[0] = 0.5 * m.mu_e;
                ps[1] = 0.0;
                ps[2] = (-m.mu_e + m.lambda_e * L) / J;
#pragma unroll
                for (int c = 0; c < 6; ++c) ph[c] = 0.0;
                ph[5] = (m.lambda_e + m.mu_e - m.lambda_e * L) / (J * J);
            } else {
                const double *o = sOut + pt * 10;
                const NetConst nc = own_consts(A.netc[valid ? spec_of(A, e_me) : 0]);
#pragma unroll
                for (int i = 0; i < 3; ++i) ps[i] = o[1 + i];
#pragma unroll
                for (int c = 0; c < 6; ++c) ph[c] = o[4 + c];
                if (m.energy == GD_ENERGY_ICNN_ISO) {
                    // chain through the input map: dN/dx = T^T dN/dy, d2N/dx2 = T^T H T + sum_m dN/dy_m d2y_m/dx2,
                    // T = dy/dx and T2 = d2y/dx2 for x = (I1-3, I2-3, J-1)
                    double Tm[3][3], T2[3][6];
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
#pragma unroll
                        for (int j = 0; j < 3; ++j) Tm[i][j] = (i == j) ? 1.0 : 0.0;
#pragma unroll
                        for (int j = 0; j < 6; ++j) T2[i][j] = 0.0;
                    }
                    const double E = exp(-2.0 / 3.0 * log1p(x3)), I1 = 3.0 + st[P_::X], I2 = 3.0 + st[P_::X + 1];
                    const double J4 = J * J * J * J;
                    Tm[0][0] = E;
                    Tm[0][2] = -2.0 / 3.0 * I1 * E / J;
                    Tm[1][1] = I2 * I2 / (3.0 * J4);
                    Tm[1][2] = -4.0 * I2 * I2 * I2 / (9.0 * J4 * J);
                    T2[0][2] = -2.0 / 3.0 * E / J;                       // d2 y1 / dx1 dx3
                    T2[0][5] = 10.0 / 9.0 * I1 * E / (J * J);            // d2 y1 / dx3^2
                    T2[1][3] = 2.0 * I2 / (3.0 * J4);                    // d2 y2 / dx2^2
                    T2[1][4] = -4.0 * I2 * I2 / (3.0 * J4 * J);          // d2 y2 / dx2 dx3
                    T2[1][5] = 20.0 * I2 * I2 * I2 / (9.0 * J4 * J * J); // d2 y2 / dx3^2
                    const double gy[3] = {ps[0], ps[1], ps[2]};
                    const double hy[6] = {ph[0], ph[1], ph[2], ph[3], ph[4], ph[5]};
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        double s = 0.0;
#pragma unroll
                        for (int mm = 0; mm < 3; ++mm) s += Tm[mm][i] * gy[mm];
                        ps[i] = s;
                    }
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int j = i; j < 3; ++j) {
                            double s = 0.0;
#pragma unroll
                            for (int a = 0; a < 3; ++a)
#pragma unroll
                                for (int b = 0; b < 3; ++b) s += Tm[a][i] * hy[sym6(a, b)] * Tm[b][j];
#pragma unroll
                            for (int mm = 0; mm < 3; ++mm) s += gy[mm] * T2[mm][sym6(i, j)];
                            ph[sym6(i, j)] = s;
                        }
                }
                // psi_e = mu_e (N - N0 - n x3) + lambda_e t^2, t = (J-1)^2 / J
                const double ij = 1.0 / J;
                double t = x3 * x3 * ij, dt = 1.0 - ij * ij, d2t = 2.0 * ij * ij * ij;
                pe = m.mu_e * (o[0] - nc.psi_N0 - nc.psi_n * x3) + m.lambda_e * t * t;
#pragma unroll
                for (int i = 0; i < 3; ++i) ps[i] *= m.mu_e;
#pragma unroll
                for (int c = 0; c < 6; ++c) ph[c] *= m.mu_e;
                ps[2] += -m.mu_e * nc.psi_n + m.lambda_e * 2.0 * t * dt;
                ph[5] += m.lambda_e * 2.0 * (dt * dt + t * d2t);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) st[P_::PS + i] = ps[i];
#pragma unroll
            for (int c = 0; c < 6; ++c) st[P_::PH + c] = ph[c];
            sIn[pt * 4 + 0] = pe;
            sIn[pt * 4 + 1] = st[P_::PHI];
            sIn[pt * 4 + 2] = valid ? __ldg(A.kappa_n + e_me * NQ + q) : 0.0;
        }
        __syncthreads();

        // ================= net mode: local damage update =================
        if (A.kappa_fixed) {
            // frozen history (staggered scheme): the point keeps the given kappa
            if (qp) {
                double *o = sOut + pt * 10;
                o[0] = valid ? __ldg(A.kappa_fixed + e_me * NQ + q) : 0.0;
                o[1] = 0.0;
                o[2] = 0.0;
                o[3] = -1.0;
                o[4] = 0.0;
            }
        } else {
            const e32::MatF mf = e32::to_f(A.mat);
            int n_eval = 0;
#pragma unroll 1
            for (int p0 = warp * grp::kPts; p0 < NP; p0 += KW * grp::kPts) {
                int s0, s1;
                specimens(p0, s0, s1);
                for (int sn = s0; sn <= s1; ++sn)
                    n_eval += local_update<DIM>(A, mf, e0, p0, sn, sIn, sOut, nbuf, lane);
            }
            n_eval = __reduce_add_sync(0xffffffffu, n_eval);
            if (lane == 0 && n_eval) atomicAdd(A.counters + 2, n_eval);
        }
        __syncthreads();

        // ================= qp mode: stress and the point's tangent =================
        bool loading = false;
        if (qp) {
            const double *o = sOut + pt * 10;
            const double kappa = o[0];
            loading = valid && o[1] > 0.5;
            if (valid) {
                if (A.kappa_new) A.kappa_new[e_me * NQ + q] = kappa;
                if (A.loading) A.loading[e_me * NQ + q] = loading ? 1 : 0;
                if (o[4] > 0.5) atomicAdd(A.counters, 1);
            }
            double F[DIM][DIM], Ji[DIM][DIM], gx[DIM];
#pragma unroll
            for (int i = 0; i < DIM; ++i) {
                gx[i] = st[P_::GX + i];
#pragma unroll
                for (int j = 0; j < DIM; ++j) {
                    F[i][j] = st[P_::F + i * DIM + j];
                    Ji[i][j] = st[P_::JI + i * DIM + j];
                }
            }
            const double fd = kappa > m.kappa_d ? fx::exp_neg(m.eta_d * (kappa - m.kappa_d)) : 1.0;
            rows::point_record<double, DIM>(m, F, Ji, gx, st + P_::X, st[P_::PHI], valid ? st[P_::DET] : 0.0, st + P_::PS,
                                            st + P_::PH, kappa, fd, loading, o[2], o[3], A.tangent != 0,
                                            sRec + pt * R_::SIZE);
        }
        {
            const unsigned n_load = __ballot_sync(0xffffffffu, loading);
            if (lane == 0 && n_load) atomicAdd(A.counters + 1, __popc(n_load));
        }
        __syncthreads();

        // ================= row mode: element residual and tangent =================
        if (warp < NP / 8)
            rows::add_rows<double, DIM>(A, sRec + warp * 8 * R_::SIZE, sRef, e0 + warp * (8 / NQ), lane);
    }
}

template <int DIM, int NP, int KW>
cudaError_t launch_cta(const AsmArgs &a, int num_sms, const AsmTune &t, cudaStream_t s)
{
    using S_ = Smem<DIM, NP, KW>;
    auto fn = asm_fp64_kernel<DIM, NP, KW>;
    const size_t sm = (size_t)S_::total(a.wmax) * sizeof(double);
    int dev = 0, optin = 0;
    cudaError_t e0 = cudaGetDevice(&dev);
    if (e0 == cudaSuccess) e0 = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e0 != cudaSuccess) return e0;
    if (sm > (size_t)optin) return cudaErrorInvalidConfiguration;   // this CTA width does not fit
    cudaError_t err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    int per_sm = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * KW, sm);
    if (err != cudaSuccess) return err;
    if (per_sm < 1) per_sm = 1;
    if (t.cta_per_sm > 0 && t.cta_per_sm < per_sm) per_sm = t.cta_per_sm;
    const int64_t need = (a.n_elems + S_::EL - 1) / S_::EL;
    int64_t grid = (int64_t)num_sms * per_sm;
    if (grid > need) grid = need;
    if (t.grid_max > 0 && grid > t.grid_max) grid = t.grid_max;
    if (grid < 1) grid = 1;
    fn<<<(unsigned)grid, 32 * KW, sm, s>>>(a);
    return cudaGetLastError();
}

// The requested CTA width (gd_autotune's choice of warps, eight points each), or the widest
// narrower one whose shared memory fits.  Meshes that would leave SMs without a CTA take
// narrower ones, at the end eight points on two warps (one round of the networks each).
template <int DIM>
cudaError_t launch_dim(const AsmArgs &a, int num_sms, const AsmTune &t, cudaStream_t s)
{
    int warps = t.warps >= 8 ? 8 : t.warps >= 4 ? 4 : 2;
    const int64_t points = a.n_elems * Geo<DIM>::NQ;
    if (!t.exact)
        while (warps > 1 && (points + 8 * warps - 1) / (8 * warps) < num_sms) warps /= 2;
    cudaError_t e = cudaErrorInvalidConfiguration;
    if (warps == 8) e = launch_cta<DIM, 64, 8>(a, num_sms, t, s);
    if (warps == 4 || (e == cudaErrorInvalidConfiguration && warps > 4 && !t.exact))
        e = launch_cta<DIM, 32, 4>(a, num_sms, t, s);
    if (warps == 2 || (e == cudaErrorInvalidConfiguration && warps > 2 && !t.exact))
        e = launch_cta<DIM, 16, 2>(a, num_sms, t, s);
    if (warps == 1) e = launch_cta<DIM, 8, 2>(a, num_sms, t, s);
    return e;
}

}  // namespace

cudaError_t launch_assemble_fp64(int dim, const AsmArgs &a, int num_sms, cudaStream_t s, const AsmTune &t)
{
    if (a.n_elems <= 0) return cudaSuccess;
    return dim == 2 ? launch_dim<2>(a, num_sms, t, s) : launch_dim<3>(a, num_sms, t, s);
}

// ---------------------------------------------------------------------------
// network constants: N(0), n (S(C=I) = 0), N_k(0), s = 1/N_k'(0)  (Sec. 4.2), by the FP64
// functions and by the element kernel's.  Two roundings of N(0) would leave psi_e and G near
// +-1e-16 at a point without strain, and half of those above zero: "loading".
// ---------------------------------------------------------------------------
namespace {
__global__ void prep_nets_kernel(DevNet psi, DevNet yld, int energy, NetConst *out)
{
    __shared__ __align__(16) double buf[grp::buf_bytes(kMaxWidth) / sizeof(double)];
    __shared__ double sY[grp::kPts * 4], sO[grp::kPts * 10];
    const int lane = threadIdx.x;
    const bool need = lane < grp::kLanes;            // one point
    NetConst nc;
    nc.psi_N0 = 0.0;
    nc.psi_n = 0.0;
    nc.y_N0 = 0.0;
    nc.y_s = 1.0;
    nc.psi_N0_own = nc.psi_n_own = nc.y_N0_own = 0.0;
    nc.y_s_own = 1.0;
    if (energy != GD_ENERGY_NEO_HOOKE && psi.width > 0) {
        double x0[3] = {0.0, 0.0, 0.0}, o[10];
        psi_net_unit(psi, x0, o, buf, lane);
        nc.psi_N0 = o[0];
        // dI1/dC = I, dI2/dC = 2 I, dJ/dC = I/2 at C = I (raw); dI1G/dC = dI2G/dC = 0 (Eq. (dd_1))
        nc.psi_n = (energy == GD_ENERGY_ICNN_RAW) ? 2.0 * o[1] + 4.0 * o[2] + o[3] : o[3];
        if (lane < grp::kPts * 4) sY[lane] = 0.0;
        __syncwarp();
        grp::energy(psi, grp::path_of(psi), sY, sO, reinterpret_cast<unsigned char *>(buf), lane, need, false);
        nc.psi_N0_own = sO[0];
        nc.psi_n_own = (energy == GD_ENERGY_ICNN_RAW) ? 2.0 * sO[1] + 4.0 * sO[2] + sO[3] : sO[3];
        __syncwarp();
    }
    if (yld.width > 0) {
        NetConst unit;
        unit.y_N0 = 0.0;
        unit.y_s = 1.0;
        double G, Gp;
        yield_unit(yld, unit, 0.0, G, Gp, buf, lane);   // raw N_k(0), N_k'(0)
        nc.y_N0 = G;
        nc.y_s = 1.0 / Gp;
        const double2 n = grp::yield<true>(yld.p, yld.W2T, yld.fx, yld.width, grp::path_of(yld), 0.0,
                                             reinterpret_cast<unsigned char *>(buf), lane, need);
        nc.y_N0_own = __shfl_sync(0xffffffffu, n.x, 0);
        nc.y_s_own = 1.0 / __shfl_sync(0xffffffffu, n.y, 0);
    }
    if (lane == 0) *out = nc;
}

__global__ void transpose_kernel(const double *W2, double *W2T, int w)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < w * w) {
        int k = t / w, j = t % w;
        W2T[j * w + k] = W2[k * w + j];
    }
}
}  // namespace

cudaError_t launch_prep_nets(const DevNet &psi, const DevNet &yld, int energy, NetConst *out, cudaStream_t s)
{
    prep_nets_kernel<<<1, 32, 0, s>>>(psi, yld, energy, out);
    return cudaGetLastError();
}

namespace {
__global__ void to_float_kernel(const double *in, float *out, int n)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) out[t] = (float)in[t];
}
}  // namespace

cudaError_t launch_net_to_float(const DevNet &net, cudaStream_t s)
{
    if (net.width <= 0) return cudaSuccess;
    to_float_kernel<<<(net.n_params + 255) / 256, 256, 0, s>>>(net.p, net.pf, net.n_params);
    const int ww = net.width * net.width;
    to_float_kernel<<<(ww + 255) / 256, 256, 0, s>>>(net.W2T, net.W2Tf, ww);
    return cudaGetLastError();
}

namespace {
// Networks with a unit whose pre-activation at zero argument lies below this (the tail of softplus
// begins at -3.47; strain and driving force raise it) are evaluated with the tails at once.
// A pass over 39,936 Q4 points, widths 32: 0.64 ms without the tails, 0.71-0.77 with them, 1.25-1.34
// where they follow a first evaluation; 64,000 HEX8 points, widths 64: 2.85, 3.30-3.45, 5.0 ms.
constexpr double kTailRest = -3.4;

// fixed-point copies of one network (layout of fx::Net): each row of W2 and W2^T, each column of
// W1 and each output weight is scaled by the power of two above its largest magnitude
__global__ void net_fixed_kernel(DevNet net)
{
    using namespace fx;
    const int w = net.width, wp = pad16(w), n_in = net.n_in, t0 = threadIdx.x, nt = blockDim.x;
    const double *W1 = net.p, *W2 = W1 + w * n_in + w, *w3 = W2 + w * w + w * n_in + w;
    const Net f = net_of(net.fx, w);
    int *e = const_cast<int *>(f.e);
    for (int t = t0; t < 3 * w + 3; t += nt) {
        double m = 0.0;
        if (t < w) for (int j = 0; j < w; ++j) m = fmax(m, fabs(W2[t * w + j]));
        else if (t < 2 * w) for (int k = 0; k < w; ++k) m = fmax(m, fabs(W2[k * w + t - w]));
        else if (t < 3 * w) m = fabs(w3[t - 2 * w]);
        else if (t - 3 * w < n_in) for (int j = 0; j < w; ++j) m = fmax(m, fabs(W1[j * n_in + t - 3 * w]));
        e[t] = m == 0.0 ? kZero : bound_exp(m);
    }
    __syncthreads();
    int path = kPlain;
    for (int t = t0; t < net.n_params; t += nt)
        if (!isfinite(net.p[t])) path = kFp64;
    for (int t = t0; t < 3 * w + 3; t += nt)
        if (e[t] > kLargest) path = kFp64;
    const double *b1 = W1 + w * n_in, *b2 = w3 - w;
    for (int t = t0; t < w; t += nt) {
        double h = b2[t];
        for (int j = 0; j < w; ++j) h += W2[t * w + j] * softplus(b1[j]);
        if (path == kPlain && (b1[t] < kTailRest || h < kTailRest)) path = kTails;
    }
    const bool fp64 = __syncthreads_or(path == kFp64), tails = __syncthreads_or(path == kTails);
    if (t0 == 0) e[3 * w + kPath] = fp64 ? kFp64 : tails ? kTails : kPlain;
    if (t0 < 3) {
        int m = kZero;
        for (int k = 0; k < w; ++k) m = max(m, e[t0 * w + k]);
        e[3 * w + kRows + t0] = m;
    }
    __syncthreads();
    for (int t = t0; t < w * wp; t += nt) {
        const int a = t / wp, b = t % wp, at = a * wp + perm16(b);
        const bool in = b < w;
        const_cast<int2 *>(f.W2)[at] = in ? limbs(from_double(W2[b * w + a], kBits - e[b])) : make_int2(0, 0);
        const_cast<int2 *>(f.W2T)[at] = in ? limbs(from_double(W2[a * w + b], kBits - e[w + b])) : make_int2(0, 0);
        const_cast<float *>(f.W2P)[at] = in ? (float)W2[b * w + a] : 0.0f;
    }
    for (int j = t0; j < w; j += nt) {
        double v[3] = {0.0, 0.0, 0.0};
        for (int c = 0; c < n_in && c < 3; ++c) v[c] = W1[j * n_in + c];
        for (int c = 0; c < 4; ++c) const_cast<i64 *>(f.W1)[4 * j + c] = c < 3 ? from_double(v[c], 62 - e[3 * w + c]) : 0;
        const_cast<i64 *>(f.w3)[j] = from_double(w3[j], 62 - e[2 * w + j]);
        double *ww = const_cast<double *>(f.WW) + 6 * j;
        ww[0] = v[0] * v[0]; ww[1] = v[0] * v[1]; ww[2] = v[0] * v[2];
        ww[3] = v[1] * v[1]; ww[4] = v[1] * v[2]; ww[5] = v[2] * v[2];
    }
}
}  // namespace

size_t net_fixed_bytes(int width) { return fx::net_bytes(width); }

cudaError_t launch_net_fixed(const DevNet &net, cudaStream_t s)
{
    if (net.width <= 0) return cudaSuccess;
    net_fixed_kernel<<<1, 256, 0, s>>>(net);
    return cudaGetLastError();
}

cudaError_t launch_transpose(const DevNet &net, cudaStream_t s)
{
    if (net.width <= 0) return cudaSuccess;
    const int w = net.width;
    const double *W2 = net.p + w * net.n_in + w;
    transpose_kernel<<<(w * w + 255) / 256, 256, 0, s>>>(W2, net.W2T, w);
    return cudaGetLastError();
}

}  // namespace gd
