// gd_asm_mixed.cu -- FP32 element kernel of the gradient-enhanced damage model
// (GD_MIXED): the same three lane mappings as the FP64 kernel with FP32 element
// math and FP32 networks; FP64 is kept for the loading/unloading decision
// (Phi_d(kappa_n) > 0 evaluated as FP64 G - kappa_n), the history kappa, and the
// residual accumulation (FP32 element rows added into the FP64 global residual).
// Tangent values are FP32.
//
// One warp owns a batch of 32 quadrature points (4 HEX8 or 8 Q4 elements) and
// switches between three lane mappings:
//   qp mode    lane = quadrature point: kinematics, invariants, energy chain,
//              stress and the per-point records of the tangent;
//   unit mode  lane = network unit, four points of an element at a time: both ICNN
//              layers of the energy network (value, gradient by forward tangents,
//              Hessian by one reverse sweep through layer 2) and every yield-network
//              evaluation of the local damage solve, whose points iterate together;
//   row mode   lane = element row (node a, dof i): the row of the consistent
//              tangent and of the residual, accumulated over the points of one
//              element and scattered into CSR through the slot map.
//
// Instruction fetches bound the kernel (10 of 14 cycles per issued instruction with 190 KB of
// code, 16 warps per SM in different modes), so each network is in the code once, loops over
// units and rows stay loops, and the three kinds of yield evaluation share one call.
// Measured (96 specimens, 690,000 Q4 points, widths 16 to 32, GB300): one point at a time
// 3.37 ms; four at a time with three copies 3.29, with one copy and loops 1.84.
//
// Paper passages: Sec. 3.1f (F, phi_q, grad phi_q, element residual, Table
// kernel_inputs), Sec. 2.1f (P, Y vector, Y), Sec. 2.2f and Sec. 3.2f Eq. (dd_7_no_nn)
// (local update, KKT), Sec. 3.2f (monolithic scheme), Sec. 4.1f (degradation,
// gradient and penalty energies, Eq. (ostwald_potential)), Sec. 4.2f Eqs. (dd_0),
// (dd_1), (Gq_NN), (dd_7).
#include <cuda_runtime.h>

#include "gd_elem32.cuh"

namespace gd {
namespace {

using namespace e32;

// Energy network in unit mode for four points of one element: value, gradient and Hessian of
// N(x) (Sec. 4.2f ICNN).  Layer 1 and the gradient columns of layer 2 are
// forward tangents; the second derivative uses the identity
//   d2N/dx2 = sum_k w3_k sp''(h2_k) g_k g_k^T + sum_j v_j sp''(h1_j) W1_j W1_j^T,
//   g_k = dh2_k/dx,  v = W2^T (w3 o sp'(h2)),
// so layer 2 costs 4 forward columns and 1 reverse column per point.
// in: [4][4] inputs, out: [4][10] results (shared memory).
__device__ __forceinline__ void psi_net_unit4(const DevNet &net, const float *in, float *out, float *buf, int lane)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int w = net.width;
    const float *W1 = net.pf, *b1 = W1 + 3 * w, *W2 = b1 + w, *A2 = W2 + w * w, *b2 = A2 + 3 * w, *w3 = b2 + w,
                 *a3 = w3 + w;
    float4 *sZ = reinterpret_cast<float4 *>(buf);         // [w][kNP]: value, three tangents
    PVec *sU = reinterpret_cast<PVec *>(buf + 16 * w);        // [w]
    PVec *sE = sU + w;                                       // [w] sp'' of layer 1 (own units)
    float x[kNP][3];
#pragma unroll
    for (int p = 0; p < kNP; ++p)
#pragma unroll
        for (int i = 0; i < 3; ++i) x[p][i] = in[p * 4 + i];
#pragma unroll 1
    for (int t = 0; t < kUnits; ++t) {
        const int j = lane + 32 * t;
        if (j < w) {
            const float a0 = __ldg(W1 + 3 * j), a1 = __ldg(W1 + 3 * j + 1), a2 = __ldg(W1 + 3 * j + 2), b = __ldg(b1 + j);
            PVec e1;
#pragma unroll
            for (int p = 0; p < kNP; ++p) {
                float sg, spv;
                sp_sig(b + a0 * x[p][0] + a1 * x[p][1] + a2 * x[p][2], spv, sg);
                sZ[j * kNP + p] = make_float4(spv, sg * a0, sg * a1, sg * a2);
                e1.v[p] = sg * (1.0f - sg);
            }
            sE[j] = e1;
        }
    }
    __syncwarp();
    float acc[kNP][10];
#pragma unroll
    for (int p = 0; p < kNP; ++p)
#pragma unroll
        for (int c = 0; c < 10; ++c) acc[p][c] = 0.0f;
#pragma unroll 1
    for (int t = 0; t < kUnits; ++t) {
        const int k = lane + 32 * t;
        if (k < w) {
            const float c0 = __ldg(A2 + 3 * k), c1 = __ldg(A2 + 3 * k + 1), c2 = __ldg(A2 + 3 * k + 2),
                        bk = __ldg(b2 + k), wk = __ldg(w3 + k);
            float h[kNP], g0[kNP], g1[kNP], g2[kNP];
#pragma unroll
            for (int p = 0; p < kNP; ++p) {
                h[p] = bk + c0 * x[p][0] + c1 * x[p][1] + c2 * x[p][2];
                g0[p] = c0;
                g1[p] = c1;
                g2[p] = c2;
            }
            const float *col = net.W2Tf + k;     // W2[k][j] = W2T[j*w + k]
#pragma unroll 2
            for (int j = 0; j < w; ++j) {
                const float wkj = __ldg(col + j * w);
#pragma unroll
                for (int p = 0; p < kNP; ++p) {
                    const float4 z = sZ[j * kNP + p];
                    h[p] += wkj * z.x;
                    g0[p] += wkj * z.y;
                    g1[p] += wkj * z.z;
                    g2[p] += wkj * z.w;
                }
            }
            PVec u;
#pragma unroll
            for (int p = 0; p < kNP; ++p) {
                float sg, spv;
                sp_sig(h[p], spv, sg);
                const float e2 = wk * sg * (1.0f - sg);
                u.v[p] = wk * sg;
                acc[p][0] += wk * spv;
                acc[p][1] += wk * sg * g0[p];
                acc[p][2] += wk * sg * g1[p];
                acc[p][3] += wk * sg * g2[p];
                acc[p][4] += e2 * g0[p] * g0[p];
                acc[p][5] += e2 * g0[p] * g1[p];
                acc[p][6] += e2 * g0[p] * g2[p];
                acc[p][7] += e2 * g1[p] * g1[p];
                acc[p][8] += e2 * g1[p] * g2[p];
                acc[p][9] += e2 * g2[p] * g2[p];
            }
            sU[k] = u;
        }
    }
    __syncwarp();
#pragma unroll 1
    for (int t = 0; t < kUnits; ++t) {
        const int j = lane + 32 * t;
        if (j < w) {
            float v[kNP];
#pragma unroll
            for (int p = 0; p < kNP; ++p) v[p] = 0.0f;
            const float *row = W2 + j;          // W2[k][j] at k*w + j
#pragma unroll 4
            for (int k = 0; k < w; ++k) {
                const float wkj = __ldg(row + k * w);
                const PVec u = sU[k];
#pragma unroll
                for (int p = 0; p < kNP; ++p) v[p] += wkj * u.v[p];
            }
            const float a0 = __ldg(W1 + 3 * j), a1 = __ldg(W1 + 3 * j + 1), a2 = __ldg(W1 + 3 * j + 2);
            const PVec e1 = sE[j];
#pragma unroll
            for (int p = 0; p < kNP; ++p) {
                const float c = v[p] * e1.v[p];
                acc[p][4] += c * a0 * a0;
                acc[p][5] += c * a0 * a1;
                acc[p][6] += c * a0 * a2;
                acc[p][7] += c * a1 * a1;
                acc[p][8] += c * a1 * a2;
                acc[p][9] += c * a2 * a2;
            }
        }
    }
    // Sums over the units.  Each exchange halves the values a lane holds (4 points x 10, 2 x 10,
    // 10, 5): 45 exchanges for the four points where a butterfly per value takes 200.  The eight
    // lanes 8 p .. 8 p + 7 end with point p, the upper four of them with values 5..9.
    float r2[2][10], r1[10], rv[5];
    const bool h4 = lane & 16, h3 = lane & 8;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int c = 0; c < 10; ++c)
            r2[i][c] = (h4 ? acc[2 + i][c] : acc[i][c]) + __shfl_xor_sync(kAll, h4 ? acc[i][c] : acc[2 + i][c], 16);
#pragma unroll
    for (int c = 0; c < 10; ++c) r1[c] = (h3 ? r2[1][c] : r2[0][c]) + __shfl_xor_sync(kAll, h3 ? r2[0][c] : r2[1][c], 8);
    const bool up = lane & 4;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        rv[c] = (up ? r1[5 + c] : r1[c]) + __shfl_xor_sync(kAll, up ? r1[c] : r1[5 + c], 4);
        rv[c] += __shfl_xor_sync(kAll, rv[c], 2);
        rv[c] += __shfl_xor_sync(kAll, rv[c], 1);
    }
    if ((lane & 3) == 0) {
        const int p = lane >> 3;
        if (!up) {
            const float s0 = __ldg(a3), s1 = __ldg(a3 + 1), s2 = __ldg(a3 + 2);
            rv[0] += s0 * in[p * 4] + s1 * in[p * 4 + 1] + s2 * in[p * 4 + 2];
            rv[1] += s0;
            rv[2] += s1;
            rv[3] += s2;
        }
#pragma unroll
        for (int c = 0; c < 5; ++c) out[p * 10 + (up ? 5 : 0) + c] = rv[c];
    }
    __syncwarp();
}

// floats of a warp's shared-memory scratch
template <int DIM>
__host__ __device__ constexpr int scratch_floats(int wmax)
{
    using G_ = Geo<DIM>;
    const int rec = 32 * rows::Rec<DIM>::SIZE, unit = unit_floats(wmax);
    return G_::EPW * G_::NEN * (DIM + G_::NDOF) + (rec > unit ? rec : unit) + 32 * 4 + 32 * 10;
}

template <int DIM, int KW>
__global__ void __launch_bounds__(32 * KW, (DIM == 2 ? 16 : 12) / KW) asm_fp32_kernel(AsmArgs A)
{
    using G_ = Geo<DIM>;
    using R_ = rows::Rec<DIM>;
    constexpr int NEN = G_::NEN, NQ = G_::NQ, NDOF = G_::NDOF, EPW = G_::EPW;
    extern __shared__ float smem_f[];
    float *sRef = smem_f;                            // [NQ][NEN][4]
    float *smem = smem_f + NQ * NEN * 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wmax = A.wmax;
    // per-warp scratch
    const int scratch = scratch_floats<DIM>(wmax);
    float *ws = smem + warp * scratch;
    float *sX = ws;                                  // [EPW][NEN][DIM]
    float *sD = sX + EPW * NEN * DIM;                // [EPW][NEN][NDOF]
    float *sIn = sD + EPW * NEN * NDOF;              // [32][4]: network input x (3), then kappa out
    float *sOut = sIn + 32 * 4;                      // [32][10]: N, grad, Hess / local-solve results
    float *sBuf = sOut + 32 * 10;                    // unit-mode buffers, then
    float *sRec = sBuf;                              // [32] records of the points
    const MatF m = to_f(A.mat);
    ref_table<DIM>(sRef, threadIdx.x, 32 * KW);
    __syncthreads();

    int evals = 0, n_loading = 0;        // the lane's share of the counters
    const int64_t n_batches = (A.n_elems + EPW - 1) / EPW;
    for (int64_t batch = (int64_t)blockIdx.x * KW + warp; batch < n_batches;
         batch += (int64_t)gridDim.x * KW) {
        const int64_t e0 = batch * EPW;
        load_nodes<DIM>(A, e0, sX, sD, lane);
        __syncwarp();

        // ================= qp mode: kinematics and invariants =================
        const int el = lane / NQ, q = lane % NQ;
        const int64_t e_me = e0 + el;
        const bool valid = e_me < A.n_elems;
        const NcF nc = ncf(A.netc[valid ? spec_of(A, e_me) : 0]);
        float F[DIM][DIM], Ji[DIM][DIM], gx[DIM], phi, x[3], det;
        qp_kinematics<DIM>(sX, sD, sRef + q * NEN * 4, el, F, Ji, gx, phi, x, det);
        const float Jdet = 1.0f + x[2];
        // network input (raw or isochoric map)
        float Tm[3][3], T2[3][6];   // dy/dx and d2y/dx2 of the iso map (raw: identity)
        {
            float y[3];
            input_map(m, x, Jdet, Tm, T2, y);
            sIn[lane * 4 + 0] = y[0];
            sIn[lane * 4 + 1] = y[1];
            sIn[lane * 4 + 2] = y[2];
        }
        __syncwarp();

        // ================= unit mode: energy network =================
        if (m.energy != GD_ENERGY_NEO_HOOKE) {
#pragma unroll 1
            for (int p = 0; p < 32; p += 4) {
                if (e0 + p / NQ >= A.n_elems) break;
                const DevNet &net = psi_of(A, spec_of(A, e0 + p / NQ));
                psi_net_unit4(net, sIn + p * 4, sOut + p * 10, sBuf, lane);
            }
        }
        __syncwarp();

        // ================= qp mode: energy derivatives wrt (I1-3, I2-3, J-1) =================
        float ps[3], ph[6], pe;
        energy_derivs(m, nc, x, Jdet, sOut + lane * 10, Tm, T2, ps, ph, pe);
        sIn[lane * 4 + 0] = pe;
        sIn[lane * 4 + 1] = phi;
        sIn[lane * 4 + 2] = valid ? (float)__ldg(A.kappa_n + e_me * NQ + q) : 0.0f;
        __syncwarp();

        // ================= unit mode: local damage update per point =================
        if (A.kappa_fixed) {
            // frozen history (staggered scheme): the point keeps the given kappa
            float *o = sOut + lane * 10;
            o[0] = valid ? (float)__ldg(A.kappa_fixed + e_me * NQ + q) : 0.0f;
            o[1] = 0.0f;
            o[2] = 0.0f;
            o[3] = -1.0f;
            o[4] = 0.0f;
            o[5] = 0.0f;
        } else
#pragma unroll 1
        for (int p4 = 0; p4 < 32; p4 += 4) {
            if (e0 + p4 / NQ >= A.n_elems) break;
            const int p = p4 + (lane >> 3);                 // the lane's point
            const float ppe = sIn[p * 4], pphi = sIn[p * 4 + 1], kn = sIn[p * 4 + 2];
            const int sp = spec_of(A, e0 + p4 / NQ);
            const DevNet &yn = yld_of(A, sp);
            const NcF ncp = ncf(A.netc[sp]);
            const double kn_d = __ldg(A.kappa_n + e0 * NQ + p);
            const float kg = A.kappa_guess ? (float)__ldg(A.kappa_guess + e0 * NQ + p) : kn;
            float kappa, dr, Gp;
            bool loading;
            int n_eval;
            const bool ok = local_update4(yn, m, ncp, ppe, pphi, kn, kn_d, kg, kappa, loading, dr, Gp, n_eval, sBuf, lane);
            if ((lane & 7) == 0) {
                float *o = sOut + p * 10;
                evals += n_eval;
                o[0] = kappa;
                o[1] = loading ? 1.0f : 0.0f;
                o[2] = Gp;
                o[3] = dr;
                o[4] = ok ? 0.0f : 1.0f;
                o[5] = loading ? 0.0f : 1.0f;   // elastic: keep the FP64 history exactly
            }
        }
        __syncwarp();

        // ================= qp mode: stress and records =================
        {
            const float *o = sOut + lane * 10;
            const float kappa = o[0];
            const bool loading = o[1] > 0.5f;
            if (valid) {
                if (A.kappa_new) {
                    const double kn_d = __ldg(A.kappa_n + e_me * NQ + q);
                    A.kappa_new[e_me * NQ + q] = A.kappa_fixed ? __ldg(A.kappa_fixed + e_me * NQ + q)
                                                 : o[5] > 0.5f ? kn_d : fmax(kn_d, (double)kappa);
                }
                if (A.loading) A.loading[e_me * NQ + q] = loading ? 1 : 0;
                if (o[4] > 0.5f) atomicAdd(A.counters, 1);
                if (loading) ++n_loading;
            }
            const float fd = kappa > m.kappa_d ? expf(-m.eta_d * (kappa - m.kappa_d)) : 1.0f;
            rows::point_record<float, DIM>(m, F, Ji, gx, x, phi, valid ? det : 0.0f, ps, ph, kappa, fd, loading, o[2],
                                           o[3], A.tangent != 0, sRec + lane * R_::SIZE);
        }
        __syncwarp();

        // ================= row mode: element residual and tangent =================
#pragma unroll 1
        for (int u = 0; u < 4; ++u) rows::add_rows<float, DIM>(A, sRec + u * 8 * R_::SIZE, sRef, e0 + u * (8 / NQ), lane);
        __syncwarp();
    }
    evals = __reduce_add_sync(0xffffffffu, evals);
    n_loading = __reduce_add_sync(0xffffffffu, n_loading);
    if (lane == 0) {
        if (evals) atomicAdd(A.counters + 2, evals);
        if (n_loading) atomicAdd(A.counters + 1, n_loading);
    }
}

template <int DIM, int KW>
cudaError_t launch_kw(const AsmArgs &a, int num_sms, const AsmTune &t, cudaStream_t s)
{
    const size_t sm = sizeof(float) * (Geo<DIM>::NQ * Geo<DIM>::NEN * 4 + (size_t)scratch_floats<DIM>(a.wmax) * KW);
    int dev = 0, optin = 0;
    cudaError_t e0 = cudaGetDevice(&dev);
    if (e0 == cudaSuccess) e0 = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e0 != cudaSuccess) return e0;
    if (sm > (size_t)optin) return cudaErrorInvalidConfiguration;   // this CTA width does not fit
    cudaError_t err = cudaFuncSetAttribute(asm_fp32_kernel<DIM, KW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    int per_sm = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, asm_fp32_kernel<DIM, KW>, 32 * KW, sm);
    if (err != cudaSuccess) return err;
    if (per_sm < 1) per_sm = 1;
    if (t.cta_per_sm > 0 && t.cta_per_sm < per_sm) per_sm = t.cta_per_sm;
    using G_ = Geo<DIM>;
    int64_t batches = (a.n_elems + G_::EPW - 1) / G_::EPW;
    int64_t need = (batches + KW - 1) / KW;
    int64_t grid = (int64_t)num_sms * per_sm;
    if (grid > need) grid = need;
    if (t.grid_max > 0 && grid > t.grid_max) grid = t.grid_max;
    if (grid < 1) grid = 1;
    asm_fp32_kernel<DIM, KW><<<(unsigned)grid, 32 * KW, sm, s>>>(a);
    return cudaGetLastError();
}

// the requested CTA width, or the widest narrower one whose shared memory fits (a
// width tuned for one kernel may not fit another: the FP64 kernel needs twice the
// FP32 kernel's scratch)
template <int DIM>
cudaError_t launch_dim(const AsmArgs &a, int num_sms, const AsmTune &t, cudaStream_t s)
{
    if (t.exact) {
        switch (t.warps) {
        case 1: return launch_kw<DIM, 1>(a, num_sms, t, s);
        case 2: return launch_kw<DIM, 2>(a, num_sms, t, s);
        case 8: return launch_kw<DIM, 8>(a, num_sms, t, s);
        default: return launch_kw<DIM, 4>(a, num_sms, t, s);
        }
    }
    cudaError_t e = cudaErrorInvalidConfiguration;
    if (t.warps >= 8) e = launch_kw<DIM, 8>(a, num_sms, t, s);
    if (e == cudaErrorInvalidConfiguration && t.warps >= 4) e = launch_kw<DIM, 4>(a, num_sms, t, s);
    if (e == cudaErrorInvalidConfiguration && t.warps >= 2) e = launch_kw<DIM, 2>(a, num_sms, t, s);
    if (e == cudaErrorInvalidConfiguration) e = launch_kw<DIM, 1>(a, num_sms, t, s);
    return e;
}

}  // namespace

cudaError_t launch_assemble_fp32(int dim, const AsmArgs &a, int num_sms, cudaStream_t s, const AsmTune &t)
{
    if (a.n_elems <= 0) return cudaSuccess;
    return dim == 2 ? launch_dim<2>(a, num_sms, t, s) : launch_dim<3>(a, num_sms, t, s);
}

}  // namespace gd
