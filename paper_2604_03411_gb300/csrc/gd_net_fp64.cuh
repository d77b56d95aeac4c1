// gd_net_fp64.cuh -- the ICNNs of the FP64 element kernel, eight lanes per quadrature
// point (four points of a warp at once): lane sub = lane mod 8 of point pt = lane / 8 owns
// the units j, k = sub (mod 8) of every layer.  (Four lanes per point halve the reductions
// but double a round's buffers and accumulators: 8 instead of 16 warps per SM.)  Pre-activations and the sums over the second
// layer's units are FP64; activations and the layer products are 64-bit fixed point
// (gd_fixed.cuh).  The FP32 evaluations of the local solve use the same mapping.
// Every function is called by the whole warp; `need` marks the points that take part (all
// lanes of a point agree) and net is the same for all of them.  Points whose fixed-point sums
// would be less accurate than FP64 (Trust) are evaluated again; those for which that does not
// help, whose argument is not finite (far past the root of the local solve f_d underflows and q
// is infinite) or whose weights are not take the FP64 functions of gd_device_fp64.cuh, one after
// the other with a lane per unit.
#pragma once

#include "gd_internal.cuh"

namespace gd {
namespace {
#include "gd_device_fp64.cuh"
}
}  // namespace gd

#include "gd_elem32.cuh"
#include "gd_fixed.cuh"

namespace gd {
namespace grp {

using fx::i64;

constexpr int kLanes = 8;                  // lanes per point
constexpr int kPts = 32 / kLanes;          // points per round
constexpr int kOut = 16 / kLanes;          // a lane's outputs of a 16-wide chunk

// shared-memory bytes of a warp's network buffers for width w: operands [w][kPts][4], one
// 64-bit word [w][kPts] per unit, reverse operands [w][kPts]
__host__ __device__ constexpr size_t buf_bytes(int w) { return (size_t)w * kPts * (4 + 1 + 1) * 8; }

template <class T>
__device__ __forceinline__ T sum_lanes(T v)
{
#pragma unroll
    for (int o = 1; o < kLanes; o *= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ int max_lanes(int v)
{
#pragma unroll
    for (int o = 1; o < kLanes; o *= 2) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ int hi_word(double v) { return __double2hiint(v); }

// bit p: a lane of the warp's point p has `take`
__device__ __forceinline__ unsigned points_of(bool take)
{
    const unsigned b = __ballot_sync(0xffffffffu, take);
    return ((b & 0xffu) != 0) | ((b & 0xff00u) != 0) << 1 | ((b & 0xff0000u) != 0) << 2 | ((b >> 24) != 0) << 3;
}
static_assert(kLanes == 8, "points_of");

// NC column products of a 16-wide output chunk: V[i][c] = sum_j W(k_i, j) z_c(j) in units of
// 2^-56 (times the operand and row scales), k_i = c0 + 8 i + sub.  Three multiply-adds per
// term: hi hi into one sum, hi lo + lo hi into the other.  z: operand c of unit j and point pt
// at z[(j kPts + pt) ZS + c].
template <int NC, int ZS>
__device__ __forceinline__ void chunk_product(const int2 *__restrict__ W, int wp, int c0, const int2 *z, int n, int pt,
                                              int sub, i64 (&V)[kOut][NC])
{
    i64 hh[kOut][NC], md[kOut][NC];
#pragma unroll
    for (int i = 0; i < kOut; ++i)
#pragma unroll
        for (int c = 0; c < NC; ++c) hh[i][c] = md[i][c] = 0;
    const int4 *wr = reinterpret_cast<const int4 *>(W + c0 + sub * kOut);
    const int2 *zr = z + pt * ZS;
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
        const int4 wa = __ldg(wr);
        wr += wp / 2;
        const int wh[kOut] = {wa.x, wa.z}, wl[kOut] = {wa.y, wa.w};
        int zh[NC], zl[NC];
        if (NC == 4) {
            const int4 a = reinterpret_cast<const int4 *>(zr)[0], b = reinterpret_cast<const int4 *>(zr)[1];
            zh[0] = a.x; zl[0] = a.y;
            if (NC > 1) { zh[1 % NC] = a.z; zl[1 % NC] = a.w; }
            if (NC > 2) { zh[2 % NC] = b.x; zl[2 % NC] = b.y; zh[3 % NC] = b.z; zl[3 % NC] = b.w; }
        } else if (NC == 2) {
            const int4 a = reinterpret_cast<const int4 *>(zr)[0];
            zh[0] = a.x; zl[0] = a.y;
            zh[1 % NC] = a.z; zl[1 % NC] = a.w;
        } else {
            const int2 a = zr[0];
            zh[0] = a.x; zl[0] = a.y;
        }
        zr += kPts * ZS;
#pragma unroll
        for (int i = 0; i < kOut; ++i)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                hh[i][c] += (i64)zh[c] * wh[i];
                md[i][c] += (i64)zh[c] * wl[i];
                md[i][c] += (i64)zl[c] * wh[i];
            }
    }
#pragma unroll
    for (int i = 0; i < kOut; ++i)
#pragma unroll
        for (int c = 0; c < NC; ++c) V[i][c] = hh[i][c] + ((md[i][c] + (1LL << 27)) >> fx::kLimb);
}

// How far a point's fixed-point sums can be trusted.  A layer product is off by about 0.4 sqrt(2 w)
// units of its scale (2^-56 of the row's bound times the operands' bound): the roundings of both
// operands, at random.  k stands for log2(sqrt(w) / 2).  A point whose estimated errors are above
// what FP64 sums would leave is evaluated again: without TAIL with it, and then by the FP64
// functions.  Networks whose weights or activations of very different size meet the wrong way
// round (the largest activations on the smallest weights) come to that; of 1,000 networks
// with weights |N(0, 0.1)| and biases N(0, 0.1) at each of eight widths from 1 to 64, none did.
struct Trust {
    int k;
    bool poor;
    __device__ __forceinline__ explicit Trust(int w) : k(w >= 64 ? 2 : w >= 16 ? 1 : w >= 4 ? 0 : -1), poor(false) {}
    // pre-activations of scale 2^e: 2^-53 max(1, sum) each, as in an FP64 sum of these terms
    bool wide = false;
    int least = 0;
    __device__ __forceinline__ void scale(int e)
    {
        wide = e + k > 3;
        least = 1 << (21 + k);
    }
    __device__ __forceinline__ void sum(i64 V) { poor |= wide && (int)(V >> 32) < least; }
    // an output sum v with errors near 2^(e - 56): not above 2^(slack - 56) of v (by its exponent)
    __device__ __forceinline__ void output(double v, int e, int slack)
    {
        poor |= e > max(fx::biased_exponent(v), 23) - 1023 + slack;
    }
};
constexpr int kWidest = 60;    // operand scale past which a point goes to the FP64 functions

// Energy network N(y) with gradient and (hess) Hessian in sym6 order, for the points with
// need: y at sY[pt 4 ..], results to sO[pt 10 ..].  Returns the points (bits) whose results cannot
// be trusted.  N(y) is the same to the last bit wherever this is compiled in (explicit fma in
// its sum): the normalising constants rely on it, as they do for both forms of yield.  Same
// identities as psi_net_unit:
//   d2N/dy2 = sum_k w3_k sp''(h2_k) g_k g_k^T + sum_j v_j sp''(h1_j) W1_j W1_j^T,
//   v = W2^T (w3 o sp'(h2)).
// TAIL: operand scales also below 1 and the activations' tails.
template <bool TAIL>
__device__ __forceinline__ unsigned energy_fixed(const double *p, const unsigned char *fxp, int w, const double *sY,
                                                 double *sO, unsigned char *buf, int lane, bool need, bool hess)
{
    const int wp = fx::pad16(w), pt = lane / kLanes, sub = lane % kLanes;
    const double *W1 = p, *b1 = W1 + 3 * w, *A2 = b1 + w + w * w, *b2 = A2 + 3 * w, *w3 = b2 + w, *a3 = w3 + w;
    const fx::Net fn = fx::net_of(fxp, w);
    int2 *z = reinterpret_cast<int2 *>(buf);                        // [w][kPts][4]
    i64 *sE = reinterpret_cast<i64 *>(z + w * kPts * 4);            // [w][kPts]: h1, then sp''(h1) in units of 2^(es - 62)
    int2 *su = reinterpret_cast<int2 *>(sE + w * kPts);             // [w][kPts]: w3 sp'(h2)
    double y0 = sY[pt * 4], y1 = sY[pt * 4 + 1], y2 = sY[pt * 4 + 2];
    Trust tr(w);
    tr.poor = !(isfinite(y0) && isfinite(y1) && isfinite(y2));
    if (tr.poor || !need) y0 = y1 = y2 = 0.0;
    // layer 1: pre-activations and the point's operand scale
    int hm = TAIL ? (int)0x80000000 : 0;
    uint32_t low = 0;
    for (int j = sub; j < w; j += kLanes) {
        const double h =
            fma(__ldg(W1 + 3 * j + 2), y2, fma(__ldg(W1 + 3 * j + 1), y1, fma(__ldg(W1 + 3 * j), y0, __ldg(b1 + j))));
        sE[j * kPts + pt] = __double_as_longlong(h);
        hm = max(hm, TAIL ? fx::order_key(hi_word(h)) : hi_word(h));
        low = max(low, (uint32_t)hi_word(h));
    }
    hm = max_lanes(hm);
    const int ep = TAIL ? fx::softplus_exp_tail(hm) : fx::softplus_exp(hm), es = TAIL ? min(ep, 0) : 0;
    tr.poor |= ep > kWidest;
    const int *e1 = fn.e + 3 * w, e10 = __ldg(e1), e11 = __ldg(e1 + 1), e12 = __ldg(e1 + 2);
    for (int j = sub; j < w; j += kLanes) {
        const double h = __longlong_as_double(sE[j * kPts + pt]);
        const fx::Act r = fx::activation<TAIL>(h);
        const i64 *w1 = fn.W1 + 4 * j, g = fx::sigmoid_factor<TAIL>(r, es);
        const int2 l0 = fx::limbs(fx::softplus_operand(h, r, ep));
        const int2 l1 = fx::limbs((fx::mulhi_s(g, __ldg(w1)) + 8) >> 4);
        const int2 l2 = fx::limbs((fx::mulhi_s(g, __ldg(w1 + 1)) + 8) >> 4);
        const int2 l3 = fx::limbs((fx::mulhi_s(g, __ldg(w1 + 2)) + 8) >> 4);
        int4 *zz = reinterpret_cast<int4 *>(z + (j * kPts + pt) * 4);
        zz[0] = make_int4(l0.x, l0.y, l1.x, l1.y);
        zz[1] = make_int4(l2.x, l2.y, l3.x, l3.y);
        sE[j * kPts + pt] = fx::mulhi_s(g, r.c) << 2;
    }
    __syncwarp();
    double acc[10];
#pragma unroll
    for (int c = 0; c < 10; ++c) acc[c] = 0.0;
    const int rows = __ldg(e1 + fx::kRows), cols = __ldg(e1 + fx::kCols);
    int eu = __ldg(e1 + fx::kOuts);                  // w3 sp'(h2) < 2^eu
    tr.scale(rows + ep);
    int um = 0;
    for (int c0 = 0; c0 < wp; c0 += 16) {
        i64 V[kOut][4];
        chunk_product<4, 4>(fn.W2, wp, c0, z, w, pt, sub, V);
#pragma unroll
        for (int i = 0; i < kOut; ++i) {
            const int k = c0 + kLanes * i + sub;
            if (k < w) {
                const int er = __ldg(fn.e + k) - fx::kBits, eg = er + es, ew3 = __ldg(fn.e + 2 * w + k);
                const double q0 = __ldg(A2 + 3 * k), q1 = __ldg(A2 + 3 * k + 1), q2 = __ldg(A2 + 3 * k + 2);
                tr.sum(V[i][0]);
                const double h =
                    fx::to_double(V[i][0], er + ep) + fma(q2, y2, fma(q1, y1, fma(q0, y0, __ldg(b2 + k))));
                const double g0 = fx::to_double(V[i][1], eg + e10) + q0, g1 = fx::to_double(V[i][2], eg + e11) + q1,
                             g2 = fx::to_double(V[i][3], eg + e12) + q2;
                low = max(low, (uint32_t)hi_word(h));
                const fx::Act r = fx::activation<TAIL>(h);
                const i64 uq = fx::mulhi_s(__ldg(fn.w3 + k), r.g);            // units of 2^(ew3 - 60 - n)
                const double u = fx::to_double(uq, ew3 - 60 - r.n);
                acc[0] = fma(__ldg(w3 + k), fx::softplus_value(h, r), acc[0]);
                acc[1] += u * g0;
                acc[2] += u * g1;
                acc[3] += u * g2;
                if (hess) {
                    const double e2 = fx::to_double(fx::mulhi_s(uq, r.c), ew3 - 58 - r.n);
                    const double e0 = e2 * g0, e1g = e2 * g1;
                    acc[4] += e0 * g0;
                    acc[5] += e0 * g1;
                    acc[6] += e0 * g2;
                    acc[7] += e1g * g1;
                    acc[8] += e1g * g2;
                    acc[9] += e2 * g2 * g2;
                    if (TAIL) {
                        reinterpret_cast<double *>(su)[k * kPts + pt] = u;
                        um = max(um, fx::biased_exponent(u));
                    } else {
                        su[k * kPts + pt] = fx::limbs(fx::shift_round(uq, 4 + eu - ew3));
                    }
                }
            }
        }
    }
    if (!TAIL) tr.poor |= low >= fx::kTailHigh;
    if (hess) {
        if (TAIL) {
            // the reverse operands at the scale of the point's largest
            eu = max_lanes(um) - 1022;
            for (int k = sub; k < w; k += kLanes)
                su[k * kPts + pt] = fx::limbs(fx::from_double(reinterpret_cast<double *>(su)[k * kPts + pt], fx::kBits - eu));
        }
        __syncwarp();
        for (int c0 = 0; c0 < wp; c0 += 16) {
            i64 V[kOut][1];
            chunk_product<1, 1>(fn.W2T, wp, c0, su, w, pt, sub, V);
#pragma unroll
            for (int i = 0; i < kOut; ++i) {
                const int j = c0 + kLanes * i + sub;
                if (j < w) {
                    const double c =
                        fx::to_double(fx::mulhi_s(V[i][0], sE[j * kPts + pt]), __ldg(fn.e + w + j) + eu + es - 54);
                    const double *ww = fn.WW + 6 * j;
#pragma unroll
                    for (int m = 0; m < 6; ++m) acc[4 + m] += c * __ldg(ww + m);
                }
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 10; ++c)
        if (c < 4 || hess) acc[c] = sum_lanes(acc[c]);
    double *o = sO + pt * 10;
    if (sub == 0 && need) {
#pragma unroll
        for (int c = 0; c < 10; ++c) o[c] = c < 4 || hess ? acc[c] : 0.0;
    }
    __syncwarp();
    // Errors of the sums over the units, lane sub for entry (a, b) of the Hessian and component b of
    // the gradient, relative: 2^-51 of the gradient (2^2k units' roundings add up at random); of
    // the Hessian's first part, sum u (1 - sp') g_a g_b, at most the gradient's times the other
    // factor's error, 2^-52.8; of its second, 2^-51.  (One lane per entry: written out for every
    // lane the tests are 2 KB of code.)
    if (need && sub < 6) {
        const int a = sub < 3 ? 0 : (sub < 5 ? 1 : 2), b = sub < 3 ? sub : (sub < 5 ? sub - 2 : 2);
        const int ea = __ldg(e1 + a) + es, eb = __ldg(e1 + b) + es;
        tr.output(o[1 + b], eu + rows + eb + 2 * tr.k, 5);
        if (hess) {
            const double H = o[4 + sub];
            tr.output(H, fx::biased_exponent(o[1 + a]) - 1023 + rows + eb, 5);
            tr.output(H, fx::biased_exponent(o[1 + b]) - 1023 + rows + ea, 5);
            tr.output(H, eu + cols - 2 + ea + eb - es + 2 * tr.k, 6);
        }
    }
    __syncwarp();
    if (need && sub < 4) o[sub] += sub ? __ldg(a3 + sub - 1) : __ldg(a3) * y0 + __ldg(a3 + 1) * y1 + __ldg(a3 + 2) * y2;
    __syncwarp();
    return points_of(need && tr.poor);
}
// The points in `mask` with the tails, and what still cannot be trusted (fp64: all of them) by the
// FP64 functions, a warp per point.  Out of line: few points come here.
static __device__ __noinline__ void energy_rare(const double *p, double *W2T, const unsigned char *fxp, int w,
                                                const double *sY, double *sO, unsigned char *buf, int lane,
                                                unsigned mask, bool hess, bool fp64)
{
    if (!fp64) mask = energy_fixed<true>(p, fxp, w, sY, sO, buf, lane, (mask >> lane / kLanes & 1u) != 0, hess);
    DevNet net;
    net.p = const_cast<double *>(p);
    net.W2T = W2T;
    net.width = w;
    for (int pt = 0; pt < kPts; ++pt) {
        if (!(mask >> pt & 1u)) continue;
        double o[10];
        psi_net_unit(net, sY + pt * 4, o, reinterpret_cast<double *>(buf), lane, hess);
        if (lane == 0)
#pragma unroll
            for (int c = 0; c < 10; ++c) sO[pt * 10 + c] = c < 4 || hess ? o[c] : 0.0;
    }
    __syncwarp();
}
// how a network's points start; read by the callers well before it is needed
__device__ __forceinline__ int path_of(const DevNet &net)
{
    return net.width > 0 ? __ldg(fx::net_of(net.fx, net.width).e + 3 * net.width + fx::kPath) : 0;
}
__device__ __forceinline__ void energy(const DevNet &net, int path, const double *sY, double *sO, unsigned char *buf,
                                       int lane, bool need, bool hess)
{
    const unsigned mask = path == fx::kPlain
                              ? energy_fixed<false>(net.p, net.fx, net.width, sY, sO, buf, lane, need, hess)
                              : points_of(need);
    if (mask) energy_rare(net.p, net.W2T, net.fx, net.width, sY, sO, buf, lane, mask, hess, path == fx::kFp64);
}

// Yield network N_k(q) (r.x) and, with SLOPE, N_k'(q) (r.y) of a network of width w > 0; returns the
// points whose results cannot be trusted.  Every lane of a point gets the same values.
template <bool SLOPE, bool TAIL>
__device__ __forceinline__ unsigned yield_fixed(const double *p, const unsigned char *fxp, int w, double q,
                                                unsigned char *buf, int lane, bool need, double2 &r)
{
    constexpr int NC = SLOPE ? 2 : 1;
    const int wp = fx::pad16(w), pt = lane / kLanes, sub = lane % kLanes;
    const double *V1 = p, *c1 = V1 + w, *B2 = c1 + w + w * w, *c2 = B2 + w, *v3 = c2 + w, *b3 = v3 + w;
    const fx::Net fn = fx::net_of(fxp, w);
    int2 *z = reinterpret_cast<int2 *>(buf);                       // [w][kPts][NC]
    double *sE = reinterpret_cast<double *>(z + w * kPts * NC);    // [w][kPts]: h1
    Trust tr(w);
    tr.poor = !isfinite(q);
    if (!need || tr.poor) q = 0.0;
    int hm = TAIL ? (int)0x80000000 : 0;
    uint32_t low = 0;
    for (int j = sub; j < w; j += kLanes) {
        const double h = fma(__ldg(V1 + j), q, __ldg(c1 + j));
        sE[j * kPts + pt] = h;
        hm = max(hm, TAIL ? fx::order_key(hi_word(h)) : hi_word(h));
        low = max(low, (uint32_t)hi_word(h));
    }
    hm = max_lanes(hm);
    const int ep = TAIL ? fx::softplus_exp_tail(hm) : fx::softplus_exp(hm), es = TAIL ? min(ep, 0) : 0;
    tr.poor |= ep > kWidest;
    const int *e1 = fn.e + 3 * w, ew1 = __ldg(e1) + es, rows = __ldg(e1 + fx::kRows);
    for (int j = sub; j < w; j += kLanes) {
        const double h = sE[j * kPts + pt];
        const fx::Act r1 = fx::activation<TAIL>(h);
        int2 *zz = z + (j * kPts + pt) * NC;
        zz[0] = fx::limbs(fx::softplus_operand(h, r1, ep));
        if (SLOPE)
            zz[NC - 1] = fx::limbs((fx::mulhi_s(fx::sigmoid_factor<TAIL>(r1, es), __ldg(fn.W1 + 4 * j)) + 8) >> 4);
    }
    __syncwarp();
    double n0 = 0.0, n1 = 0.0;
    int um = 0;
    tr.scale(rows + ep);
    for (int c0 = 0; c0 < wp; c0 += 16) {
        i64 V[kOut][NC];
        chunk_product<NC, NC>(fn.W2, wp, c0, z, w, pt, sub, V);
#pragma unroll
        for (int i = 0; i < kOut; ++i) {
            const int k = c0 + kLanes * i + sub;
            if (k < w) {
                const int er = __ldg(fn.e + k) - fx::kBits;
                const double b = __ldg(B2 + k);
                tr.sum(V[i][0]);
                const double h = fx::to_double(V[i][0], er + ep) + fma(b, q, __ldg(c2 + k));
                low = max(low, (uint32_t)hi_word(h));
                const fx::Act r2 = fx::activation<TAIL>(h);
                n0 = fma(__ldg(v3 + k), fx::softplus_value(h, r2), n0);
                if (SLOPE) {
                    const double u =
                        fx::to_double(fx::mulhi_s(__ldg(fn.w3 + k), r2.g), __ldg(fn.e + 2 * w + k) - 60 - r2.n);
                    n1 += u * (fx::to_double(V[i][NC - 1], er + ew1) + b);
                    if (TAIL) um = max(um, fx::biased_exponent(u));
                }
            }
        }
    }
    if (!TAIL) tr.poor |= low >= fx::kTailHigh;
    const double b = __ldg(b3);
    r = make_double2(sum_lanes(n0) + b * q, 0.0);
    if (SLOPE) {
        n1 = sum_lanes(n1);
        tr.output(n1, (TAIL ? max_lanes(um) - 1022 : __ldg(e1 + fx::kOuts)) + rows + ew1 + 2 * tr.k, 5);
        r.y = n1 + b;
    }
    __syncwarp();
    return points_of(need && tr.poor);
}
static __device__ __noinline__ double2 yield_rare(const double *p, double *W2T, const unsigned char *fxp, int w,
                                                  double q, double2 r, unsigned char *buf, int lane, unsigned mask,
                                                  bool fp64)
{
    const int pt_me = lane / kLanes;
    if (!fp64) {
        double2 t;
        const bool mine = mask >> pt_me & 1u;
        mask = yield_fixed<true, true>(p, fxp, w, q, buf, lane, mine, t);
        if (mine) r = t;
    }
    DevNet net;
    net.p = const_cast<double *>(p);
    net.W2T = W2T;
    net.width = w;
    NetConst unit;
    unit.y_N0 = 0.0;
    unit.y_s = 1.0;
    for (int pt = 0; pt < kPts; ++pt) {
        if (!(mask >> pt & 1u)) continue;
        double N, Np;
        yield_unit(net, unit, __shfl_sync(0xffffffffu, q, pt * kLanes), N, Np, reinterpret_cast<double *>(buf), lane);
        if (pt_me == pt) r = make_double2(N, Np);
    }
    return r;
}
template <bool SLOPE>
static __device__ __noinline__ double2 yield(const double *p, double *W2T, const unsigned char *fxp, int w, int path,
                                             double q, unsigned char *buf, int lane, bool need)
{
    double2 r = make_double2(0.0, 0.0);
    const unsigned mask =
        path == fx::kPlain ? yield_fixed<SLOPE, false>(p, fxp, w, q, buf, lane, need, r) : points_of(need);
    if (mask) r = yield_rare(p, W2T, fxp, w, q, r, buf, lane, mask, path == fx::kFp64);
    return r;
}

// r(kappa) = G(q(kappa)) - kappa (Eq. (potential_function)), q = psi_e + qcoef (phi - kappa) /
// f_d(kappa) (Eq. (ostwald_potential)); SLOPE: dr/dkappa and G' too
template <bool SLOPE>
__device__ __forceinline__ void residual(const MatConst &m, const DevNet &yld, int path, const NetConst &nc, double pe,
                                         double phi, double kappa, double &r, double &dr, double &Gp,
                                         unsigned char *buf, int lane, bool need)
{
    const bool dmg = kappa > m.kappa_d;
    const double f = dmg ? fx::exp_neg(m.eta_d * (kappa - m.kappa_d)) : 1.0;
    const double q = pe + m.qcoef * (phi - kappa) / f;
    // G(q) = s (N_k(q) - N_k(0)) (Eq. (Gq_NN)); width 0 is the identity G(q) = q
    double G = q, Gs = 1.0;
    if (yld.width > 0) {
        const double2 n = yield<SLOPE>(yld.p, yld.W2T, yld.fx, yld.width, path, q, buf, lane, need);
        G = nc.y_s * (n.x - nc.y_N0);
        Gs = nc.y_s * n.y;
    }
    r = G - kappa;
    if (SLOPE) {
        Gp = Gs;
        dr = Gs * (m.qcoef * ((dmg ? (phi - kappa) * m.eta_d - 1.0 : -1.0) / f)) - 1.0;
    }
}

// Softplus and sigmoid for the FP32 part of the local solve, with relative errors of a few 1e-7 plus
// those of __expf (1.2 |v| units in the last place).  The trial decision rests on G = (N_k(q) -
// N_k(0)) / N_k'(0), which amplifies an absolute error wherever the units are in the flat part of
// softplus: the logarithm of the rounded 1 + e moved G by 4e-3 with biases of -10.  log1p(e) / e for
// 0 <= e <= 1 is a minimax polynomial (Lawson's iteration on the Chebyshev basis, 1.9e-7).
// (A pass over the notched plate, 159,744 points: expf, log1pf and a division 5 % more, expf and one
// more term here 1.5 %.)
__device__ __forceinline__ void sp_sig_start(float v, float &sp, float &sg)
{
    const float e = __expf(-fabsf(v)), r = __fdividef(1.0f, 1.0f + e);
    float p = -0.0085391989f;
    p = fmaf(p, e, 0.0440895967f);
    p = fmaf(p, e, -0.107681662f);
    p = fmaf(p, e, 0.177452385f);
    p = fmaf(p, e, -0.244954616f);
    p = fmaf(p, e, 0.332754791f);
    p = fmaf(p, e, -0.499974042f);
    p = fmaf(p, e, 0.999999821f);
    sp = fmaxf(v, 0.0f) + e * p;
    sg = v >= 0.0f ? r : e * r;
}

// N_k(q) and N_k'(q) in FP32
static __device__ __noinline__ float2 yield32(const float *p, const unsigned char *fxp, int w, float q,
                                              unsigned char *buf, int lane)
{
    const int wp = fx::pad16(w), pt = lane / kLanes, sub = lane % kLanes;
    const float *V1 = p, *c1 = V1 + w, *B2 = c1 + w + w * w, *c2 = B2 + w, *v3 = c2 + w, *b3 = v3 + w;
    const float2 *W2P = reinterpret_cast<const float2 *>(fx::net_of(fxp, w).W2P);
    float2 *z = reinterpret_cast<float2 *>(buf);                   // [w][kPts]
    for (int j = sub; j < w; j += kLanes) {
        const float a = __ldg(V1 + j);
        float s, g;
        sp_sig_start(__ldg(c1 + j) + a * q, s, g);
        z[j * kPts + pt] = make_float2(s, g * a);
    }
    __syncwarp();
    float n0 = 0.0f, n1 = 0.0f;
    for (int c0 = 0; c0 < wp; c0 += 16) {
        float h[kOut] = {0.0f, 0.0f}, t[kOut] = {0.0f, 0.0f};
        const float2 *wr = W2P + c0 / 2 + sub;
#pragma unroll 8
        for (int j = 0; j < w; ++j) {
            const float2 a = __ldg(wr + j * (wp / 2));
            const float2 v = z[j * kPts + pt];
            h[0] += a.x * v.x; t[0] += a.x * v.y;
            h[1] += a.y * v.x; t[1] += a.y * v.y;
        }
#pragma unroll
        for (int i = 0; i < kOut; ++i) {
            const int k = c0 + kLanes * i + sub;
            if (k < w) {
                const float b = __ldg(B2 + k), vk = __ldg(v3 + k);
                float s, g;
                sp_sig_start(h[i] + __ldg(c2 + k) + b * q, s, g);
                n0 += vk * s;
                n1 += vk * g * (t[i] + b);
            }
        }
    }
    const float b = __ldg(b3);
    const float2 r = make_float2(sum_lanes(n0) + b * q, sum_lanes(n1) + b);
    __syncwarp();
    return r;
}

// r and dr/dkappa in FP32; scale: what the rounding of r is relative to (the network's constant
// and the two terms of q)
__device__ __forceinline__ void residual32(const e32::MatF &m, const DevNet &yld, const e32::NcF &nc, float pe,
                                           float phi, float kappa, float &r, float &dr, float &Gp, float &scale,
                                           unsigned char *buf, int lane)
{
    const bool dmg = kappa > m.kappa_d;
    const float f = dmg ? expf(-m.eta_d * (kappa - m.kappa_d)) : 1.0f;
    const float qp = m.qcoef * (phi - kappa) / f, q = pe + qp;
    const float dq = m.qcoef * (-1.0f / f + (dmg ? (phi - kappa) * m.eta_d / f : 0.0f));
    float G = q;
    Gp = 1.0f;
    if (yld.width > 0) {
        const float2 n = yield32(yld.pf, yld.fx, yld.width, q, buf, lane);
        G = nc.y_s * (n.x - nc.y_N0);
        Gp = nc.y_s * n.y;
    }
    r = G - kappa;
    dr = Gp * dq - 1.0f;
    scale = fabsf(nc.y_s * nc.y_N0) + fabsf(Gp) * (fabsf(pe) + fabsf(qp)) + fabsf(kappa);
}

}  // namespace grp
}  // namespace gd
