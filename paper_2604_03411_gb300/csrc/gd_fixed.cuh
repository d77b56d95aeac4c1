// gd_fixed.cuh -- 64-bit fixed-point arithmetic for the ICNNs of the FP64 element kernel.
//
// sm_103a issues FP64 at 1.7 lanes per clock and SM but 32-bit integer multiply-adds
// (32 x 32 + 64 -> 64) at 62 (both measured with independent chains, 4-16 warps per SM).
// The networks' layers are sums of bounded terms, so they are evaluated in fixed point:
//  - softplus and sigmoid of an FP64 argument come from integer polynomials on two
//    256-entry tables, with relative errors below 2^-51 down to arguments of -3.47 and, in a
//    second form with a power of two for each value, below that (exp and log1p in FP64: 43
//    FP64 operations per unit, here about 175 integer instructions: 3 clocks instead of 25
//    per unit and SM);
//  - a layer's product sum_j W_kj z_j runs on 56-bit operands split into two 28-bit limbs,
//    three multiply-adds per term (lo x lo, 2^-58 of the scale at most, is left out) with exact
//    64-bit accumulation.  Its scale is the power of two above the row's largest weight times
//    the one above the point's largest operand, and its error a few 2^-56 of that, whatever the
//    sum is.  Where the largest terms meet that is below the rounding of the FP64 sum; where a
//    row's large weights meet the small operands it is not.  Every point's sums are checked
//    (gd_net_fp64.cuh, Trust), and a point that would lose accuracy is evaluated again, with the
//    second form and scales of its own and, where that does not help, by the FP64 functions.
// Compiles for the host as well (the tables are constant expressions).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace gd {
namespace fx {

using i64 = long long;
using u64 = unsigned long long;
#define GD_FX __host__ __device__ __forceinline__

constexpr i64 kOne62 = 1LL << 62;
constexpr int kBits = 56;                 // operand bits of the layer products
constexpr int kLimb = 28;

GD_FX u64 mulhi_u(u64 a, u64 b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (u64)(((unsigned __int128)a * b) >> 64);
#endif
}
GD_FX i64 mulhi_s(i64 a, i64 b)
{
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (i64)(((__int128)a * b) >> 64);
#endif
}
GD_FX int mulhi_s32(int a, int b) { return (int)(((i64)a * b) >> 32); }
GD_FX uint32_t mulhi_u32(uint32_t a, uint32_t b) { return (uint32_t)(((u64)a * b) >> 32); }
GD_FX u64 bits_of(double v)
{
#ifdef __CUDA_ARCH__
    return (u64)__double_as_longlong(v);
#else
    u64 b;
    __builtin_memcpy(&b, &v, 8);
    return b;
#endif
}
GD_FX double of_bits(u64 b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((i64)b);
#else
    double v;
    __builtin_memcpy(&v, &b, 8);
    return v;
#endif
}
GD_FX int clz64(u64 a)
{
#ifdef __CUDA_ARCH__
    return __clzll((i64)a);
#else
    return a ? __builtin_clzll(a) : 64;
#endif
}

// Tables, computed in 110-bit integer arithmetic: e[i] = 2^64 2^(-i/256) (e[0] = 2^64 - 1),
// n[i] = 2^16 / (1 + (i + 1/2) / 256) rounded to an integer, l[i] = 2^62 ln(2^16 / n[i]).
struct Tables {
    u64 e[256];
    u64 l[256];
    uint32_t n[256];
};
using u128 = unsigned __int128;
constexpr u128 mul_q110(u128 a, u128 b)   // (a b) >> 110 for operands below 2^111
{
    const u128 m = ((u128)1 << 55) - 1;
    const u128 ah = a >> 55, al = a & m, bh = b >> 55, bl = b & m;
    return ah * bh + ((ah * bl + al * bh) >> 55) + ((al * bl) >> 110);
}
constexpr Tables make_tables()
{
    Tables t{};
    const u128 one = (u128)1 << 110;
    // ln 2 = 0.B17217F7D1CF79ABC9E3B39803F2F6AF (hexadecimal)
    const u128 ln2 = (((u128)0xB17217F7D1CF79ABull << 64) | 0xC9E3B39803F2F6AFull) >> 18;
    const u128 x = ln2 >> 8;
    u128 q = one, term = one;              // q = exp(-ln2 / 256)
    for (int n = 1; n < 20; ++n) {
        term = mul_q110(term, x) / n;
        q = (n & 1) ? q - term : q + term;
    }
    u128 v = one;
    for (int i = 0; i < 256; ++i) {
        const u128 r = (v + ((u128)1 << 45)) >> 46;
        t.e[i] = (r >> 64) ? ~0ull : (u64)r;
        v = mul_q110(v, q);
        const uint32_t num = (2u * 65536u * 512u / (513u + 2u * i) + 1u) / 2u;
        t.n[i] = num;
        // ln(65536 / num) = 2 atanh z
        const u128 z = (((u128)(65536u - num)) << 110) / (65536u + num);
        const u128 z2 = mul_q110(z, z);
        u128 p = z, s = 0;
        for (int k = 1; k < 80 && p; k += 2) {
            s += p / k;
            p = mul_q110(p, z2);
        }
        t.l[i] = (u64)((s + ((u128)1 << 46)) >> 47);
    }
    return t;
}
#ifdef __CUDACC__
__device__ const Tables d_tab = make_tables();
#endif
#ifndef __CUDA_ARCH__
constexpr Tables h_tab = make_tables();
#endif
GD_FX u64 tab_e(int i)
{
#ifdef __CUDA_ARCH__
    return __ldg(&d_tab.e[i]);
#else
    return h_tab.e[i];
#endif
}
GD_FX u64 tab_l(int i)
{
#ifdef __CUDA_ARCH__
    return __ldg(&d_tab.l[i]);
#else
    return h_tab.l[i];
#endif
}
GD_FX uint32_t tab_n(int i)
{
#ifdef __CUDA_ARCH__
    return __ldg(&d_tab.n[i]);
#else
    return h_tab.n[i];
#endif
}

// v 2^e rounded to the nearest double (0 below the normal range, infinity above)
GD_FX double to_double(i64 v, int e)
{
    if (v == 0) return 0.0;
    const u64 s = (u64)v & (1ull << 63);
    u64 a = s ? 0ull - (u64)v : (u64)v;
    const int lz = clz64(a);
    a <<= lz;
    const u64 m = (a >> 11) + ((a >> 10) & 1);      // 53 bits; a carry raises the exponent
    int ex = 1023 + 63 - lz + e;
    if (ex <= 0) return 0.0;
    if (ex >= 2046) return of_bits(s | 0x7ff0000000000000ull);
    return of_bits(s | (((u64)(ex - 1) << 52) + m));
}
// z 2^f rounded to an integer (0 for zero and subnormal z); |z| 2^f below 2^62
GD_FX i64 from_double(double z, int f)
{
    const u64 b = bits_of(z), ab = b & 0x7fffffffffffffffull;
    const int sh = (int)(ab >> 52) - 1075 + f;
    const u64 m = (ab & 0xfffffffffffffull) | 0x10000000000000ull;
    i64 x;
    if (ab < (1ull << 52)) x = 0;
    else if (sh >= 0) x = (i64)(m << (sh < 10 ? sh : 10));
    else x = sh < -53 ? 0 : (i64)((m + (1ull << (-sh - 1))) >> -sh);
    return (b >> 63) ? -x : x;
}
// two signed 28-bit limbs: x = hi 2^28 + lo, |lo| <= 2^27
GD_FX int2 limbs(i64 x)
{
    const i64 hi = (x + (1LL << (kLimb - 1))) >> kLimb;
    int2 r;
    r.x = (int)hi;
    r.y = (int)(x - (hi << kLimb));
    return r;
}

// exponent e with |v| < 2^e (0 for v = 0)
GD_FX int bound_exp(double v)
{
    const u64 ab = bits_of(v) & 0x7fffffffffffffffull;
    return ab == 0 ? 0 : (int)(ab >> 52) - 1022;
}

// |h| in units of 2^-57, the largest 64-bit word where |h| >= 128
GD_FX u64 magnitude57(u64 ab)
{
    const int sh = (int)(ab >> 52) - 1023 + 5;
    const u64 m = (ab & 0xfffffffffffffull) | 0x10000000000000ull;
    if (sh > 11) return ~0ull;
    return sh >= 0 ? m << sh : (sh < -53 ? 0 : m >> -sh);
}
// exp(-T 2^-57) = 2^-n e 2^-64; e is returned
GD_FX u64 exp_parts(u64 T, int &n)
{
    const u64 y = mulhi_u(T, 0xB8AA3B295C17F0BCull);               // T log2(e), 56 fraction bits
    n = (int)(y >> 56);
    const u64 rr = (y & 0xffffffffffffull) << 8;                   // r, 64 fraction bits
    const uint32_t rh = (uint32_t)(rr >> 24);                      // r, 40 fraction bits
    // ln2^3/6, ln2^4/24, ln2^5/120 with 36 fraction bits; ln2^2/2, ln2 with 64
    const uint32_t q = 3814213304u - (mulhi_u32(rh, 660952799u - (mulhi_u32(rh, 91627514u) >> 8)) >> 8);
    const u64 a = 4431396893595737425ull - mulhi_u(rr, (u64)q << 28);
    const u64 b = 12786308645202655660ull - mulhi_u(rr, a);
    return mulhi_u(tab_e((int)(y >> 48) & 255), ~mulhi_u(rr, b));
}
// exp(-t) for 0 <= t
GD_FX double exp_neg(double t)
{
    if (!(t < 60.0)) return exp(-t);
    int n;
    const u64 e = exp_parts(magnitude57(bits_of(t)), n);
    return to_double((i64)(e >> 1), -63 - n);
}

// softplus and sigmoid of h:
//   softplus(h) = s 2^es (h < 64; beyond, softplus is h to that precision and the caller takes h),
//   sigmoid(h) = g 2^(-62 - n), 1 - sigmoid(h) = c 2^-62, sp''(h) their product.
// E = exp(-|h|) = 2^-n 2^(-i/256) 2^-r, 2^-r by its Taylor series (r < 2^-8, degree 5);
// log(1 + E) = ln(2^16/n_i) + log1p(r'), 1 + r' = (1 + E) n_i / 2^16, |r'| < 2^-8.9, degree 6, and
// 1 / (1 + E) = (n_i / 2^16) / (1 + r'), geometric series to r'^6: absolute errors of a few 2^-58,
// with which softplus and sigmoid are as accurate as an FP64 evaluation (2^-51) down to
// E = 2^-5, h = -3.4657, and 1 - sigmoid for all positive h.
// TAIL: also below.  log(1 + E) = E (log1p(E) / E) by its own series, sigmoid = E / (1 + E), each with
// a power of two of its own.  (Without it es = -57 and n = 0.)
struct Act {
    i64 s, g, c;
    int es, n;
};
constexpr uint32_t kTailHigh = 0xc00bb9d3u;   // high word of -5 ln 2: the tail's arguments have at least this
template <bool TAIL>
GD_FX Act activation(double h)
{
    const u64 hb = bits_of(h), ab = hb & 0x7fffffffffffffffull;
    const bool neg = (hb >> 63) != 0;
    const u64 T = magnitude57(ab);
    int n;
    const u64 e0 = exp_parts(T, n);
    const u64 e = n > 63 ? 0 : e0 >> n;                            // exp(-|h|), 64 fraction bits
    // logarithm
    const int i = (int)(e >> 56);
    const u64 inv = (u64)tab_n(i) << 48;
    const i64 rs = (i64)(mulhi_u((1ull << 63) | (e >> 1), inv) - (1ull << 63)) << 8;   // r', 71 bits
    const int rx = (int)(rs >> 32);                                // r', 39 bits
    const int L = 715827883 -
                  (mulhi_s32(rx, 536870912 - (mulhi_s32(rx, 429496730 - (mulhi_s32(rx, 357913941) >> 7)) >> 7)) >> 7);
    const i64 x2 = (1LL << 61) - (mulhi_s(rs, (i64)L << 31) >> 7);
    const i64 x1 = kOne62 - (mulhi_s(rs, x2) >> 7);
    const i64 lg = (i64)tab_l(i) + (mulhi_s(rs, x1) >> 7);
    // sigmoid
    const int k1 = 1 << 30;
    const int qs = k1 - (mulhi_s32(rx, k1 - (mulhi_s32(rx, k1 - (rx >> 9)) >> 7)) >> 7);
    const i64 w2 = kOne62 - (mulhi_s(rs, (i64)qs << 32) >> 7);
    const i64 w1 = kOne62 - (mulhi_s(rs, w2) >> 7);
    const i64 w0 = kOne62 - (mulhi_s(rs, w1) >> 7);
    const i64 a = (i64)mulhi_u((u64)w0, inv);
    Act r;
    r.s = (i64)(neg ? 0ull : T) + ((lg + 16) >> 5);
    r.es = -57;
    r.g = neg ? kOne62 - a : a;
    r.c = kOne62 - r.g;
    r.n = 0;
    if (TAIL && neg && e < (1ull << 59)) {
        if (T == ~0ull) {                                          // h <= -128: E itself
            const u64 b = bits_of(exp(h));
            const int ex = (int)(b >> 52);
            r.n = 1022 - (ex ? ex : 1);
            r.s = r.g = (i64)(((b & 0xfffffffffffffull) | (ex ? 0x10000000000000ull : 0)) << 9);
        } else {
            // log1p(E) / E = 1 - E (1/2 - E (1/3 - ...)) to E^10, five levels in 64 bits
            const i64 E66 = (i64)(e << 2);
            const int x = (int)(E66 >> 32);                        // E, 34 bits
            int p = 195225786;                                     // 1/11, 31 bits
            p = 214748365 - (mulhi_s32(x, p) >> 2);
            p = 238609294 - (mulhi_s32(x, p) >> 2);
            p = 268435456 - (mulhi_s32(x, p) >> 2);
            p = 306783378 - (mulhi_s32(x, p) >> 2);
            p = 357913941 - (mulhi_s32(x, p) >> 2);
            i64 v = 922337203685477581LL - (mulhi_s(E66, (i64)p << 31) >> 2);
            v = (1LL << 60) - (mulhi_s(E66, v) >> 2);
            v = 1537228672809129301LL - (mulhi_s(E66, v) >> 2);
            v = (1LL << 61) - (mulhi_s(E66, v) >> 2);
            v = kOne62 - (mulhi_s(E66, v) >> 2);
            r.n = n;
            r.s = (i64)mulhi_u(e0, (u64)v);
            r.g = (i64)mulhi_u(e0, (u64)a);
        }
        r.es = -62 - r.n;
        r.c = a;
    }
    return r;
}

// scale of a point's softplus operands: exponent e_p >= 0 with softplus(h) < 2^e_p for every h
// whose high word is at most hi_max (the largest signed high word of the point's units)
GD_FX int softplus_exp(int hi_max)
{
    const int ex = hi_max <= 0 ? -1023 : (hi_max >> 20) - 1023;
    return ex < -1 ? 0 : (ex == -1 ? 1 : ex + 2);
}
// the same, also below zero, from the largest order_key of the high words; min(e_p, 0) serves the
// sigmoids
GD_FX int order_key(int hi) { return hi ^ ((hi >> 31) & 0x7fffffff); }
GD_FX int softplus_exp_tail(int key)
{
    if (key >= 0) return softplus_exp(key);
    const int ex = (~key >> 20 & 0x7ff) - 1023;
    if (ex < -3) return 0;
    if (ex > 8) return -1100;                     // h <= -512: zeros at this scale
    // softplus(h) < exp(h) = 2^(-|h| log2(e)), |h| rounded down
    const uint32_t fb = (uint32_t)(((key ^ 0x7fffffff) & 0x7fffffff) - (896 << 20)) << 3;
    float v;
#ifdef __CUDA_ARCH__
    v = __uint_as_float(fb);
#else
    __builtin_memcpy(&v, &fb, 4);
#endif
    return (int)floorf(-1.442694f * v) + 1;
}
// x 2^-sh, rounded; |result| < 2^63
GD_FX i64 shift_round(i64 x, int sh)
{
    if (sh <= 0) return (i64)((u64)x << (-sh & 63));
    return sh > 62 ? 0 : (x + (1LL << (sh - 1))) >> sh;
}
// h >= 64
GD_FX bool is_far(double h) { return (int)(bits_of(h) >> 32) >= 0x40500000; }
// softplus as an operand: units of 2^(e_p - 56)
GD_FX i64 softplus_operand(double h, const Act &r, int e_p)
{
    return is_far(h) ? from_double(h, kBits - e_p) : shift_round(r.s, e_p - kBits - r.es);
}
// sigmoid as a factor of operands: units of 2^(e_s - 62)
template <bool TAIL>
GD_FX i64 sigmoid_factor(const Act &r, int e_s)
{
    if (!TAIL) return r.g;
    const int sh = r.n + e_s;
    return sh >= 0 ? r.g >> (sh < 63 ? sh : 63) : (i64)((u64)r.g << (-sh & 63));
}
GD_FX double softplus_value(double h, const Act &r) { return is_far(h) ? h : to_double(r.s, r.es); }

// biased exponent of |v| (0 for zero)
GD_FX int biased_exponent(double v) { return (int)(bits_of(v) >> 52) & 0x7ff; }

// Fixed-point copies of one network (built on the device whenever its weights change).
// Weight tables are stored [j][wp] with the outputs of a 16-wide chunk permuted so that the
// lane sub = k mod 8 of a point finds its two outputs k = c0 + 8 i + sub in 16 consecutive
// bytes.
struct Net {
    const int2 *W2, *W2T;      // [w][wp] limbs: W2[k][j] at (j, perm k), scaled by 2^(56 - e[k]);
                               // transposed: W2[k][j] at (k, perm j), scaled by 2^(56 - e[w + j])
    const float *W2P;          // [w][wp] FP32 W2[k][j] at (j, perm k)
    const i64 *W1;             // [w][4] first-layer weights of input c in units of 2^(e1_c - 62)
    const i64 *w3;             // [w] output weights, each in units of 2^(e3 - 62)
    const double *WW;          // [w][6] products W1_a W1_b (sym6 order; energy network)
    const int *e;              // [w] rows of W2, [w] rows of W2^T, [w] e3, [3] e1, then
                               // kPath, kRows, kCols, kOuts: the largest of each of the three sets
};
enum : int { kPath = 3, kRows = 4, kCols = 5, kOuts = 6, kWords = 8 };      // behind 3 w words
// e[3 w + kPath]: how a network's points start
enum : int {
    kPlain = 0,
    kTails = 1,                // units in the tail of softplus at rest: with the activations' tails
    kFp64 = 2                  // weights that are not finite or beyond 2^kLargest: the FP64 functions
};
constexpr int kZero = -900;    // exponent of a row or column of zeros (its products are exact)
constexpr int kLargest = 150;
GD_FX int pad16(int w) { return (w + 15) / 16 * 16; }
GD_FX int perm16(int k) { return (k & ~15) + (k & 7) * 2 + ((k >> 3) & 1); }
GD_FX size_t net_bytes(int w)
{
    const size_t wp = pad16(w);
    return (size_t)w * wp * 20 + (size_t)w * (32 + 8 + 48) + (size_t)(3 * w + kWords) * 4;
}
GD_FX Net net_of(const unsigned char *base, int w)
{
    const size_t t = (size_t)w * pad16(w);
    Net n;
    n.W2 = reinterpret_cast<const int2 *>(base);
    n.W2T = n.W2 + t;
    n.W2P = reinterpret_cast<const float *>(n.W2T + t);
    n.W1 = reinterpret_cast<const i64 *>(n.W2P + t);
    n.w3 = n.W1 + (size_t)w * 4;
    n.WW = reinterpret_cast<const double *>(n.w3 + w);
    n.e = reinterpret_cast<const int *>(n.WW + (size_t)w * 6);
    return n;
}

}  // namespace fx
}  // namespace gd
