// stage_fp64_body.cuh -- one source x target term of the FP64 stage kernels.
//
// The chip's FP64 pipe takes 2 lanes per cycle and SM, 1/64 of the FP32 and
// integer rate, and the term spelled out in doubles (square root, division,
// sincos, compensated sums) is 54 double instructions (63 for an interface) and
// comparisons of that pipe, which they kept busy: 8 Gpair/s.  Only what decides
// the phase needs 53 bits, since a path is hundreds of radians long: the offset,
// its square, the first estimate g of the distance, its error and k g less whole
// turns, 9 operations.  From there on the numbers are of the order of one and go
// on as integers (the phase, in units of 2^-50 quarter turns) and as pairs of
// floats of 48 bits (sine and cosine from a table, amplitude, products): some 150
// FP32 and integer operations beside the 9, which leave the FP64 pipe the bound.
// The phase is off by 1.6e-15 rad (root mean square) and the rounding of the
// squared distance, a term's amplitude by some 2e-15.  Relative L2 error against
// 128-bit floats, doubles throughout and here, of 200, 1000, 4096 and 8192 sources
// (random frequencies and distances): piston 7.7e-14, 7.3e-14, 5.9e-14, 4.2e-14 and
// 5.0e-14, 5.0e-14, 4.2e-14, 2.9e-14; curved interface 8.7e-15, 1.0e-14, 9.6e-15,
// 6.4e-15 and 8.1e-15, 9.8e-15, 7.3e-15, 5.0e-15; flat interface, whose phases are
// the shortest, 6.9e-15, 5.6e-15, 3.0e-15, 2.5e-15 and 7.5e-15, 5.9e-15, 4.2e-15,
// 3.2e-15.  A chain has the piston's.  Variant 1 of a stage takes every term in
// doubles.
#pragma once
#include "stage.cuh"

namespace rsi_fp64 {

__device__ __forceinline__ float rsqrt_approx(float x) {  // relative error 2^-22.9
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

struct DF {
    float h, l;
};
__device__ __forceinline__ DF df_norm(float h, float l) {  // |l| <= |h|
    const float s = __fadd_rn(h, l);
    return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ DF df_mul(const DF& a, const DF& b) {
    const float p = __fmul_rn(a.h, b.h);
    return df_norm(p, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ DF df_add(const DF& a, const DF& b) {
    const float s = __fadd_rn(a.h, b.h), t = __fsub_rn(s, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
    return df_norm(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ DF df_neg(const DF& a) { return {-a.h, -a.l}; }

// a float as a double by moving bits; normal or 0
__device__ __forceinline__ double widen(float f) {
    const int b = __float_as_int(f);
    return b << 1 ? __hiloint2double(((b & 0x7fffffff) >> 3) + 0x38000000 | (b & 0x80000000), b << 29) : 0.0;
}
// A double as a pair of floats by moving bits (a conversion would be FP64 pipe
// time).  leading_float: the leading 24 bits of the significand, truncated.
// df_of: those rounded to nearest and the signed rest, whose 28 bits a float
// rounds to 24 (2^-50 of the whole).  |d| < 2^127; below 2^-74: 0.
__device__ __forceinline__ float leading_float(int hi, int lo) {
    return __int_as_float(__funnelshift_l(lo, (hi & 0x7fffffff) - 0x38000000, 3));
}
__device__ __forceinline__ DF df_of(double d) {
    const int hi = __double2hiint(d), lo = __double2loint(d), sign = hi & 0x80000000;
    const int top = (hi & 0x7fffffff) - 0x38000000, e = (top >> 20) - 52;  // e: the biased exponent of the last bit
    if (e <= 0) return {0.0f, 0.0f};
    const int rest = int(unsigned(lo) << 3) >> 3, up = rest < 0 ? 1 : 0;
    return {__int_as_float((__funnelshift_l(lo, top, 3) + up) | sign),
            __fmul_rn(float(rest), __int_as_float((e << 23) | sign))};
}

// cos and sin of i / 1024 turns as pairs of floats
constexpr int kTabSize = 1024;
struct TabEntry {
    float ch, cl, sh, sl;
};
struct Tab {
    TabEntry e[kTabSize];
};
constexpr double taylor(double x, bool sine) {  // to x^27 / 27!, |x| <= pi/2
    double term = sine ? x : 1.0, sum = 0.0, small = 0.0;
    for (int n = sine ? 2 : 1; n < 28; n += 2) {
        const double t = sum + term;  // the larger first: Neumaier
        small += (sum > 0 ? sum : -sum) >= (term > 0 ? term : -term) ? (sum - t) + term : (term - t) + sum;
        sum = t;
        term *= -x * x / (double(n) * double(n + 1));
    }
    return sum + small;
}
constexpr Tab make_tab() {
    Tab t = {};
    for (int i = 0; i <= kTabSize / 8; ++i) {
        const double x = 6.283185307179586476925 * i / kTabSize;
        const double c = taylor(x, false), s = taylor(x, true);
        const float ch = float(c), sh = float(s), cl = float(c - double(ch)), sl = float(s - double(sh));
        const int q = kTabSize / 4;
        // the eight octants
        t.e[i] = {ch, cl, sh, sl};
        t.e[q - i] = {sh, sl, ch, cl};
        t.e[q + i] = {-sh, -sl, ch, cl};
        t.e[2 * q - i] = {-ch, -cl, sh, sl};
        t.e[2 * q + i] = {-ch, -cl, -sh, -sl};
        t.e[3 * q - i] = {-sh, -sl, -ch, -cl};
        t.e[3 * q + i] = {sh, sl, -ch, -cl};
        t.e[(4 * q - i) % kTabSize] = {ch, cl, -sh, -sl};
    }
    return t;
}

// k and what is made of it once per thread
struct Wave {
    double k, kq;        // kq = 2 k / pi: quarter turns per metre
    float kqf, rho;      // kq in single precision; (2 k / pi - kq) / kq
    DF ik;               // 1 / k
    unsigned first, span;  // high words of the squared distances that fast_term takes
};
__device__ __forceinline__ Wave make_wave(double k) {
    Wave w;
    w.k = k;
    const double ch = 0.63661977236758138, cl = -3.9357353350364972e-17;  // 2 / pi
    w.kq = k * ch;
    w.kqf = float(w.kq);
    w.rho = float((fma(k, ch, -w.kq) + k * cl) / w.kq);
    const double ik = 1.0 / k;
    w.ik.h = float(ik);
    w.ik.l = float(ik - double(w.ik.h));
    // distances of 1e-8 m to 2^18 quarter turns (1e14 m): outside, fixed point
    // and floats run out of range, and the term is taken in doubles
    const double far = 262144.0 / w.kq;
    const double r2 = fmin(far * far, 1e28);
    w.first = unsigned(__double2hiint(1e-16));
    w.span = (k > 1e-20 && k < 1e20 && r2 > 1e-16) ? unsigned(__double2hiint(r2)) - w.first : 0u;
    return w;
}
__device__ __forceinline__ bool in_range(const Wave& w, double r2) {
    return unsigned(__double2hiint(r2)) - w.first < w.span;  // NaN and negative: beyond the span
}

// 1/r and e^{ikr} for a squared distance in range
__device__ __forceinline__ void fast_wave(const Wave& w, double r2, const TabEntry* __restrict__ tab, DF& ir, DF& c,
                                          DF& s) {
    const float rf = leading_float(__double2hiint(r2), __double2loint(r2));
    const float y0 = rsqrt_approx(rf);
    const double y = widen(y0);
    // r = g (1 - u)^(-1/2), 1 - u = g y, |u| < 2^-21: 2.5 - g y lies in [1, 2),
    // so the low word of the sum is u in units of 2^-52
    const double g = r2 * y;
    const int ui = __double2loint(__fma_rn(-g, y, 2.5));
    // whole quarter turns n by single precision: off by 0.1 at most, so f = kq g - n
    // stays within 0.6 and 6 + f in [4, 8), where a double's last bit is 2^-50
    const float nf = rintf(__fmul_rn(__fmul_rn(rf, y0), w.kqf));
    const int n = int(nf);
    long long x = __double_as_longlong(__fma_rn(g, w.kq, widen(__fsub_rn(6.0f, nf)))) - 0x4018000000000000ll;
    // r - g and the rest of kq: (n + f)(u/2 + 3 u^2/8 + rho)
    const float ff = __fmul_rn(float(int(x >> 21)), 0x1p-29f);
    const float hu = __fmul_rn(float(ui >> 8), 0x1p-45f), hul = __fmul_rn(float(ui & 255), 0x1p-53f);  // u / 2
    const float u2 = __fmaf_rn(__fmul_rn(1.5f, hu), hu, hul);  // 3 u^2 / 8 and the low part of u / 2
    const float p = __fmul_rn(nf, hu);
    const float lo = __fmaf_rn(ff, hu, __fmaf_rn(__fadd_rn(nf, ff), __fadd_rn(u2, w.rho), __fmaf_rn(nf, hu, -p)));
    const float ci = rintf(__fmul_rn(p, 0x1p26f));
    const float rem = __fadd_rn(__fmaf_rn(ci, -0x1p-26f, p), lo);
    x += ((long long)(int(ci)) << 24) + (long long)(__float2int_rn(__fmul_rn(rem, 0x1p50f)));
    const float yh = __fmul_rn(y0, hu);
    ir = df_add({y0, __fmaf_rn(y0, u2, __fmaf_rn(y0, hu, -yh))}, {yh, 0.0f});
    // the nearest table entry and the angle from it
    const unsigned long long a = ((unsigned long long)(unsigned(n)) << 50) + (unsigned long long)(x);
    const TabEntry t = tab[unsigned((a + (1ull << 41)) >> 42) & (kTabSize - 1)];
    const long long d = (long long)(a << 22) >> 22;
    const float dh = __fmul_rn(float(int(d >> 18)), 0x1p-32f), dl = __fmul_rn(float(int(d) & 0x3ffff), 0x1p-50f);
    const float ph = 1.57079637f, pl = -4.37113900e-8f;  // pi / 2
    const float e = __fmul_rn(ph, dh);
    const float el = __fadd_rn(__fmaf_rn(ph, dh, -e), __fmaf_rn(pl, dh, __fmul_rn(ph, dl)));
    const float z = __fmul_rn(e, e);
    // sin = e - e^3/6 + e^5/120, 1 - cos = e^2/2 - e^4/24; |e| <= 0.0031
    const DF sd = {e, __fmaf_rn(__fmul_rn(e, z), __fmaf_rn(z, 0.00833333333f, -0.166666667f), el)};
    const float zl = __fmaf_rn(__fadd_rn(e, e), el, __fmaf_rn(e, e, -z));
    const DF wd = {__fmul_rn(0.5f, z), __fmaf_rn(__fmul_rn(z, z), -0.0416666667f, __fmul_rn(0.5f, zl))};
    const DF C = {t.ch, t.cl}, S = {t.sh, t.sl};
    c = df_add(C, df_neg(df_add(df_mul(S, sd), df_mul(C, wd))));
    s = df_add(S, df_add(df_mul(C, sd), df_neg(df_mul(S, wd))));
}

// A staged source: position and normal, and the amplitude over the tile's scale
struct Record {
    double x, y, z, nx, ny, nz;
    DF a, b;
};
static_assert(sizeof(Record) == 64, "fp64_record_bytes");

// The term of a pair in range, without the tile's scale and, of an interface,
// without k, which as a pair of floats would be off by the same share in every term
template <int KIND>
__device__ __forceinline__ void fast_term(const Wave& w, double r2, double nd, const DF& a, const DF& b,
                                          const TabEntry* __restrict__ tab, DF& re, DF& im) {
    DF ir, c, s;
    fast_wave(w, r2, tab, ir, c, s);
    if (KIND == RSI_STAGE_PISTON) {
        const DF amp = df_mul(a, ir);  // -v0 w / (2 pi r)
        re = df_mul(amp, c);
        im = df_mul(amp, s);
        return;
    }
    // B (i - 1/(kr)) e^{ikr} cos(theta) / r,  B = -w sigma / (2 pi)
    const DF h = df_mul(df_of(nd), df_mul(ir, ir)), q = df_mul(ir, w.ik);
    const DF vr = df_neg(df_add(b, df_mul(q, a)));
    const DF vi = df_add(a, df_neg(df_mul(q, b)));
    re = df_mul(h, df_add(df_mul(vr, c), df_neg(df_mul(vi, s))));
    im = df_mul(h, df_add(df_mul(vr, s), df_mul(vi, c)));
}

// the term in doubles throughout: pairs out of range
template <int KIND>
__device__ __noinline__ double2 slow_term(double k, double r2, double nd, double a, double b) {
    if (!(r2 >= 1e-24)) return make_double2(0.0, 0.0);  // pairs closer than 1e-12 m contribute nothing
    const double rr = sqrt(r2), ir = 1.0 / rr;
    double s, c;
    sincos(k * rr, &s, &c);
    if (KIND == RSI_STAGE_PISTON) return make_double2(a * ir * c, a * ir * s);
    const double h = nd * ir * ir, vr = -ir * a - k * b, vi = -ir * b + k * a;
    return make_double2(h * (vr * c - vi * s), h * (vr * s + vi * c));
}

}  // namespace rsi_fp64
