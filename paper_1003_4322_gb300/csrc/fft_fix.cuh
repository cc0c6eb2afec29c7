// fft_fix.cuh -- 64-bit block fixed-point arithmetic for the FP64 line
// transforms (the 1D FFTs of Sec. 2 in the plain form's precision).
//
// Why: GB300 issues two FP64 instructions per SM and clock, 1/64 of its FP32
// rate, and the FP64 passes sat on that limit (FP64 pipe 85 % busy, 17 clocks
// per point and SM where a point's bytes take 1.2).  Integer instructions run
// at 64 per SM and clock on each of two pipes: measured per SM and clock, a
// 64-bit add 60 against 1.7 FP64 additions, the complex product cmul_w 2.0
// against 0.4.  A Fourier transform of a line is linear with unit-modulus
// factors, so one power-of-two scale per line serves every intermediate value,
// and 63 bits under that scale are more than the 53 of a double.  At 512^3
// (three components) the passes went from 11.5 / 6.7 / 4.5 ms (z c2r, y, x)
// in FP64 to 2.35 / 1.44 / 0.98 ms, bound by integer instruction issue.
//
// The scale: with S >= sum |x_j| over the line, every sub-transform of every
// stage is bounded by S in modulus (it is a sum of x_j times unit factors), so
// scaling S below 2^63 excludes overflow whatever the input, and the inputs
// are known to 2^-62 S.  S lies between the line's 2-norm (one entry stands
// out) and sqrt(n) times it (a flat line), so the relative error grows like
// 2^-62 n at worst.  Against long double arithmetic, relative L2 error of one
// line, worst over plans, signs and scales: 0.5-0.7e-16 for lines with a
// decaying spectrum at any length, where FP64 gives 1.4-5e-16; for flat lines
// 0.7e-16 (n = 128), 1.6e-16 (512), 2.9e-16 (1024; FP64: 3.4e-16 or more).
//
// Format: stage 0 works in |v| < 2^63.  The twiddle products of stage 1 take
// their operand's upper 32 bits and next 30 bits and return v w / 4 (the
// split that needs no shift), so from there |v| < 2^61 and a split at bit 30
// makes the upper part fit 32 bits.  A twiddle is w = H 2^-30 + L 2^-60,
// |H| <= 2^30, |L| <= 2^29 (balanced, so +-1 is exact and negation is exact).
// The dropped terms and roundings of a product are about one unit.
#pragma once
#include <stdint.h>

#include "fft_core.cuh"

namespace nsk {

#define NSK_FIX __host__ __device__ __forceinline__

typedef long long i64;

// A complex fixed-point value.  Its operations are the names the generic
// register DFTs of fft_core.cuh use.
struct L2 {
    i64 x, y;
};
NSK_FIX L2 mkl(i64 a, i64 b) {
    L2 r;
    r.x = a;
    r.y = b;
    return r;
}
NSK_FIX L2 ladd(L2 a, L2 b) { return mkl(a.x + b.x, a.y + b.y); }
NSK_FIX L2 lsub(L2 a, L2 b) { return mkl(a.x - b.x, a.y - b.y); }
// a + S i b
template <int S> NSK_FIX L2 ladd_i(L2 a, L2 b) {
    return S > 0 ? mkl(a.x - b.y, a.y + b.x) : mkl(a.x + b.y, a.y - b.x);
}

NSK_FIX int lhi(i64 a) { return (int)(a >> 32); }
NSK_FIX unsigned llo(i64 a) { return (unsigned)(unsigned long long)a; }
// One wide multiply(-add) each.  The instruction is spelled out because the
// compiler otherwise turns a (-b) + c into c - a b, which takes three
// instructions (a complex product 57 instead of 28, 0.76 against 0.50 clocks
// per SM).
NSK_FIX i64 madw(int a, int b, i64 c) {
#ifdef __CUDA_ARCH__
    i64 d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return (i64)a * b + c;
#endif
}
NSK_FIX i64 mulw(int a, int b) {
#ifdef __CUDA_ARCH__
    i64 d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
#else
    return (i64)a * b;
#endif
}
// Lower word of (hi:lo) shifted right by s < 32.
NSK_FIX unsigned fshr(unsigned lo, unsigned hi, int s) {
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, s);
#else
    return s ? (lo >> s) | (hi << (32 - s)) : lo;
#endif
}
// Upper word of (hi:lo) shifted left by s < 32.
NSK_FIX unsigned fshl(unsigned lo, unsigned hi, int s) {
#ifdef __CUDA_ARCH__
    return __funnelshift_l(lo, hi, s);
#else
    return s ? (hi << s) | (lo >> (32 - s)) : hi;
#endif
}

// A constant c in (0, 1) as add + H 2^-32 + L 2^-62.
struct FixC {
    int add, H, L;
};

// cos(2 pi key / 288), 0 < key < 72, for the angles of the register DFTs
// (values of the mathematical constants; sin key = cos (72 - key)).
__host__ __device__ constexpr FixC fixcos(int key) {
    switch (key) {
    case 8: return FixC{1, -65250204, 37236404};
    case 16: return FixC{1, -259018221, -463849674};
    case 18: return FixC{1, -326934918, -451244975};
    case 24: return FixC{1, -575416509, -258386713};
    case 32: return FixC{1, -1004831466, 513831524};
    case 36: return FixC{1, -1257966796, -25716447};
    case 40: return FixC{1, -1534215534, -131319465};
    case 48: return FixC{0, 2147483647, 1073741824};   // 1/2; -H must not overflow
    case 54: return FixC{0, 1643612827, -290889006};
    case 56: return FixC{0, 1468965330, 168555869};
    case 64: return FixC{0, 745813244, 96060625};
    default: return FixC{0, 0, 0};
    }
}

// x c for a constant c, |x| < 2^63.
NSK_FIX i64 mulc(i64 x, FixC c) {
    const int xh = lhi(x), xl = (int)(llo(x) >> 2);
    const i64 t = c.L ? madw(xh, c.L, mulw(xl, c.H)) : mulw(xl, c.H);
    return madw(xh, c.H, (t >> 30) + (c.add ? x : 0));
}

// v exp(DIR 2 pi i m / R), m and R compile-time constants once unrolled.
template <int R, int DIR> NSK_FIX L2 lrot(L2 v, int m) {
    int key = (m % R) * (288 / R);
    if (DIR < 0) key = (288 - key) % 288;
    const int q = key / 72, r = key % 72;
    if (q == 1) v = mkl(-v.y, v.x);
    if (q == 2) v = mkl(-v.x, -v.y);
    if (q == 3) v = mkl(v.y, -v.x);
    if (r == 0) return v;
    if (r == 36) {
        const FixC c = fixcos(36);
        const i64 p = mulc(v.x, c), s = mulc(v.y, c);
        return mkl(p - s, p + s);
    }
    const FixC c = fixcos(r), s = fixcos(72 - r);
    const int xh = lhi(v.x), xl = (int)(llo(v.x) >> 2), yh = lhi(v.y), yl = (int)(llo(v.y) >> 2);
    const i64 tx = madw(yh, -s.L, madw(yl, -s.H, madw(xh, c.L, mulw(xl, c.H))));
    const i64 ty = madw(xh, s.L, madw(xl, s.H, madw(yh, c.L, mulw(yl, c.H))));
    i64 rx = madw(xh, c.H, madw(yh, -s.H, tx >> 30));
    i64 ry = madw(yh, c.H, madw(xh, s.H, ty >> 30));
    if (c.add) {
        rx += v.x;
        ry += v.y;
    }
    if (s.add) {
        rx -= v.y;
        ry += v.x;
    }
    return mkl(rx, ry);
}

// v w (DIR < 0) or v conj(w) (DIR > 0) with w = (H, L) parts {re.H, re.L,
// im.H, im.L}; first: v in stage 0's range, the result v w / 4.
template <int DIR> NSK_FIX L2 cmul_w(L2 v, int4 w, bool first) {
    int xh, yh;
    unsigned xl, yl;
    if (first) {
        xh = lhi(v.x);
        yh = lhi(v.y);
        xl = llo(v.x) >> 2;
        yl = llo(v.y) >> 2;
    } else {
        xh = (int)fshr(llo(v.x), (unsigned)lhi(v.x), 30);
        yh = (int)fshr(llo(v.y), (unsigned)lhi(v.y), 30);
        xl = llo(v.x) & 0x3fffffffu;
        yl = llo(v.y) & 0x3fffffffu;
    }
    const int ih = DIR < 0 ? w.z : -w.z, il = DIR < 0 ? w.w : -w.w;
    const i64 tx = madw(yh, -il, madw((int)yl, -ih, madw(xh, w.y, mulw((int)xl, w.x))));
    const i64 ty = madw(xh, il, madw((int)xl, ih, madw(yh, w.y, mulw((int)yl, w.x))));
    return mkl(madw(xh, w.x, madw(yh, -ih, tx >> 30)), madw(yh, w.x, madw(xh, ih, ty >> 30)));
}

// Register DFTs, the decompositions of fft_core.cuh in this arithmetic.
template <int R, int DIR> struct LDft;
template <int DIR> struct LDft<2, DIR> {
    static NSK_FIX void run(L2 *a) {
        const L2 t = a[0];
        a[0] = ladd(t, a[1]);
        a[1] = lsub(t, a[1]);
    }
};
template <int DIR> struct LDft<3, DIR> {
    static NSK_FIX void run(L2 *a) {
        const FixC h = fixcos(24);   // sqrt(3)/2
        const L2 s = ladd(a[1], a[2]), d = lsub(a[1], a[2]);
        const L2 t = mkl(a[0].x - (s.x >> 1), a[0].y - (s.y >> 1)), e = mkl(mulc(d.x, h), mulc(d.y, h));
        a[0] = ladd(a[0], s);
        a[1] = ladd_i<DIR>(t, e);
        a[2] = ladd_i<-DIR>(t, e);
    }
};
template <int DIR> struct LDft<4, DIR> {
    static NSK_FIX void run(L2 *a) {
        const L2 s02 = ladd(a[0], a[2]), d02 = lsub(a[0], a[2]);
        const L2 s13 = ladd(a[1], a[3]), d13 = lsub(a[1], a[3]);
        a[0] = ladd(s02, s13);
        a[2] = lsub(s02, s13);
        a[1] = ladd_i<DIR>(d02, d13);
        a[3] = ladd_i<-DIR>(d02, d13);
    }
};
template <int R1, int R2, int DIR> struct LDftComposite {
    static NSK_FIX void run(L2 *a) {
        constexpr int R = R1 * R2;
        L2 B[R];
#pragma unroll
        for (int j2 = 0; j2 < R2; j2++) {
            L2 b[R1];
#pragma unroll
            for (int j1 = 0; j1 < R1; j1++) b[j1] = a[R2 * j1 + j2];
            LDft<R1, DIR>::run(b);
#pragma unroll
            for (int k1 = 0; k1 < R1; k1++) B[j2 * R1 + k1] = lrot<R, DIR>(b[k1], j2 * k1);
        }
#pragma unroll
        for (int k1 = 0; k1 < R1; k1++) {
            L2 c[R2];
#pragma unroll
            for (int j2 = 0; j2 < R2; j2++) c[j2] = B[j2 * R1 + k1];
            LDft<R2, DIR>::run(c);
#pragma unroll
            for (int k2 = 0; k2 < R2; k2++) a[k1 + R1 * k2] = c[k2];
        }
    }
};
template <int DIR> struct LDft<6, DIR> : LDftComposite<2, 3, DIR> {};
template <int DIR> struct LDft<8, DIR> : LDftComposite<2, 4, DIR> {};
template <int DIR> struct LDft<9, DIR> : LDftComposite<3, 3, DIR> {};
template <int DIR> struct LDft<12, DIR> : LDftComposite<4, 3, DIR> {};
template <int DIR> struct LDft<16, DIR> : LDftComposite<4, 4, DIR> {};

// ---------------------------------------------------------------- conversions

NSK_FIX int fix_clz(unsigned a) {
#ifdef __CUDA_ARCH__
    return __clz((int)a);
#else
    return a ? __builtin_clz(a) : 32;
#endif
}
NSK_FIX float fix_u2f(unsigned u) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    union { unsigned u; float f; } c;
    c.u = u;
    return c.f;
#endif
}
NSK_FIX unsigned fix_f2u(float f) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(f);
#else
    union { unsigned u; float f; } c;
    c.f = f;
    return c.u;
#endif
}

// The line sum S is accumulated in FP32 from the upper words of the doubles:
// exponent field e - 896 is the FP32 field of the same power of two, and the
// upper 20 mantissa bits follow.  Entries below 2^-126 count as zero and
// those above 2^127 as that; lines whose sum leaves [kFixLow, kFixHigh] are
// first multiplied by a power of two (line_scale in fft_fix.cu).
#define NSK_FIX_LOW 8.271806e-25f   // 2^-80
#define NSK_FIX_HIGH 1.2676506e30f  // 2^100

// Upper bound of |z|, within 8 %, of a complex value given by the upper words
// of its parts (max + (sqrt(2) - 1) min); mx collects the largest word.
NSK_FIX float fix_mag(int hx, int hy, unsigned &mx) {
    unsigned m = (unsigned)hx & 0x7fffffffu, k = (unsigned)hy & 0x7fffffffu;
    mx = mx > m ? mx : m;
    mx = mx > k ? mx : k;
    m = m > (896u << 20) ? m : (896u << 20);
    k = k > (896u << 20) ? k : (896u << 20);
    const float a = fix_u2f((m << 3) + 0x40000000u), b = fix_u2f((k << 3) + 0x40000000u);
    return fmaxf(a, b) + 0.41421360f * fminf(a, b);
}

// Power of two above S sqrt(2) (|z| <= sqrt(2) max) and the truncated
// mantissas, as the biased double exponent of the range [2^e, 2^(e+1)) that
// holds it: a double with this exponent maps to bit 62.
NSK_FIX int fix_top(float S) { return S > 0.f ? (int)(fix_f2u(S * 1.001f) >> 23) + 896 : 1023; }

// The double with upper and lower words (hi, lo) times 2^(62 - (top - 1023)),
// truncated towards zero; exponents above top do not occur.
NSK_FIX i64 fix_from(int hi, unsigned lo, int top) {
    const unsigned e = ((unsigned)hi >> 20) & 0x7ffu, m = ((unsigned)hi & 0xfffffu) | 0x100000u;
    const unsigned long long M = ((unsigned long long)m << 42) | ((unsigned long long)lo << 10);
    unsigned r = (unsigned)top - e;
#ifndef __CUDA_ARCH__
    r = r < 63u ? r : 63u;   // the device's shift yields zero beyond 63
#endif
    const i64 t = (i64)(M >> r), s = (i64)(hi >> 31);
    return (t ^ s) - s;
}

// The double nearest v, scaled so that a leading bit at bit 63 gives the
// biased exponent ebase (bit 62: ebase - 1, ...); halves round up in
// magnitude, and negative values go through their one's complement (off by one
// unit of v).  The result must be a normal number or zero.
NSK_FIX void fix_to(i64 v, int ebase, unsigned &hi, unsigned &lo) {
    const unsigned s = (unsigned)(lhi(v) >> 31), ah = (unsigned)lhi(v) ^ s, al = llo(v) ^ s;
    const bool high = ah != 0;
    const unsigned a = high ? ah : al, b = high ? al : 0u;
    const int z = fix_clz(a);   // 32 for zero: the shifts then see a = b = 0
    const unsigned nh = fshl(b, a, z & 31), nl = b << (z & 31);
    const unsigned long long r = (((((unsigned long long)nh << 32) | nl) >> 1) + 0x200) >> 10;
    const unsigned e = (unsigned)((high ? ebase - 1 : ebase - 33) - z) << 20;
    hi = (a ? (unsigned)(r >> 32) + e : 0u) | (s & 0x80000000u);
    lo = (unsigned)r;
}

}  // namespace nsk
