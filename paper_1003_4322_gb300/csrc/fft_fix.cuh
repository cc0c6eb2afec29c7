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
// in FP64 to 2.38 / 1.49 / 0.98 ms, most of it integer instruction issue.
//
// The scale: with S >= sum |x_j| over the line, every sub-transform of every
// stage is bounded by S in modulus (it is a sum of x_j times unit factors), so
// scaling S below 2^63 excludes overflow whatever the input, and the inputs
// are known to 2^-62 S.  S lies between the line's 2-norm (one entry stands
// out) and sqrt(n) times it (a flat line), so the relative error grows like
// 2^-62 n at worst.  Against long double arithmetic, relative L2 error of one line
// with its results as doubles (whose own rounding is 5e-17): 5-6e-17 for lines
// with a decaying spectrum at any length, where FP64 gives 1.4-5e-16; for flat
// lines 6e-17 (n = 256), 0.8e-16 (512), 1.5e-16 (1024; FP64: 3.4e-16 or more).
//
// Rounding: every shift here has a mean error of zero on either sign of its
// operand (halves upwards where 2^-31 of the operands are halves; elsewhere to
// even or by a bit of the data), and products split their operand into a high
// word and a SIGNED low word, so that the partial product they drop has mean zero
// too.  That matters more than the size of the errors: a loss of half a unit
// with the same sign in every line adds up in phase over a transform's N^2 lines
// where the data add up like noise.  With shifts that round down, the L2 error of
// r2c on Gaussian 256^3 data was 1.1e-16, but that of the lowest modes 7.1e-14 of
// the rms mode (3.9e-13 at 512^3), against 8e-16 in FP64 arithmetic (1.0e-15).  As
// it is here no mode on the axes is off by more than 2.7e-16 (4.2e-16), for 2 %
// of the 512^3 step (32.5 -> 33.2 ms).
//
// Format: stage 0 works in |v| < 2^63, the later ones in |v| < 2^61: the
// twiddle products of stage 1 return v w / 4.  A twiddle is w = H 2^-30 + L 2^-62,
// |H| <= 2^30, |L| < 2^31 (balanced, so +-1 is exact and negation is exact).
// With v = xh 2^30 + xl / 4 (v / 4 in stage 1: the words of v themselves), v w =
// xh H + (xl H + xh L) 2^-32 + (xl L) 2^-64, of which the last is dropped and the
// middle one is the upper word of a sum that starts at 2^31.  To round xh to
// nearest, the butterflies before a twiddled stage add 2^31 or 2^29 to
// their input 0, which adds it to each of their outputs (fft_fix_line.cuh).
// The sum stays below 2^63 while |v| < 0.914 of its range: fix_top's 1.1.
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
// Lower word of (hi:lo) shifted right by s <= 32.
NSK_FIX unsigned fshr(unsigned lo, unsigned hi, int s) {
#ifdef __CUDA_ARCH__
    return __funnelshift_rc(lo, hi, s);
#else
    return s == 32 ? hi : s ? (lo >> s) | (hi << (32 - s)) : lo;
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

// A constant c in (0, 1) as add + H 2^-31 + L 2^-63, |H| <= 2^30.
struct FixC {
    int add, H, L;
};

// cos(2 pi key / 288), 0 < key < 72, for the angles of the register DFTs
// (values of the mathematical constants; sin key = cos (72 - key)).
__host__ __device__ constexpr FixC fixcos(int key) {
    switch (key) {
    case 8: return FixC{1, -32625102, 74472808};
    case 16: return FixC{1, -129509111, 1219784300};
    case 18: return FixC{1, -163467459, -902489949};
    case 24: return FixC{1, -287708255, 1630710223};
    case 32: return FixC{1, -502415733, 1027663049};
    case 36: return FixC{1, -628983398, -51432894};
    case 40: return FixC{1, -767107767, -262638930};
    case 48: return FixC{0, 1 << 30, 0};   // 1/2
    case 54: return FixC{0, 821806413, 1565705635};
    case 56: return FixC{0, 734482665, 337111738};
    case 64: return FixC{0, 372906622, 192121251};
    default: return FixC{0, 0, 0};
    }
}

// x = xh 2^32 + xl with xl signed: x c = xh 2H + (xl H + xh L) 2^-31 + add x, the
// middle term rounded (below 0.72 2^63 for every pair of constants of a rotation).
NSK_FIX int xhi(i64 x) { return lhi(x) + (int)(llo(x) >> 31); }
NSK_FIX i64 mad2h(int xh, int H, i64 c) {   // xh 2H + c; 2^31 is no int
    if (H == 1 << 30) return c + (i64)((unsigned long long)(i64)xh << 31);
    if (H == -(1 << 30)) return c - (i64)((unsigned long long)(i64)xh << 31);
    return madw(xh, 2 * H, c);
}
// x c for a constant c, |x| < 2^63.
NSK_FIX i64 mulc(i64 x, FixC c) {
    const int xh = xhi(x), xl = (int)llo(x);
    i64 t = madw(xl, c.H, 1LL << 30);
    if (c.L) t = madw(xh, c.L, t);
    return mad2h(xh, c.H, (t >> 31) + (c.add ? x : 0));
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
    const int xh = xhi(v.x), xl = (int)llo(v.x), yh = xhi(v.y), yl = (int)llo(v.y);
    const i64 tx = madw(yh, -s.L, madw(yl, -s.H, madw(xh, c.L, madw(xl, c.H, 1LL << 30))));
    const i64 ty = madw(xh, s.L, madw(xl, s.H, madw(yh, c.L, madw(yl, c.H, 1LL << 30))));
    i64 rx = mad2h(xh, c.H, mad2h(yh, -s.H, tx >> 31));
    i64 ry = mad2h(yh, c.H, mad2h(xh, s.H, ty >> 31));
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
// im.H, im.L}.  k2 = 2: v in stage 0's range, the result v w / 4; else k2 = 0.  v
// carries the offset NSK_FIX_OFF << k2 in both parts, which its split takes off.
// start = 2^31 rounds halves up, 2^31 - 1 down: v / 4 times +-1 or +-i is a half for
// one v in four, so stage 1 takes either by turns (fix_tie).
#define NSK_FIX_OFF (1 << 29)
template <int DIR> NSK_FIX L2 cmul_w(L2 v, int4 w, int k2, i64 start) {
    const int xh = (int)fshr(llo(v.x), (unsigned)lhi(v.x), 30 + k2), yh = (int)fshr(llo(v.y), (unsigned)lhi(v.y), 30 + k2);
    const int xl = (int)((llo(v.x) << (2 - k2)) ^ 0x80000000u), yl = (int)((llo(v.y) << (2 - k2)) ^ 0x80000000u);
    const int ih = DIR < 0 ? w.z : -w.z, il = DIR < 0 ? w.w : -w.w;
    const i64 tx = madw(yh, -il, madw(yl, -ih, madw(xh, w.y, madw(xl, w.x, start))));
    const i64 ty = madw(xh, il, madw(xl, ih, madw(yh, w.y, madw(yl, w.x, start))));
    return mkl(madw(xh, w.x, madw(yh, -ih, (i64)lhi(tx))), madw(yh, w.x, madw(xh, ih, (i64)lhi(ty))));
}

// 0 or 1 with equal probability, from a value of the line: its lowest bit and its
// sign, one of which at least varies from line to line (doubles as inputs end
// in zero bits, a mean flow fixes the sign).
NSK_FIX int fix_tie(i64 v) { return (int)((llo(v) ^ ((unsigned)lhi(v) >> 31)) & 1u); }

// v / 2, halves to even.
NSK_FIX i64 half_even(i64 v) {
    const i64 h = v >> 1;
    return h + (i64)(llo(v) & llo(h) & 1u);
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
        const L2 t = mkl(a[0].x - half_even(s.x), a[0].y - half_even(s.y)), e = mkl(mulc(d.x, h), mulc(d.y, h));
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
// first multiplied by a power of two (line_scale in fft_fix_line.cuh).
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

// Exponent e (a double's biased one) with 1.1 S < 2^(e+1): a double with this
// exponent maps to bit 62, so that a line with the sum S stays below 2^63 / 1.1.
NSK_FIX int fix_top(float S) { return S > 0.f ? (int)(fix_f2u(S * 1.1f) >> 23) + 896 : 1023; }

// M shifted right by any number of bits: PTX's shift, unlike C++'s, is defined
// beyond 63 (all zeros).
NSK_FIX unsigned long long fix_shr(unsigned long long M, unsigned r) {
#ifdef __CUDA_ARCH__
    unsigned long long d;
    asm("shr.u64 %0, %1, %2;" : "=l"(d) : "l"(M), "r"(r));
    return d;
#else
    return r < 64u ? M >> r : 0;
#endif
}

// The double with upper and lower words (hi, lo) times 2^(62 - (top - 1023)),
// truncated towards zero; exponents above top do not occur.
NSK_FIX i64 fix_from(int hi, unsigned lo, int top) {
    const unsigned e = ((unsigned)hi >> 20) & 0x7ffu, m = ((unsigned)hi & 0xfffffu) | 0x100000u;
    const unsigned long long M = ((unsigned long long)m << 42) | ((unsigned long long)lo << 10);
    const i64 t = (i64)fix_shr(M, (unsigned)top - e), s = (i64)(hi >> 31);
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
