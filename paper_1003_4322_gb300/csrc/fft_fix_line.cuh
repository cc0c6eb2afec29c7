// fft_fix_line.cuh -- the line transform of the FP64 passes in block fixed
// point (fft_fix.cuh), shared by the strided and the z kernels.
//
// A line of n values is held by T = n/E threads, E values each, in the
// Stockham stages of fft_core.cuh.  The scale of a line is found once, from
// the raw doubles the threads have just loaded: per thread the sum of |z|
// bounds, then a fixed-order reduction over the line's threads.
#pragma once
#include "fft_fix.cuh"
#include "ns_internal.h"

namespace nsk {

// What a kernel needs of a plan: the radices and the stage twiddles, laid out
// per stage s >= 1 (span p, radix R) as [q - 1][k], 1 <= q < R, k < p, so that
// a warp's lanes read consecutive entries.
struct FixK {
    int n, nst;
    unsigned long long radix;
    const int4 *tab;
    __device__ __forceinline__ int rad(int s) const { return (int)((radix >> (5 * s)) & 31u); }
};

// Where a line's threads sit in the CTA, for reductions over a line.
//  kCols: lanes run along 2^cl columns, slots along the rest; whole warps.
//  kSub:  2^cl <= 32 consecutive lanes per line.
//  kWarps: cnt whole warps per line.
//  kAny:  cnt consecutive threads per line, any count.
enum { kCols, kSub, kWarps, kAny };
struct LineGeo {
    int mode, cl, cnt, line;   // line: column (kCols) or line index in the CTA
};

struct OpAdd {
    static NSK_DEV unsigned run(unsigned a, unsigned b) {
        return __float_as_uint(__uint_as_float(a) + __uint_as_float(b));
    }
};
struct OpMax {
    static NSK_DEV unsigned run(unsigned a, unsigned b) { return a > b ? a : b; }
};

// Reduction over the threads of a line, the same value (bit for bit) in each
// and independent of the other lines; every thread of the CTA calls it.  sh
// holds one word per thread and is free again after the next barrier.
template <class Op> NSK_DEV unsigned line_reduce(unsigned v, const LineGeo &g, unsigned *sh) {
    const int tid = threadIdx.x;
    if (g.mode == kSub) {
        for (int o = 1; o < (1 << g.cl); o <<= 1) v = Op::run(v, __shfl_xor_sync(0xffffffffu, v, o));
        return v;
    }
    if (g.mode == kCols) {
        for (int o = 1 << g.cl; o < 32; o <<= 1) v = Op::run(v, __shfl_xor_sync(0xffffffffu, v, o));
        const int ct = 1 << g.cl;
        if ((tid & 31) < ct) sh[(tid >> 5) * ct + (tid & 31)] = v;
        __syncthreads();
        v = sh[g.line];
        for (int w = 1; w < (int)(blockDim.x >> 5); w++) v = Op::run(v, sh[w * ct + g.line]);
        return v;
    }
    if (g.mode == kWarps) {
        for (int o = 1; o < 32; o <<= 1) v = Op::run(v, __shfl_xor_sync(0xffffffffu, v, o));
        if ((tid & 31) == 0) sh[tid >> 5] = v;
        __syncthreads();
        v = sh[g.line * g.cnt];
        for (int w = 1; w < g.cnt; w++) v = Op::run(v, sh[g.line * g.cnt + w]);
        return v;
    }
    sh[tid] = v;
    __syncthreads();
    v = sh[g.line * g.cnt];
    for (int w = 1; w < g.cnt; w++) v = Op::run(v, sh[g.line * g.cnt + w]);
    return v;
}

// Between the passes of a transform values stay in fixed point: 64-bit
// integers v with one exponent t per line, value = v 2^(t - 1085) (t is the
// biased double exponent of bit 62).  That saves a conversion to double (23
// instructions a value) at the end of one pass and one from it (17, and the
// line sum) at the start of the next, for shifts, and two roundings to 53 bits
// (512^3: x inverse 1.10 -> 0.98 ms, y inverse 1.60 -> 1.44, r2c with products
// 2.84 -> 2.49, y forward 1.52 -> 1.32; with entries and products rounded to
// nearest they take 0.98, 1.49, 2.54 and 1.39).  kZeroT: a line of zeros; kNanT: a
// line with a NaN or an infinity; both stay beyond +-kEdgeT through the small
// steps the passes add.
constexpr int kZeroT = -(1 << 20), kNanT = 1 << 20, kEdgeT = 1 << 19;

// Scale of a line read as doubles: `top` for fix_from (of the entries, which
// line_scale has multiplied by a power of two if the line lies outside the
// range of the FP32 sum) and the line's t.
struct LineScale {
    int top, t;
};

// Bits that a line's inputs leave free below 2^63: a plan of one stage has no
// twiddle products that would return a quarter, so its inputs come in below 2^61.
NSK_DEV int fix_room(const FixK &pl) { return pl.nst > 1 ? 0 : 2; }

// The raw value x times the power of two f (a line outside the FP32 range).
NSK_DEV i64 raw_scaled(i64 x, double f) { return __double_as_longlong(__longlong_as_double(x) * f); }

// v: NV raw complex values (the bits of doubles) of this thread; TWICE says that
// they count twice in the sum (both members of a Hermitian pair).  A line of
// entries in 2^-80 .. 2^100 needs one reduction.  Others (CTA-uniform branch)
// are first brought to about 1 by a power of two taken from their largest
// entry; a line with a NaN or an infinity gets the factor NaN.  skip(i)
// (CTA-uniform): v[i] is zero in the whole CTA.
template <int NV, bool TWICE, class Skip>
NSK_DEV LineScale line_scale(L2 (&v)[NV], const LineGeo &g, unsigned *sh, int room, Skip skip) {
    auto sum = [&](unsigned &mx) {
        float s = 0.f;
        unsigned low = 0;   // the smallest subnormals have an empty upper word
#pragma unroll
        for (int i = 0; i < NV; i++) {
            if (skip(i)) continue;
            s += fix_mag(lhi(v[i].x), lhi(v[i].y), mx);
            low |= llo(v[i].x) | llo(v[i].y);
        }
        if (mx == 0 && low != 0) mx = 1;
        if (mx != 0 && s < 7.8886091e-31f) s = 7.8886091e-31f;   // 2^-100: not a zero line
        if (mx >= (1100u << 20)) s = 2.f * NSK_FIX_HIGH;
        return TWICE ? 2.f * s : s;
    };
    unsigned mx = 0;
    float S = __uint_as_float(line_reduce<OpAdd>(__float_as_uint(sum(mx)), g, sh));
    const bool odd = S != 0.f && !(S >= NSK_FIX_LOW && S <= NSK_FIX_HIGH);
    LineScale r{0, 0};
    if (__syncthreads_or(odd)) {
        const unsigned lm = line_reduce<OpMax>(mx, g, sh);
        if (odd) {
            const int e = (int)(lm >> 20);
            int a = 1023 - e;
            a = a < -1000 ? -1000 : a > 1000 ? 1000 : a;
            const double f = __longlong_as_double((i64)(1023 + a) << 52);
            r.t = e == 0x7ff ? kNanT : -a;
#pragma unroll
            for (int i = 0; i < NV; i++) v[i] = mkl(raw_scaled(v[i].x, f), raw_scaled(v[i].y, f));
        }
        mx = 0;
        const float s2 = sum(mx);
        __syncthreads();
        const float S2 = __uint_as_float(line_reduce<OpAdd>(__float_as_uint(s2), g, sh));
        if (odd) S = S2;
        __syncthreads();
    }
    r.top = fix_top(S) + room;
    r.t = S == 0.f ? kZeroT : r.t + r.top;
    return r;
}

// Scale of a line read in fixed point: v[i] with exponents t[i], brought to a
// common one, which is returned.  The common exponent is at least the largest
// t (an entry is not known below its own lines' unit), and leaves the line sum
// below 2^63 / 1.1 (less the room's bits).  Entries are rounded to nearest, halves
// by a bit of the data (the shift is one at least).  sh holds two words per thread.
template <int NV, bool TWICE, class Skip>
NSK_DEV int line_scale_fixed(L2 (&v)[NV], const int (&t)[NV], const LineGeo &g, unsigned *sh, int room, Skip skip) {
    int tm = kZeroT;
#pragma unroll
    for (int i = 0; i < NV; i++)
        if (!skip(i)) tm = max(tm, t[i]);
    tm = (int)line_reduce<OpMax>((unsigned)(tm + (1 << 22)), g, sh) - (1 << 22);
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < NV; i++) {
        if (skip(i)) continue;
        // in units of 2^32; 1.5 covers the lower words (while R below is zero,
        // S plays no part, and it is large against them otherwise)
        const float a = fabsf((float)lhi(v[i].x)), b = fabsf((float)lhi(v[i].y));
        const float f = __uint_as_float((unsigned)(max(t[i] - tm, -127) + 127) << 23);
        s = fmaf(fmaf(0.41421360f, fminf(a, b), fmaxf(a, b) + 1.5f), f, s);
    }
    if (TWICE) s *= 2.f;
    const float S = __uint_as_float(line_reduce<OpAdd>(__float_as_uint(s), g, sh + blockDim.x));
    const i64 down = -(i64)fix_tie(v[0].x);
    const int R = max((int)(__float_as_uint(S * 1.1f) >> 23) + 32 - (127 + 62) + room, 1);
#pragma unroll
    for (int i = 0; i < NV; i++) {
        if (skip(i)) continue;
        const int r = min(R + tm - t[i], 63);
        const i64 h = (i64)(1ull << (r - 1));   // |v| < 2^62: no overflow
        v[i] = mkl((v[i].x + h + down) >> r, (v[i].y + h + down) >> r);
    }
    return tm + R;
}

NSK_DEV i64 fix_from_raw(i64 raw, int top) { return fix_from(lhi(raw), llo(raw), top); }
NSK_DEV L2 fix_from_raw(L2 raw, int top) { return mkl(fix_from_raw(raw.x, top), fix_from_raw(raw.y, top)); }

// Conversion of a line's results with exponent t to double, on the integer
// pipes (23 instructions a value): two FP64 additions can do it too, but all of
// a CTA's conversions come together at its end, where the FP64 pipe made the
// passes 20 % slower (an eighth to a quarter of the values there: 0.6 %
// faster).  Lines whose results could leave the range of normal numbers
// convert about 1 and are multiplied by two factors.
struct FixOut {
    int ebase;
    bool odd;
    double f1, f2;
    NSK_DEV explicit FixOut(int t) {
        odd = t < 70 || t > 1980;
        ebase = odd ? 1024 : t + 1;   // of a leading bit at bit 63
        f1 = f2 = 1.0;
        if (odd && t > -kEdgeT) {
            const int h = (t - 1023) / 2;
            f1 = t > kEdgeT ? __longlong_as_double(0x7ff8000000000000LL) : power(h);
            f2 = t > kEdgeT ? 1.0 : power(t - 1023 - h);
        }
    }
    static NSK_DEV double power(int e) {   // 2^e, |e| <= 1022
        e = e < -1022 ? -1022 : e > 1023 ? 1023 : e;
        return __longlong_as_double((i64)(1023 + e) << 52);
    }
    // The bits of the doubles, in place.  The factors are a branch of their own:
    // as a predicated multiplication per value they kept the FP64 pipe busy for
    // two clocks a point.
    template <int NV> NSK_DEV void run(L2 (&v)[NV]) const {
#pragma unroll
        for (int i = 0; i < NV; i++) {
            unsigned hi, lo;
            fix_to(v[i].x, ebase, hi, lo);
            v[i].x = (i64)(((unsigned long long)hi << 32) | lo);
            fix_to(v[i].y, ebase, hi, lo);
            v[i].y = (i64)(((unsigned long long)hi << 32) | lo);
        }
        if (odd) {
#pragma unroll 1
            for (int i = 0; i < 2; i++) {
                const double f = i ? f2 : f1;
#pragma unroll
                for (int j = 0; j < NV; j++) v[j] = mkl(raw_scaled(v[j].x, f), raw_scaled(v[j].y, f));
            }
        }
    }
};

// CTAs of 256 threads an SM is to hold, by the registers that E values take.
// At E = 8 the passes that wait for their loads most (the inverse strided ones
// and the product r2c) want 64 registers and the warps of four CTAs, the
// others 80 (512^3, four against three: y inverse 1.43 / 1.51 ms, product r2c
// 2.49 / 2.67, but y forward 1.46 / 1.34, c2r the same; two: 1.60, 3.28, 1.43).
template <int E, bool MANY> struct MinCtas { enum { n = E >= 9 ? 2 : E == 8 && !MANY ? 3 : 4 }; };

// The shared line of a transform with E elements per thread: element e at
// index (e + e / E) << cl, one entry of padding after every E so that the
// stride-E stores of stage 0 spread over the banks.  Every later stage reads
// with stride n / R and writes with stride p, both multiples of E, so the
// entries of a butterfly lie one constant step apart.
template <int E> struct LineAt {
    L2 *base;
    int cl;
    NSK_DEV int step(int stride) const { return (stride + stride / E) << cl; }   // stride % E == 0
    NSK_DEV L2 *at(int e) const { return base + ((e + e / E) << cl); }
    static size_t entries(int n) { return (size_t)n + n / E; }
};

// Multiply by the stage twiddles and run the radix-R DFT of butterfly b, whose
// inputs carry the offset NSK_FIX_OFF << k2 (k2: 2 in stage 1, else 0); the
// outputs carry NSK_FIX_OFF, or none after the last stage.  tie: how this
// thread's halves are rounded.
template <int R, int E, int DIR>
NSK_DEV void fix_butterfly(L2 (&v)[E], int b, int k, int p, const int4 *__restrict__ tab, int k2, int tie,
                           bool last) {
    if (k2 || last) {   // v / 4; the offset becomes the next one
        const int add = (last ? -(NSK_FIX_OFF << k2) : 0) + (k2 ? 2 - tie : 0);
        L2 &a = v[b * R];
        a = mkl((a.x + (i64)add) >> k2, (a.y + (i64)add) >> k2);
    }
    const int4 *w = tab + k;
    const i64 start = (1ll << 31) - tie;
#pragma unroll
    for (int q = 1; q < R; q++) {
        v[b * R + q] = cmul_w<DIR>(v[b * R + q], __ldg(w + (q - 1) * p), k2, start);
    }
    LDft<R, DIR>::run(&v[b * R]);
}

// One stage s >= 1.  The line comes from ln; every stage but the last writes it
// back there (between barriers); the last leaves its results in v, in the
// order of the line: v[j] is element slot + j T.
template <int R, int E, int DIR>
NSK_DEV void fix_stage(L2 (&v)[E], bool active, int slot, int T, int p, const int4 *__restrict__ tab,
                       int k2, int tie, bool last, const LineAt<E> &ln) {
    constexpr int B = E / R;
    const int nR = T * B;
    const unsigned magic = 0xffffffffu / (unsigned)p + 1u;   // i / p for i p < 2^32
    if (active) {
        const int step = ln.step(nR);
#pragma unroll
        for (int b = 0; b < B; b++) {
            const L2 *x = ln.at(slot + b * T);
#pragma unroll
            for (int q = 0; q < R; q++) v[b * R + q] = x[q * step];
        }
#pragma unroll
        for (int b = 0; b < B; b++) {
            const int i = slot + b * T;
            fix_butterfly<R, E, DIR>(v, b, i - p * (int)__umulhi((unsigned)i, magic), p, tab, k2, tie, last);
        }
    }
    if (last) {   // p = n / R: butterfly i writes element i + q p = slot + (b + q B) T
        L2 w[E];
#pragma unroll
        for (int j = 0; j < E; j++) w[j] = v[j];
#pragma unroll
        for (int b = 0; b < B; b++)
#pragma unroll
            for (int q = 0; q < R; q++) v[b + q * B] = w[b * R + q];
        return;
    }
    __syncthreads();
    if (active) {
        const int step = ln.step(p);
#pragma unroll
        for (int b = 0; b < B; b++) {
            const int i = slot + b * T;
            const int k = i - p * (int)__umulhi((unsigned)i, magic);
            L2 *x = ln.at((i - k) * R + k);
#pragma unroll
            for (int q = 0; q < R; q++) x[q * step] = v[b * R + q];
        }
    }
    __syncthreads();
}

// The stages of one line.  v holds the fixed-point elements slot + q T on
// entry and the transform's on return.  smem_read: the inputs came from the
// shared line, so a barrier must precede the first store.
template <int E, int DIR>
NSK_DEV void fix_line(L2 (&v)[E], bool active, int slot, int T, const FixK &pl, bool smem_read, const LineAt<E> &ln) {
    const int nst = pl.nst, tie = fix_tie(v[0].x);
    if (active) {
        if (nst > 1) v[0] = ladd(v[0], mkl((i64)NSK_FIX_OFF << 2, (i64)NSK_FIX_OFF << 2));
        LDft<E, DIR>::run(v);
    }
    if (nst == 1) return;   // T = 1: element q is v[q]
    if (smem_read) __syncthreads();
    if (active) {
        L2 *x = ln.base + ((slot * (E + 1)) << ln.cl);
#pragma unroll
        for (int q = 0; q < E; q++) x[q << ln.cl] = v[q];
    }
    __syncthreads();
    int p = E;
    const int4 *tab = pl.tab;
    for (int s = 1; s < nst; s++) {
        const bool last = s == nst - 1;
        const int k2 = s == 1 ? 2 : 0;
        const int R = pl.rad(s);
#define NSK_FIX_ST(RR)                                                                                  \
    case RR:                                                                                            \
        if constexpr (E % RR == 0) fix_stage<RR, E, DIR>(v, active, slot, T, p, tab, k2, tie, last, ln); \
        break;
        switch (R) {
            NSK_FIX_ST(2)
            NSK_FIX_ST(3)
            NSK_FIX_ST(4)
            NSK_FIX_ST(6)
            NSK_FIX_ST(8)
            NSK_FIX_ST(9)
            NSK_FIX_ST(12)
            NSK_FIX_ST(16)
        }
#undef NSK_FIX_ST
        tab += (R - 1) * p;
        p *= R;
    }
}

}  // namespace nsk
