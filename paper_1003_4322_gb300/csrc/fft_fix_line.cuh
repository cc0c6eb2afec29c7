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

// Scale of one line: `top` (fix_from) and, for lines outside the range of the
// FP32 sum (odd), a factor that the results are multiplied by.
struct LineScale {
    int top;
    bool any;    // some line of the CTA is odd
    double mul;  // 1 for the others
};

// The raw value x times the power of two f (a line outside the FP32 range).
NSK_DEV i64 raw_scaled(i64 x, double f) { return __double_as_longlong(__longlong_as_double(x) * f); }

// v: NV raw complex values (the bits of doubles) of this thread; TWICE says that
// they count twice in the sum (both members of a Hermitian pair).  A line of
// entries in 2^-80 .. 2^100 needs one reduction.  Others (CTA-uniform branch)
// are first brought to about 1 by a power of two taken from their largest
// entry; a line with a NaN or an infinity gets the factor NaN.  skip(i)
// (CTA-uniform): v[i] is zero in the whole CTA.
template <int NV, bool TWICE, class Skip>
NSK_DEV LineScale line_scale(L2 (&v)[NV], const LineGeo &g, unsigned *sh, Skip skip) {
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
    LineScale r{0, __syncthreads_or(odd) != 0, 1.0};
    if (r.any) {
        const unsigned lm = line_reduce<OpMax>(mx, g, sh);
        if (odd) {
            const int e = (int)(lm >> 20);
            int a = 1023 - e;
            a = a < -1000 ? -1000 : a > 1000 ? 1000 : a;
            const double f = __longlong_as_double((i64)(1023 + a) << 52);
            r.mul = e == 0x7ff ? __longlong_as_double(0x7ff8000000000000LL)
                               : __longlong_as_double((i64)(1023 - a) << 52);
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
    r.top = fix_top(S);
    return r;
}

NSK_DEV i64 fix_from_raw(i64 raw, int top) { return fix_from(lhi(raw), llo(raw), top); }
NSK_DEV L2 fix_from_raw(L2 raw, int top) { return mkl(fix_from_raw(raw.x, top), fix_from_raw(raw.y, top)); }

// Conversion of a line's results; ebase as fix_to's.  On the integer pipes (23
// instructions a value): two FP64 additions can do it too, but all of a CTA's
// conversions come together at its end, where the FP64 pipe made the passes
// 20 % slower (an eighth to a quarter of the values there: 0.6 % faster).
struct FixOut {
    int ebase;
    NSK_DEV double operator()(i64 v) const {
        unsigned hi, lo;
        fix_to(v, ebase, hi, lo);
        return __hiloint2double((int)hi, (int)lo);
    }
};

// CTAs of 256 threads an SM is to hold, by the registers E values take; more
// or fewer change a 512^3 step by less than 1 %, the passes being bound by
// instruction issue.
template <int E> struct MinCtas { enum { n = E >= 9 ? 2 : E == 8 ? 3 : 4 }; };

// Multiply by the stage twiddles and run the radix-R DFT of butterfly b.
template <int R, int E, int DIR>
NSK_DEV void fix_butterfly(L2 (&v)[E], int b, int k, int p, const int4 *__restrict__ tab, bool first) {
    const int sh = first ? 2 : 0;
    v[b * R] = mkl(v[b * R].x >> sh, v[b * R].y >> sh);
#pragma unroll
    for (int q = 1; q < R; q++) {
        const int4 w = __ldg(tab + (q - 1) * p + k);
        v[b * R + q] = cmul_w<DIR>(v[b * R + q], w, first);
    }
    LDft<R, DIR>::run(&v[b * R]);
}

// One stage s >= 1.  The line comes from sl; every stage but the last writes
// it back through ss (between barriers); the last leaves its results in v, in
// the order of the line: v[j] is element slot + j T.
template <int R, int E, int DIR, class SL, class SS>
NSK_DEV void fix_stage(L2 (&v)[E], bool active, int slot, int T, int p, const int4 *__restrict__ tab,
                       bool first, bool last, SL sl, SS ss) {
    constexpr int B = E / R;
    const int nR = T * B;
    const unsigned magic = 0xffffffffu / (unsigned)p + 1u;   // i / p for i p < 2^32
    if (active) {
#pragma unroll
        for (int b = 0; b < B; b++)
#pragma unroll
            for (int q = 0; q < R; q++) v[b * R + q] = sl(slot + b * T + q * nR);
#pragma unroll
        for (int b = 0; b < B; b++) {
            const int i = slot + b * T;
            fix_butterfly<R, E, DIR>(v, b, i - p * (int)__umulhi((unsigned)i, magic), p, tab, first);
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
#pragma unroll
        for (int b = 0; b < B; b++) {
            const int i = slot + b * T;
            const int k = i - p * (int)__umulhi((unsigned)i, magic);
            const int j = (i - k) * R + k;
#pragma unroll
            for (int q = 0; q < R; q++) ss(j + q * p, v[b * R + q]);
        }
    }
    __syncthreads();
}

// The stages of one line.  v holds the fixed-point elements slot + q T on
// entry and the transform's on return.  sl / ss: the shared line.  smem_read:
// the inputs came from it, so a barrier must precede the first store.
template <int E, int DIR, class SL, class SS>
NSK_DEV void fix_line(L2 (&v)[E], bool active, int slot, int T, const FixK &pl, bool smem_read, SL sl, SS ss) {
    const int nst = pl.nst;
    if (active) LDft<E, DIR>::run(v);
    if (nst == 1) return;   // T = 1: element q is v[q]
    if (smem_read) __syncthreads();
    if (active) {
#pragma unroll
        for (int q = 0; q < E; q++) ss(slot * E + q, v[q]);
    }
    __syncthreads();
    int p = E;
    const int4 *tab = pl.tab;
    for (int s = 1; s < nst; s++) {
        const bool last = s == nst - 1;
        const int R = pl.rad(s);
#define NSK_FIX_ST(RR)                                                                                   \
    case RR:                                                                                             \
        if constexpr (E % RR == 0) fix_stage<RR, E, DIR>(v, active, slot, T, p, tab, s == 1, last, sl, ss); \
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
