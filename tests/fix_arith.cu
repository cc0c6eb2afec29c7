// Host check of the arithmetic of csrc/fft_fix.cuh against exact 128-bit
// products: prints, per operation, the largest |mean error| over its constants
// and the largest error of a single operation, in units of the result.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include "fft_fix.cuh"

using namespace nsk;
typedef __int128 i128;

static unsigned long long rs = 88172645463325252ull;
static unsigned long long rnd() {
    rs ^= rs << 13;
    rs ^= rs >> 7;
    rs ^= rs << 17;
    return rs * 0x2545f4914f6cdd1dull;
}
// Random direction, modulus below 2^bits / 1.1; every fourth one at that limit;
// `zeros` trailing zero bits (inputs that were doubles have some).
static L2 value(int bits, int zeros) {
    const double a = 6.283185307179586 * (double)(rnd() >> 11) * 0x1p-53, lim = ldexp(1.0, bits) / 1.1;
    const double r = rnd() % 4 ? lim * sqrt((double)(rnd() >> 11) * 0x1p-53) : lim;
    const i64 m = -(1ll << zeros), low = (i64)(rnd() >> 44);
    return mkl(((i64)(r * cos(a) * 0.999) + low) & m, ((i64)(r * sin(a) * 0.999) - low) & m);
}
struct Err {
    double sx = 0, sy = 0, worst = 0;
    long n = 0;
    void add(L2 got, i128 ex, i128 ey, int sh) {   // exact value: (ex, ey) 2^-sh
        const double dx = (double)(((i128)got.x << sh) - ex) * ldexp(1.0, -sh);
        const double dy = (double)(((i128)got.y << sh) - ey) * ldexp(1.0, -sh);
        sx += dx;
        sy += dy;
        worst = fmax(worst, fmax(fabs(dx), fabs(dy)));
        n++;
    }
    double mean() const { return fmax(fabs(sx), fabs(sy)) / n; }
};
static double mean_max, worst_max;
static void note(const Err &e) {
    mean_max = fmax(mean_max, e.mean());
    worst_max = fmax(worst_max, e.worst);
}
static void report(const char *name) {
    printf("%s %.6f %.6f\n", name, mean_max, worst_max);
    mean_max = worst_max = 0;
}

static int4 twiddle(double a) {
    const double part[2] = {cos(a), -sin(a)};
    int h[2], l[2];
    for (int i = 0; i < 2; i++) {
        h[i] = (int)llround(part[i] * 0x1p30);
        l[i] = (int)((long long)(rnd() >> 32) - 0x80000000ll);   // any low word
        if (l[i] == (int)0x80000000) l[i]++;
    }
    return make_int4(h[0], l[0], h[1], l[1]);
}

template <int DIR> static void products(int k2, long M) {
    for (int t = 0; t < 24; t++) {
        int4 w = twiddle(0.2617 * t + 0.01);
        const int one = t & 2 ? -(1 << 30) : 1 << 30;   // +-1, +-i exactly, and with the largest low words
        if (t < 4) w = t & 1 ? make_int4(0, 0, one, 0) : make_int4(one, 0, 0, 0);
        else if (t < 8) w = t & 1 ? make_int4(0, 0x7fffffff, one, -0x7fffffff) : make_int4(one, 0x7fffffff, 0, 0x7fffffff);
        const i128 wr = ((i128)w.x << 32) + w.y, wi = (DIR < 0 ? 1 : -1) * (((i128)w.z << 32) + w.w);
        Err e;
        const i64 off = (i64)NSK_FIX_OFF << k2;
        for (long i = 0; i < M; i++) {
            const L2 v = value(61 + k2, i % 3 * 4);
            const L2 g = cmul_w<DIR>(mkl(v.x + off, v.y + off), w, k2, (1ll << 31) - fix_tie((i64)rnd()));
            e.add(g, (i128)v.x * wr - (i128)v.y * wi, (i128)v.y * wr + (i128)v.x * wi, 62 + k2);
        }
        note(e);
    }
}

template <int R, int DIR> static void rotations(long M) {
    for (int m = 1; m < R; m++) {
        int key = m * (288 / R) % 72;
        if (DIR < 0) key = (288 - m * (288 / R)) % 288 % 72;
        if (key == 0) continue;
        // the exact product with the constants that lrot uses, quadrant by quadrant
        const int q = (DIR < 0 ? 288 - m * (288 / R) : m * (288 / R)) % 288 / 72;
        const FixC c = fixcos(key), s = fixcos(72 - key);
        const i128 C = ((i128)c.add << 63) + ((i128)c.H << 32) + c.L, S = ((i128)s.add << 63) + ((i128)s.H << 32) + s.L;
        Err e;
        for (long i = 0; i < M; i++) {
            L2 v = value(63, i % 3 * 4);
            const L2 g = lrot<R, DIR>(v, m);
            for (int j = 0; j < q; j++) v = mkl(-v.y, v.x);
            e.add(g, (i128)v.x * C - (i128)v.y * S, (i128)v.y * C + (i128)v.x * S, 63);
        }
        note(e);
    }
}

int main() {
    const long M = 400000;
    products<-1>(2, M);
    products<1>(2, M);
    products<-1>(0, M);
    products<1>(0, M);
    report("cmul_w");
    rotations<16, 1>(M);
    rotations<16, -1>(M);
    rotations<9, 1>(M);
    rotations<12, -1>(M);
    report("lrot");
    Err e;
    for (long i = 0; i < M; i++) {
        const L2 v = value(63, i % 3);
        e.add(mkl(half_even(v.x), half_even(v.y)), v.x, v.y, 1);
    }
    note(e);
    report("half");
    // an offset added to input 0 of a register DFT reaches every output unchanged
    int bad = 0;
    for (int i = 0; i < 1000; i++) {
        L2 a[16], b[16];
        for (int j = 0; j < 16; j++) a[j] = b[j] = mkl(value(58, 0).x, value(58, 0).y);
        b[0] = ladd(b[0], mkl(NSK_FIX_OFF, NSK_FIX_OFF));
        L2 c[12], d[12];
        for (int j = 0; j < 12; j++) c[j] = a[j], d[j] = b[j];
        LDft<16, 1>::run(a);
        LDft<16, 1>::run(b);
        LDft<12, -1>::run(c);
        LDft<12, -1>::run(d);
        for (int j = 0; j < 16; j++) bad += b[j].x != a[j].x + NSK_FIX_OFF || b[j].y != a[j].y + NSK_FIX_OFF;
        for (int j = 0; j < 12; j++) bad += d[j].x != c[j].x + NSK_FIX_OFF || d[j].y != c[j].y + NSK_FIX_OFF;
    }
    printf("offset %d 0\n", bad);
    // doubles of any exponent: below the line's unit they are zero
    bad = 0;
    for (int e = 0; e < 2046; e++)
        for (int top = e; top < 2047; top += 1 + (top - e) / 8) {
            const int hi = (e << 20) | 0x54321;
            const i64 v = fix_from(hi, 0x9abcdef0u, top), n = fix_from(hi | (int)0x80000000, 0x9abcdef0u, top);
            const long double want = ldexpl((long double)(0x154321ll << 32 | 0x9abcdef0ll), 10 - (top - e));
            bad += v != (i64)want || n != -v;
        }
    printf("from %d 0\n", bad);
    return 0;
}
