// fft_fix_strided.cu -- the x and y passes of the FP64 transforms (1D FFTs
// along a strided axis, Sec. 2) in block fixed point (fft_fix.cuh).
//
// One CTA: 2^cl contiguous columns of one plane, T = n/E threads per column,
// lanes along columns (rows of 2^cl 16-byte values); the exchange tile
// holds element (e, c) at (e + (e >> SK)) 2^cl + c, one row of padding every E
// elements, so that the stride-E stores of stage 0 spread over the banks.
#include "fft_fix_line.cuh"

namespace nsk {

// Component d of i k x a for the curl of a column's elements (input KIND 1:
// the x pass of a vorticity, planes = components, from the velocity's three
// fields M apart): re = k2 a1.y - k1 a2.y, im = k1 a2.x - k2 a1.x with a1, a2 the
// components d + 1, d + 2 (mod 3) and k1, k2 the same of k.  Four FP64
// instructions an element, which share the SM with other CTAs' integer stages;
// a kernel of its own took 0.63 ms at 512^3, this pass takes 0.40 ms more than a plain one.

template <int E> struct SkewE { enum { shift = E == 4 ? 2 : E == 16 ? 4 : 3 }; };

template <int E, int DIR, int KIND>
__global__ void __launch_bounds__(256, MinCtas<E>::n)
k_fix_strided(const longlong2 *in, longlong2 *out, SelK sel, long es, long ps_in, long ps_out, FixK pl, int cl,
              FixCurl cu) {
    grid_dep();
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned red[256];
    L2 *sm = reinterpret_cast<L2 *>(smraw);
    const int T = pl.n / E, ct = 1 << cl;
    const int c = threadIdx.x & (ct - 1), slot = threadIdx.x >> cl;
    const bool active = slot < T;   // the CTA is rounded up to whole warps
    const int ro = blockIdx.x / sel.tpr;
    const long inner = (long)(blockIdx.x - ro * sel.tpr) * ct + c;
    const long col = (long)(ro < sel.o1 ? ro : ro - sel.o1 + sel.o2) * sel.inner + inner;
    const bool valid = active && inner < sel.keep;
    const longlong2 *src = in + (KIND == 1 ? 0 : (long)blockIdx.y * ps_in) + col;
    longlong2 *dst = out + (long)blockIdx.y * ps_out + col;
    auto in_gap = [&](int e) { return e >= sel.gap_lo && e < sel.gap_hi; };
    // elements q T .. (q + 1) T - 1 all in the gap: zeros that need no work
    auto skip = [&](int q) { return DIR > 0 && q * T >= sel.gap_lo && (q + 1) * T <= sel.gap_hi; };
    const int d = blockIdx.y;
    long o1 = 0, o2 = 0;
    double k1 = 0.0, k2 = 0.0;
    if constexpr (KIND == 1) {
        o1 = (d + 1) % 3 * ps_in;
        o2 = (d + 2) % 3 * ps_in;
        const int yi = (int)(col / cu.nz), zi = (int)(col - (long)yi * cu.nz);
        const double ky = cu.iy * (2 * yi < cu.ny ? yi : yi - cu.ny), kz = cu.iz * zi;
        k1 = d == 0 ? ky : kz;   // d = 1: k2, d = 2: k1 are k_x, which varies along the line
        k2 = d == 0 ? kz : ky;
    }
    L2 v[E];
#pragma unroll
    for (int q = 0; q < E; q++) {
        const int e = slot + q * T;
        v[q] = mkl(0, 0);
        if (skip(q)) continue;
        if (valid && (DIR < 0 || !in_gap(e))) {
            if constexpr (KIND == 1) {
                const double2 a1 = reinterpret_cast<const double2 *>(src)[o1 + e * es];
                const double2 a2 = reinterpret_cast<const double2 *>(src)[o2 + e * es];
                const double kx = cu.ix * (2 * e < pl.n ? e : e - pl.n);
                const double p1 = d == 2 ? kx : k1, p2 = d == 1 ? kx : k2;
                v[q] = mkl(__double_as_longlong(p2 * a1.y - p1 * a2.y),
                           __double_as_longlong(p1 * a2.x - p2 * a1.x));
            } else {
                const longlong2 t = src[e * es];
                v[q] = mkl(t.x, t.y);
            }
        }
    }
    LineGeo g{kCols, cl, 0, c};
    const LineScale sc = line_scale<E, false>(v, g, red, skip);
#pragma unroll
    for (int q = 0; q < E; q++)
        if (!skip(q)) v[q] = fix_from_raw(v[q], sc.top);
    auto at = [&](int e) { return ((e + (e >> SkewE<E>::shift)) << cl) + c; };
    auto sl = [&](int e) { return sm[at(e)]; };
    auto ss = [&](int e, L2 x) { sm[at(e)] = x; };
    fix_line<E, DIR>(v, active, slot, T, pl, false, sl, ss);
    if (!valid) return;
    const FixOut fo{sc.top + 1 + (pl.nst > 1 ? 2 : 0)};
#pragma unroll
    for (int q = 0; q < E; q++) {
        const int e = slot + q * T;
        if (DIR < 0 && in_gap(e)) continue;
        double2 d = make_double2(fo(v[q].x), fo(v[q].y));
        if (sc.any) d = make_double2(d.x * sc.mul, d.y * sc.mul);
        reinterpret_cast<double2 *>(dst)[e * es] = d;
    }
}

template <int DIR, int KIND> static const void *kernel_of(int E) {
    switch (E) {
    case 4: return (const void *)k_fix_strided<4, DIR, KIND>;
    case 6: return (const void *)k_fix_strided<6, DIR, KIND>;
    case 8: return (const void *)k_fix_strided<8, DIR, KIND>;
    case 9: return (const void *)k_fix_strided<9, DIR, KIND>;
    case 12: return (const void *)k_fix_strided<12, DIR, KIND>;
    case 16: return (const void *)k_fix_strided<16, DIR, KIND>;
    }
    return nullptr;
}

cudaError_t prepare_fix_strided() {
    for (int E : {4, 6, 8, 9, 12, 16})
        for (const void *k : {kernel_of<-1, 0>(E), kernel_of<1, 0>(E), kernel_of<1, 1>(E)}) {
            cudaError_t e = allow_smem(k, 48 * 1024 + 1);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

int fix_threads(int n, int E, int ct) { return (n / E * ct + 31) / 32 * 32; }

cudaError_t fix_strided(const double2 *in, double2 *out, long ncols, long es, long ps_in, long ps_out, int planes,
                        int dir, const FixPlan &fp, int ct, cudaStream_t s, const StridedSel *sel,
                        const FixCurl *curl) {
    const Plan &pl = fp.pl;
    const void *k = dir < 0 ? kernel_of<-1, 0>(pl.E) : curl ? kernel_of<1, 1>(pl.E) : kernel_of<1, 0>(pl.E);
    int cl = 0;
    while ((1 << cl) < ct) cl++;
    const int threads = fix_threads(pl.n, pl.E, ct);
    if (curl && (dir < 0 || planes != 3)) return cudaErrorInvalidValue;
    if (!k || !fp.tab || (1 << cl) != ct || ct > 32 || threads > 256) return cudaErrorInvalidValue;
    SelK sk;
    unsigned nx;
    cudaError_t e = strided_selection(ncols, planes, pl.n, ct, sel, &sk, &nx);
    if (e != cudaSuccess || nx == 0) return e;
    const size_t smem = (size_t)(pl.n + pl.n / 4 + 1) * ct * sizeof(L2);
    if ((e = allow_smem(k, smem)) != cudaSuccess) return e;
    FixK kp{pl.n, pl.nst, pl.radix, fp.tab};
    FixCurl cu = curl ? *curl : FixCurl{};
    void *args[] = {(void *)&in, (void *)&out, (void *)&sk, (void *)&es, (void *)&ps_in, (void *)&ps_out,
                    (void *)&kp, (void *)&cl, (void *)&cu};
    return launch_dep(k, dim3(nx, (unsigned)planes), dim3(threads), args, smem, s);
}

}  // namespace nsk
