// fft_fix_strided.cuh -- the x and y passes of the FP64 transforms (1D FFTs
// along a strided axis, Sec. 2) in block fixed point (fft_fix.cuh); compiled
// for the inverse in fft_fix_inv.cu and the forward direction in fft_fix_fwd.cu.
//
// One CTA: 2^cl contiguous columns of one plane, T = n/E threads per column,
// lanes along columns (rows of 2^cl 16-byte values).
#pragma once
#include "fft_fix_line.cuh"

namespace nsk {

// What a launch passes beside its plan (FixIo, with the columns selected).
struct StridedK {
    SelK sel;
    long es, ps, ncols;
    int cl;
    FixIo io;
};

// Component d of i k x a for the curl of a column's elements: re = k2 a1.y - k1
// a2.y, im = k1 a2.x - k2 a1.x with a1, a2 the components d + 1, d + 2 (mod 3)
// and k1, k2 the same of k.  Four FP64 instructions an element, which share the
// SM with other CTAs' integer stages; a kernel of its own took 0.63 ms at
// 512^3, this pass takes 0.40 ms more than a plain one.
template <int E, int DIR, int IN, int OUT>
__global__ void __launch_bounds__(256, MinCtas<E, (DIR > 0)>::n)
k_fix_strided(const longlong2 *in, longlong2 *out, FixK pl, StridedK k) {
    grid_dep();
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned red[512];
    L2 *sm = reinterpret_cast<L2 *>(smraw);
    const SelK &sel = k.sel;
    const FixIo &io = k.io;
    const int cl = k.cl, T = pl.n / E, ct = 1 << cl;
    const int c = threadIdx.x & (ct - 1), slot = threadIdx.x >> cl;
    const bool active = slot < T;   // the CTA is rounded up to whole warps
    const int ro = blockIdx.x / sel.tpr, b = blockIdx.y;
    const int inner = (blockIdx.x - ro * sel.tpr) * ct + c;
    const long col = (long)(ro < sel.o1 ? ro : ro - sel.o1 + sel.o2) * sel.inner + inner;
    const bool valid = active && inner < sel.keep;
    const bool plain = IN != kIoCurl || (io.both && b < 3);
    const int d = IN == kIoCurl && b >= 3 ? b - 3 : b;   // component of the curl
    const longlong2 *src = in + (plain ? b * k.ps : 0) + col;
    longlong2 *dst = out + b * k.ps + col;
    auto in_gap = [&](int e) { return e >= sel.gap_lo && e < sel.gap_hi; };
    // elements q T .. (q + 1) T - 1 all in the gap: zeros that need no work
    auto skip = [&](int q) { return DIR > 0 && q * T >= sel.gap_lo && (q + 1) * T <= sel.gap_hi; };
    const int yi = IN == kIoDouble ? 0 : (int)(col / io.nzh), kz = IN == kIoDouble ? 0 : (int)(col - (long)yi * io.nzh);
    long o1 = 0, o2 = 0;
    double k1 = 0.0, k2 = 0.0;
    if constexpr (IN == kIoCurl) {
        o1 = (d + 1) % 3 * k.ps;
        o2 = (d + 2) % 3 * k.ps;
        const double ky = io.iy * (2 * yi < io.ny ? yi : yi - io.ny), kzz = io.iz * kz;
        k1 = d == 0 ? ky : kzz;   // d = 1: k2, d = 2: k1 are k_x, which varies along the line
        k2 = d == 0 ? kzz : ky;
    }
    const long gstep = T * k.es;   // element slot + q T: q steps on
    const int *tin = nullptr;
    int tstep = 0;
    if constexpr (IN == kIoFixed) {
        tin = io.tin + (b / io.pdiv) * io.eps + (io.ecol ? kz : 0) + (long)slot * io.estride;
        tstep = T * io.estride;
    }
    src += slot * k.es;
    L2 v[E];
    int t[E];
#pragma unroll
    for (int q = 0; q < E; q++) {
        const int e = slot + q * T;
        v[q] = mkl(0, 0);
        t[q] = kZeroT;
        if (!skip(q) && valid && (DIR < 0 || !in_gap(e))) {
            if (!plain) {
                const double2 a1 = reinterpret_cast<const double2 *>(src)[o1];
                const double2 a2 = reinterpret_cast<const double2 *>(src)[o2];
                const double kx = io.ix * (2 * e < pl.n ? e : e - pl.n);
                const double p1 = d == 2 ? kx : k1, p2 = d == 1 ? kx : k2;
                v[q] = mkl(__double_as_longlong(p2 * a1.y - p1 * a2.y),
                           __double_as_longlong(p1 * a2.x - p2 * a1.x));
            } else {
                const longlong2 x = *src;
                v[q] = mkl(x.x, x.y);
                if constexpr (IN == kIoFixed) t[q] = *tin;
            }
        }
        src += gstep;
        tin += tstep;
    }
    LineGeo g{kCols, cl, 0, c};
    int tl;
    if constexpr (IN == kIoFixed) {
        tl = line_scale_fixed<E, false>(v, t, g, red, fix_room(pl), skip);
    } else {
        const LineScale sc = line_scale<E, false>(v, g, red, fix_room(pl), skip);
#pragma unroll
        for (int q = 0; q < E; q++)
            if (!skip(q)) v[q] = fix_from_raw(v[q], sc.top);
        tl = sc.t;
    }
    const LineAt<E> ln{sm + c, cl};
    fix_line<E, DIR>(v, active, slot, T, pl, false, ln);
    if (!valid) return;
    tl += pl.nst > 1 ? 2 : 0;
    if (OUT == kIoFixed && slot == 0) io.tout[b * k.ncols + col] = tl;
    if constexpr (OUT == kIoDouble) FixOut(tl).run(v);
    dst += slot * k.es;
#pragma unroll
    for (int q = 0; q < E; q++) {
        if (DIR > 0 || !in_gap(slot + q * T)) *dst = longlong2{v[q].x, v[q].y};
        dst += gstep;
    }
}

template <int DIR, int IN, int OUT> const void *fix_kernel_of(int E) {
    switch (E) {
    case 4: return (const void *)k_fix_strided<4, DIR, IN, OUT>;
    case 6: return (const void *)k_fix_strided<6, DIR, IN, OUT>;
    case 8: return (const void *)k_fix_strided<8, DIR, IN, OUT>;
    case 9: return (const void *)k_fix_strided<9, DIR, IN, OUT>;
    case 12: return (const void *)k_fix_strided<12, DIR, IN, OUT>;
    case 16: return (const void *)k_fix_strided<16, DIR, IN, OUT>;
    }
    return nullptr;
}

// The kernels of a direction by input and output (nullptr: no such pass).
const void *fix_inv_kernel(int E, int in, int out);
const void *fix_fwd_kernel(int E, int in, int out);

}  // namespace nsk
