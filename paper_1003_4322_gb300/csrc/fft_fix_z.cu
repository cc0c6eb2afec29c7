// fft_fix_z.cu -- the z passes of the FP64 transforms (real lines, Sec. 2,
// Fig. 1) in block fixed point (fft_fix.cuh): lines 2p and 2p + 1 through one
// complex transform of length N.
//  c2r: Z[k] = X1[k] + i X2[k] and Z[N-k] = conj X1[k] + i conj X2[k] from the
//       half spectra (imaginary parts of X[0] and X[N/2] dropped); the inverse
//       transform of Z is x1 + i x2.
//  r2c: the transform Z of x1 + i x2 gives X1[k] = (Z[k] + conj Z[N-k]) / 2
//       and X2[k] = (Z[k] - conj Z[N-k]) / 2i.
// The pairing adds are fixed-point too, and c2r converts each loaded entry
// once for both of its places.  The spectra are in fixed point with their
// lines' exponents.  Entries kz >= kzk are not read (c2r) or not
// written (r2c).
#include "fft_fix_line.cuh"

namespace nsk {

// One CTA holds lb line pairs, T = N/E threads each.
NSK_DEV LineGeo z_geo(int T, int li) {
    if (T <= 32 && (T & (T - 1)) == 0) return LineGeo{kSub, 31 - __clz(T), 0, li};
    if (T % 32 == 0) return LineGeo{kWarps, 0, T / 32, li};
    return LineGeo{kAny, 0, T, li};
}

// r2c's input: one field, or the products of the nonlinear term formed from
// the fields as they are loaded (component c of f0 x f1, or of f0 x f1 + f2 x f3,
// with f_i = 3 fields of V points).  A pass of products alone runs at the FP64
// pipe's limit (two instructions a value: 1.45 ms at 512^3) while the
// transform leaves that pipe idle; together they took 2.84 ms where the two took
// 3.65 (2.54 with the spectra in fixed point).  The lines of a product's three components go to neighbouring
// transforms, whose loads of the same lines meet in L1 and L2.
template <int KIND>
NSK_DEV double product_at(const FixProduct &f, long base, long o1, long o2, int e) {
    // o1, o2: offsets of the components (c + 1) % 3 and (c + 2) % 3
    const long i = base + e;
    if constexpr (KIND == 0) return f.f[0][i];
    double t = f.f[0][o1 + i] * f.f[1][o2 + i] - f.f[0][o2 + i] * f.f[1][o1 + i];
    if constexpr (KIND == 2) t += f.f[2][o1 + i] * f.f[3][o2 + i] - f.f[2][o2 + i] * f.f[3][o1 + i];
    return t;
}

template <int E, int KIND>
__global__ void __launch_bounds__(256, MinCtas<E, true>::n)
k_fix_r2c2(FixProduct in, longlong2 *__restrict__ out, int *__restrict__ tout, int N, long nlines, FixK pl, int kzk) {
    grid_dep();
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned red[512];
    const int nh = N / 2, T = N / E;
    const int slot = threadIdx.x % T, li = threadIdx.x / T, lb = blockDim.x / T;
    // products: pairs of lines of the components in turn (the lines of one
    // component are even in number)
    long pair = (long)blockIdx.x * lb + li, base = 0, o1 = 0, o2 = 0;
    if constexpr (KIND > 0) {
        const int c = (int)(pair % 3);
        base = 2 * (pair / 3) * N;
        o1 = (c + 1) % 3 * in.V;
        o2 = (c + 2) % 3 * in.V;
        pair = c * (nlines / 6) + pair / 3;
    } else {
        base = 2 * pair * N;
    }
    const long l1 = 2 * pair, l2 = l1 + 1;
    const bool valid = (long)blockIdx.x * lb + li < nlines / 2;
    const LineAt<E> ln{reinterpret_cast<L2 *>(smraw) + li * (N + T), 0};
    L2 v[E];
#pragma unroll
    for (int q = 0; q < E; q++) {
        const int e = slot + q * T;
        v[q] = mkl(valid ? __double_as_longlong(product_at<KIND>(in, base, o1, o2, e)) : 0,
                   valid ? __double_as_longlong(product_at<KIND>(in, base + N, o1, o2, e)) : 0);
    }
    const LineScale sc = line_scale<E, false>(v, z_geo(T, li), red, fix_room(pl), [](int) { return false; });
#pragma unroll
    for (int q = 0; q < E; q++) v[q] = fix_from_raw(v[q], sc.top);
    fix_line<E, -1>(v, true, slot, T, pl, false, ln);
    if (pl.nst > 1) __syncthreads();
#pragma unroll
    for (int q = 0; q < E; q++) *ln.at(slot + q * T) = v[q];
    __syncthreads();
    if (!valid) return;
    longlong2 *d1 = out + l1 * (nh + 1), *d2 = out + l2 * (nh + 1);
    // the halves of the pairing fall to the exponent
    if (slot < 2) tout[l1 + slot] = sc.t + (pl.nst > 1 ? 1 : -1);
    if (T == 1) tout[l2] = sc.t + (pl.nst > 1 ? 1 : -1);
    for (int k = slot; k <= nh && k < kzk; k += T) {
        const L2 a = *ln.at(k), b = *ln.at(k == 0 ? 0 : N - k);
        d1[k] = longlong2{a.x + b.x, a.y - b.y};
        d2[k] = longlong2{a.y + b.y, b.x - a.x};
    }
}

template <int E>
__global__ void __launch_bounds__(256, MinCtas<E, false>::n)
k_fix_c2r2(const longlong2 *__restrict__ in, const int *__restrict__ tin, int ny, double *__restrict__ out, int N,
           long nlines, FixK pl, int kzk) {
    grid_dep();
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned red[512];
    const int nh = N / 2, T = N / E;
    const int slot = threadIdx.x % T, li = threadIdx.x / T, lb = blockDim.x / T;
    const long l1 = 2 * ((long)blockIdx.x * lb + li), l2 = l1 + 1;
    const bool valid = l1 < nlines;
    const LineAt<E> ln{reinterpret_cast<L2 *>(smraw) + li * (N + T), 0};
    const longlong2 *s1 = in + l1 * (nh + 1), *s2 = in + l2 * (nh + 1);
    // the thread's entries m = slot + j T <= N/2 of both spectra
    constexpr int H = E / 2 + 1;
    const int top_m = kzk <= nh ? kzk : nh + 1;
    const int *tl = tin + l1 / ny * (nh + 1);
    L2 w[2 * H];
    int t[2 * H];
#pragma unroll
    for (int j = 0; j < H; j++) {
        const int m = slot + j * T;
        longlong2 a{0, 0}, b{0, 0};
        t[2 * j] = kZeroT;
        if (j * T < top_m && m < top_m && valid) {
            a = s1[m];
            b = s2[m];
            t[2 * j] = tl[m];
        }
        t[2 * j + 1] = t[2 * j];
        if (m == 0 || m == nh) a.y = b.y = 0;
        w[2 * j] = mkl(a.x, a.y);
        w[2 * j + 1] = mkl(b.x, b.y);
    }
    const int tz =
        line_scale_fixed<2 * H, true>(w, t, z_geo(T, li), red, fix_room(pl), [&](int i) { return (i / 2) * T >= top_m; });
#pragma unroll
    for (int j = 0; j < H; j++) {
        const int m = slot + j * T;
        if (m < top_m) {
            const L2 a = w[2 * j], b = w[2 * j + 1];
            *ln.at(m) = mkl(a.x - b.y, a.y + b.x);
            if (m != 0 && m != nh) *ln.at(N - m) = mkl(a.x + b.y, b.x - a.y);
        }
    }
    __syncthreads();
    L2 v[E];
#pragma unroll
    for (int q = 0; q < E; q++) {
        const int e = slot + q * T;
        v[q] = e < top_m || N - e < top_m ? *ln.at(e) : mkl(0, 0);
    }
    double *d1 = out + l1 * N, *d2 = out + l2 * N;
    fix_line<E, 1>(v, true, slot, T, pl, true, ln);
    if (!valid) return;
    FixOut(tz + (pl.nst > 1 ? 2 : 0)).run(v);
#pragma unroll
    for (int q = 0; q < E; q++) {
        const int e = slot + q * T;
        d1[e] = __longlong_as_double(v[q].x);
        d2[e] = __longlong_as_double(v[q].y);
    }
}

// Threads per CTA (one line pair at least).  Smaller CTAs drift apart, so that
// one's FP64 products and another's integer stages share an SM: 256 threads
// took 3.25 ms for the product pass at 512^3, 128 2.84, 64 2.76 but more elsewhere
// (c2r 2.36 / 2.26 / 2.28; all with the spectra as doubles).
static const int kThreads = 128;

// kind: -1 c2r, else the r2c of that kind of input.
static const void *kernel_of(int kind, int E) {
#define NSK_FZ(EE)                                                                                    \
    case EE:                                                                                          \
        return kind < 0 ? (const void *)k_fix_c2r2<EE> : kind == 0 ? (const void *)k_fix_r2c2<EE, 0>  \
             : kind == 1 ? (const void *)k_fix_r2c2<EE, 1> : (const void *)k_fix_r2c2<EE, 2>;
    switch (E) {
        NSK_FZ(4)
        NSK_FZ(6)
        NSK_FZ(8)
        NSK_FZ(9)
        NSK_FZ(12)
        NSK_FZ(16)
    }
#undef NSK_FZ
    return nullptr;
}

cudaError_t prepare_fix_z() {
    for (int E : {4, 6, 8, 9, 12, 16})
        for (int kind = -1; kind <= 2; kind++) {
            cudaError_t e = allow_smem(kernel_of(kind, E), 48 * 1024 + 1);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

static cudaError_t launch(int kind, void **args, int N, long *nlines, const FixPlan &fp, cudaStream_t s) {
    const Plan &pl = fp.pl;
    const void *k = kernel_of(kind, pl.E);
    if (!k || !fp.tab || pl.n != N || *nlines < 2 || *nlines % 2 || (kind > 0 && *nlines % 6))
        return cudaErrorInvalidValue;
    const int T = N / pl.E, lb = T > kThreads ? 1 : kThreads / T;
    if (T > 256) return cudaErrorInvalidValue;
    const size_t smem = (size_t)lb * (N + T) * sizeof(L2);   // LineAt
    cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    const long blocks = (*nlines / 2 + lb - 1) / lb;
    if (blocks > 0x7fffffffL) return cudaErrorInvalidValue;
    return launch_dep(k, dim3((unsigned)blocks), dim3(lb * T), args, smem, s);
}

cudaError_t fix_z_r2c(const FixProduct &in, void *out, int *tout, int N, long nlines, const FixPlan &fp,
                      cudaStream_t s, int kzk) {
    if (kzk < 0 || kzk > N / 2 + 1) kzk = N / 2 + 1;   // every entry
    FixK kp{fp.pl.n, fp.pl.nst, fp.pl.radix, fp.tab};
    void *args[] = {(void *)&in, (void *)&out, (void *)&tout, (void *)&N, (void *)&nlines, (void *)&kp, (void *)&kzk};
    return launch(in.kind, args, N, &nlines, fp, s);
}
cudaError_t fix_z_c2r(const void *in, const int *tin, int ny, double *out, int N, long nlines, const FixPlan &fp,
                      cudaStream_t s, int kzk) {
    if (ny < 2 || ny % 2) return cudaErrorInvalidValue;
    if (kzk < 0 || kzk > N / 2 + 1) kzk = N / 2 + 1;
    FixK kp{fp.pl.n, fp.pl.nst, fp.pl.radix, fp.tab};
    void *args[] = {(void *)&in, (void *)&tin, (void *)&ny, (void *)&out, (void *)&N, (void *)&nlines, (void *)&kp,
                    (void *)&kzk};
    return launch(-1, args, N, &nlines, fp, s);
}

}  // namespace nsk
