// fft_fix_inv.cu -- the inverse x and y passes of the FP64 transforms, and the
// launcher of both directions (kernel: fft_fix_strided.cuh).
#include "fft_fix_strided.cuh"

namespace nsk {

// Doubles on both sides go with the one-line z passes: those NS_PLAIN_Z=1 asks for,
// and those of standalone transforms without a buffer for line exponents.
const void *fix_inv_kernel(int E, int in, int out) {
    if (in == kIoFixed) return out == kIoFixed ? fix_kernel_of<1, kIoFixed, kIoFixed>(E) : nullptr;
    if (in == kIoCurl) return out == kIoFixed ? fix_kernel_of<1, kIoCurl, kIoFixed>(E) : nullptr;
    return out == kIoFixed ? fix_kernel_of<1, kIoDouble, kIoFixed>(E) : fix_kernel_of<1, kIoDouble, kIoDouble>(E);
}

cudaError_t prepare_fix_strided() {
    for (int E : {4, 6, 8, 9, 12, 16})
        for (int in : {kIoDouble, kIoCurl, kIoFixed})
            for (int out : {kIoDouble, kIoFixed})
                for (const void *k : {fix_inv_kernel(E, in, out), fix_fwd_kernel(E, in, out)}) {
                    const cudaError_t e = k ? allow_smem(k, 48 * 1024 + 1) : cudaSuccess;
                    if (e != cudaSuccess) return e;
                }
    return cudaSuccess;
}

int fix_threads(int n, int E, int ct) { return (n / E * ct + 31) / 32 * 32; }

cudaError_t fix_strided(const void *in, void *out, long ncols, long es, long ps, int planes, int dir,
                        const FixPlan &fp, int ct, cudaStream_t s, const StridedSel *sel, const FixIo &io) {
    const Plan &pl = fp.pl;
    const void *k = dir < 0 ? fix_fwd_kernel(pl.E, io.in, io.out) : fix_inv_kernel(pl.E, io.in, io.out);
    int cl = 0;
    while ((1 << cl) < ct) cl++;
    const int threads = fix_threads(pl.n, pl.E, ct);
    if (!k || !fp.tab || (1 << cl) != ct || ct > 32 || threads > 256) return cudaErrorInvalidValue;
    if ((io.in == kIoFixed && !io.tin) || (io.out == kIoFixed && !io.tout) || io.nzh < 1 || io.pdiv < 1 ||
        (io.in == kIoCurl && planes != (io.both ? 6 : 3)))
        return cudaErrorInvalidValue;
    StridedK sk{SelK{}, es, ps, ncols, cl, io};
    unsigned tiles;
    cudaError_t e = strided_selection(ncols, planes, pl.n, ct, sel, &sk.sel, &tiles);
    if (e != cudaSuccess || tiles == 0) return e;
    const size_t smem = (size_t)(pl.n + pl.n / pl.E) * ct * sizeof(L2);   // LineAt
    if ((e = allow_smem(k, smem)) != cudaSuccess) return e;
    FixK kp{pl.n, pl.nst, pl.radix, fp.tab};
    void *args[] = {(void *)&in, (void *)&out, (void *)&kp, (void *)&sk};
    return launch_dep(k, dim3(tiles, (unsigned)planes), dim3(threads), args, smem, s);
}

}  // namespace nsk
