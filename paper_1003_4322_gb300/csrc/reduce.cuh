// reduce.cuh -- deterministic FP64 reductions shared by the plain and fused
// forms: a fixed-order block tree and the shell-spectrum kernel (the
// reductions for global quantities and spectra of Sec. 3, done without
// floating-point atomics so that repeated runs agree bit for bit).
#pragma once
#include <cuda_runtime.h>

#include "grid.cuh"

namespace nsk {

// from ns_internal.h
cudaError_t allow_smem(const void *kernel, size_t bytes);

// Block tree sum of two doubles in a fixed order (deterministic).
__device__ __forceinline__ void block_sum2(double &s0, double &s1, double *sh) {
    const int t = threadIdx.x;
    sh[2 * t] = s0;
    sh[2 * t + 1] = s1;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (t < w) {
            sh[2 * t] += sh[2 * (t + w)];
            sh[2 * t + 1] += sh[2 * (t + w) + 1];
        }
        __syncthreads();
    }
    s0 = sh[0];
    s1 = sh[1];
}

// Where a step's energy and enstrophy go: ring buffer series[run][cap][2] at
// slot counter[run] % cap; ticket[run] counts the blocks that have finished.
// counter null: nothing is recorded (tuning).
struct EnergyOut {
    double *series = nullptr;
    int cap = 0;
    unsigned long long *counter = nullptr;
    unsigned *ticket = nullptr;
    int *flags = nullptr;   // bit 0: E is not finite
};

// End of a kernel whose blocks each hold a partial (e, om) in thread 0: the
// run's last block adds the nparts partials part[block][2] in a fixed order
// (independent of which block is last) and records them.  One launch less per
// step than a kernel of its own, which is 4 us of a step of 64^3 (48 us).
// Every thread of the block calls it; at least one warp.
__device__ __forceinline__ void energy_publish(double e, double om, double *part, int nparts, int run, int block,
                                               const EnergyOut &eo) {
    __shared__ unsigned last;
    if (threadIdx.x == 0) {
        part[2 * block] = e;
        part[2 * block + 1] = om;
        if (eo.counter) {
            __threadfence();
            last = atomicAdd(eo.ticket + run, 1u) == (unsigned)nparts - 1;
        } else {
            last = 0;
        }
    }
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    __threadfence();
    double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
    for (int i = threadIdx.x; i < nparts; i += 32) {
        s0 += __ldcg(part + 2 * i);
        s1 += __ldcg(part + 2 * i + 1);
    }
    for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_down_sync(0xffffffffu, s0, o);
        s1 += __shfl_down_sync(0xffffffffu, s1, o);
    }
    if (threadIdx.x == 0) {
        const unsigned long long c = eo.counter[run];
        double *sr = eo.series + 2L * run * eo.cap;
        sr[2 * (c % eo.cap)] = s0;
        sr[2 * (c % eo.cap) + 1] = s1;
        eo.counter[run] = c + 1;
        eo.ticket[run] = 0;
        if (!isfinite(s0)) atomicOr(eo.flags, 1);
    }
}

// The spectrum kernels leave partial sums after the nbins results in spec and
// ens, which hold nbins (1 + shell_parts(nbins)) doubles each; a second kernel
// adds them in a fixed order.  Up to kRowBins shells, k_shell_rows: one block
// per SM walks rows (kx, ky) and keeps a histogram per warp in shared memory.
// Beyond (boxes of extreme aspect ratio, whose histogram would not fit), the
// gather kernels: kShellParts blocks per shell look for its modes.  The
// gather reads each row once per shell it meets and finds its kz interval by
// FP64 square roots: 8.0 ms per ns_energy_spectrum at 512^3 FP64 where the rows
// take 0.90 (their FP64 arithmetic 0.35, their bytes 0.15), 21.4 ms against
// 1.14 on a 512 x 512 x 256 box in FP32.
constexpr int kShellParts = 8, kRowParts = 152, kRowBins = 4096;
inline int shell_parts(int nbins) { return nbins <= kRowBins ? kRowParts : kShellParts; }

// The largest |m| per axis that the modes of a sum reach (the rest of the
// half layout is zero).
struct Reach {
    int x, y, z;
};

// Shells of the (2 pi)^3 cube: round-half-up(|k|) from the integer |k|^2.
struct CubeShells {
    struct Row {
        int kx, ky, r2;
    };
    int n;
    __device__ Row row(int kx, int ky) const { return Row{kx, ky, kx * kx + ky * ky}; }
    __device__ double row_k2(const Row &r) const { return (double)r.r2; }
    __device__ double kz2(int z) const { return (double)(z * z); }
    __device__ int nz() const { return n; }
    __device__ int shell(const Row &r, int z, double) const {
        const int i2 = r.r2 + z * z;   // below 2^24: exact in FP32
        int K = (int)(sqrtf((float)i2) + 0.5f);
        while (K > 0 && i2 < K * K - K + 1) K--;
        while (i2 > K * K + K) K++;
        return K;
    }
    template <class Acc> __device__ double eval(const Acc &acc, const Row &r, int z) const {
        return acc(r.kx, r.ky, z);
    }
};

// Shells of any grid and box: round-half-up(|k| lmax), in FP64 with each
// operation rounded as written, so that the binning is the definition's.  An
// FP32 estimate settles the modes that are not next to a shell's edge.
struct GridShells {
    struct Row {
        int mx, my;
        double kx, ky, r2;
    };
    Grid g;
    __device__ Row row(int mx, int my) const {
        Row r{mx, my, kof(mx, g.lx), kof(my, g.ly), 0.0};
        r.r2 = __dadd_rn(__dmul_rn(r.kx, r.kx), __dmul_rn(r.ky, r.ky));
        return r;
    }
    __device__ double row_k2(const Row &r) const { return r.r2; }
    __device__ double kz2(int z) const {
        const double kz = kof(z, g.lz);
        return __dmul_rn(kz, kz);
    }
    __device__ int nz() const { return g.nz; }
    __device__ int shell(const Row &r, int, double kz2) const {
        const double k2 = __dadd_rn(r.r2, kz2);
        const float t = sqrtf((float)k2) * (float)g.lmax + 0.5f, f = floorf(t);
        const float tol = 1e-6f + 1e-6f * t;   // FP32 rounding of t: 3e-7 t at most
        if (t - f > tol && f + 1.f - t > tol) return (int)f;
        return (int)floor(__dadd_rn(__dmul_rn(__dsqrt_rn(k2), g.lmax), 0.5));
    }
    template <class Acc> __device__ double eval(const Acc &acc, const Row &r, int z) const {
        return acc(r.mx, r.my, z, r.kx, r.ky, kof(z, g.lz));
    }
};

// Bytes of shared memory of k_shell_rows: the table kz^2, then per warp the
// two histograms, the row's densities and its shells.
inline size_t shell_rows_warp_bytes(int nbins, int z) {
    return (size_t)nbins * 16 + (size_t)(z + 1) * 8 + (size_t)((z + 2 + 1) / 2) * 8;
}

// Rows (kx, ky) of the reach, one warp at a time: the lanes evaluate the row's
// modes (contiguous kz), whose shells ascend with kz; then the lane at the
// first mode of each shell adds that shell's run in order and owns its bin
// for the row.  Rows go to warps in a fixed pattern and the warps' histograms
// add up in order, so the result is deterministic.
template <class Acc, class Geo>
__global__ void k_shell_rows(Acc acc, Geo geo, Reach rc, int nbins, double *spec, double *ens) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int nzk = rc.z + 1, W = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double *kz2 = reinterpret_cast<double *>(smraw);
    const long per = 2L * nbins + nzk + (nzk + 1 + 1) / 2;   // doubles per warp
    double *he = kz2 + nzk + w * per, *ho = he + nbins, *de = ho + nbins;
    int *sh = reinterpret_cast<int *>(de + nzk);
    for (int z = threadIdx.x; z < nzk; z += blockDim.x) kz2[z] = geo.kz2(z);
    for (int k = lane; k < 2 * nbins; k += 32) he[k] = 0.0;
    __syncthreads();
    const int sy = 2 * rc.y + 1, rows = (2 * rc.x + 1) * sy;
    for (int row = blockIdx.x * W + w; row < rows; row += gridDim.x * W) {
        const int ix = row / sy;
        const typename Geo::Row r = geo.row(ix - rc.x, row - ix * sy - rc.y);
        for (int z = lane; z < nzk; z += 32) {
            const double d = geo.eval(acc, r, z);
            de[z] = z == 0 || 2 * z == geo.nz() ? 0.5 * d : d;
            sh[z] = geo.shell(r, z, kz2[z]);
        }
        if (lane == 0) sh[nzk] = -1;
        __syncwarp();
        const double k2 = geo.row_k2(r);
        for (int z = lane; z < nzk; z += 32) {
            const int K = sh[z];
            if ((z > 0 && sh[z - 1] == K) || K >= nbins) continue;
            double e = 0.0, o = 0.0;
            int j = z;
            do {
                e += de[j];
                o = fma(de[j], kz2[j], o);
                j++;
            } while (sh[j] == K);
            he[K] += e;
            ho[K] += fma(k2, e, o);
        }
        __syncwarp();
    }
    __syncthreads();
    double *h0 = kz2 + nzk;
    for (int k = threadIdx.x; k < nbins; k += blockDim.x) {
        double e = 0.0, o = 0.0;
        for (int q = 0; q < W; q++) {
            e += h0[q * per + k];
            o += h0[q * per + nbins + k];
        }
        spec[nbins + (long)blockIdx.x * nbins + k] = e;
        ens[nbins + (long)blockIdx.x * nbins + k] = o;
    }
}

// spec[K] = the sum of the blocks' partials (a warp per shell: lanes in
// strides, then a fixed tree), and ens.
static __global__ void k_rows_finish(double *spec, double *ens, int nbins, int parts) {
    const int K = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (K >= nbins) return;
    double e = 0.0, o = 0.0;
    for (int p = lane; p < parts; p += 32) {
        e += spec[nbins + (long)p * nbins + K];
        o += ens[nbins + (long)p * nbins + K];
    }
    for (int s = 16; s > 0; s >>= 1) {
        e += __shfl_down_sync(0xffffffffu, e, s);
        o += __shfl_down_sync(0xffffffffu, o, s);
    }
    if (lane == 0) {
        spec[K] = e;
        ens[K] = o;
    }
}

template <class Acc, class Geo>
static cudaError_t shell_rows(const Acc &acc, const Geo &geo, const Reach &rc, int nbins, double *spec, double *ens,
                              cudaStream_t s) {
    auto k = k_shell_rows<Acc, Geo>;
    const size_t warp = shell_rows_warp_bytes(nbins, rc.z), head = (size_t)(rc.z + 1) * 8, room = 200 * 1024;
    int W = (int)((room - head) / warp);
    W = W > 16 ? 16 : W < 1 ? 1 : W;
    const size_t smem = head + W * warp;
    cudaError_t e = allow_smem((const void *)k, smem);
    if (e != cudaSuccess) return e;
    k<<<kRowParts, 32 * W, smem, s>>>(acc, geo, rc, nbins, spec, ens);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_rows_finish<<<(nbins + 7) / 8, 256, 0, s>>>(spec, ens, nbins, kRowParts);
    return cudaGetLastError();
}

// spec[K] = the sum of the shell's kShellParts partials, in order (and ens).
static __global__ void k_shell_finish(double *spec, double *ens, int nbins) {
    const int K = blockIdx.x * blockDim.x + threadIdx.x;
    if (K >= nbins) return;
    double e = 0.0, om = 0.0;
    for (int p = 0; p < kShellParts; p++) {
        e += spec[nbins + K * kShellParts + p];
        om += ens[nbins + K * kShellParts + p];
    }
    spec[K] = e;
    ens[K] = om;
}

// Launch a shell-spectrum kernel over nbins x kShellParts blocks, then the
// ordered sum of the partials.
template <class Kernel, class... Args>
static cudaError_t shell_launch(Kernel k, int nbins, double *spec, double *ens, cudaStream_t s, Args... args) {
    k<<<dim3(nbins, kShellParts), 256, 0, s>>>(args..., spec, ens);
    k_shell_finish<<<(nbins + 255) / 256, 256, 0, s>>>(spec, ens, nbins);
    return cudaGetLastError();
}

// Re(a . conj(w)) with w = i k x a, for the helicity 1/2 <u . w>.
__device__ __forceinline__ double helicity_density(double kx, double ky, double kz, double axr,
                                                   double axi, double ayr, double ayi, double azr,
                                                   double azi) {
    // k x a
    const double cxr = ky * azr - kz * ayr, cxi = ky * azi - kz * ayi;
    const double cyr = kz * axr - kx * azr, cyi = kz * axi - kx * azi;
    const double czr = kx * ayr - ky * axr, czi = kx * ayi - ky * axi;
    // w = i (k x a) = (-ci, cr); Re(a conj w) = ar * wr + ai * wi = -ar ci + ai cr
    return -axr * cxi + axi * cxr - ayr * cyi + ayi * cyr - azr * czi + azi * czr;
}

}  // namespace nsk
