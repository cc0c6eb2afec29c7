// ns_internal.h -- host-side declarations shared by the translation units of
// libns (not part of the public ABI, which is include/ns.h).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "fft_core.cuh"

namespace nsk {

// Optional per-launch timing: when a Tracer is active, every kernel launch of
// a step is bracketed by a pair of CUDA events on the launching stream.
struct Tracer {
    struct Rec {
        const char *name;
        cudaEvent_t a, b;
    };
    cudaStream_t s = nullptr;
    std::vector<Rec> recs;
    std::vector<cudaEvent_t> pool;
    size_t used = 0;
    cudaError_t err = cudaSuccess;
    cudaEvent_t take() {
        if (used == pool.size()) {
            cudaEvent_t e;
            cudaError_t r = cudaEventCreate(&e);
            if (r != cudaSuccess) {
                err = r;
                return nullptr;
            }
            pool.push_back(e);
        }
        return pool[used++];
    }
    void begin(const char *name) {
        Rec r{name, take(), nullptr};
        if (r.a) cudaEventRecord(r.a, s);
        recs.push_back(r);
    }
    void end() {
        cudaEvent_t b = take();
        if (b) cudaEventRecord(b, s);
        recs.back().b = b;
    }
    ~Tracer() {
        for (cudaEvent_t e : pool) cudaEventDestroy(e);
    }
};

// Run one launch expression, timed when tr is non-null; yields its error.
#define NSK_TIMED(tr, name, expr)                         \
    ([&]() -> cudaError_t {                               \
        if (tr) (tr)->begin(name);                        \
        cudaError_t _te = (expr);                         \
        if (tr) (tr)->end();                              \
        return _te;                                       \
    }())

// Standalone FP32 transforms of an nx x ny x nz grid on the compile-time
// kernels (axis lengths 64 ... 1024 of the compiled set), with the twiddle
// table exp(-2 pi i t / n_i) of every axis: r2c of ncomp real fields into the
// half layout, c2r of one half field through tmp (one half field).  False
// when a length has no compiled kernel (nothing launched); else *err holds
// the launch status.
struct StdGrid {
    int nx, ny, nz;
    const float2 *twx, *twy, *twz;
};
bool std_r2c_fp32_grid(const float *in, float2 *out, const StdGrid &g, int ncomp, cudaStream_t s,
                       cudaError_t *err);
bool std_c2r_fp32_grid(const float2 *in, float2 *tmp, float *out, const StdGrid &g, cudaStream_t s,
                       cudaError_t *err);

// Radix plan for a line of length n = 2^a 3^b (false if n has another factor).
bool make_plan(int n, Plan *pl);

// Radix plan with E elements per thread (the first, largest radix is E and
// every radix divides E); false if E does not suit n.
bool make_plan_e(int n, int E, Plan *pl);

// Is N a supported grid size (2^a 3^b, even, >= 8)?
bool supported_n(int n);

// Twiddle table exp(-2 pi i t / n), t < n, computed on the host in FP64,
// rounded once to float and uploaded.
float2 *make_twiddles(int n, cudaError_t *err);

// A subset of the columns and rows of a strided pass: the lines that the
// dealiasing rule leaves zero (inverse) or whose result it discards
// (forward).  A plane's ncols columns are nouter rows of `inner` columns
// (inner x nouter = ncols); the pass transforms the first `keep` columns of
// rows [0, o1) and [o2, nouter), and treats the elements e of the transform
// axis in [gap_lo, gap_hi) as zero on input (dir +1) or leaves them
// unwritten (dir -1).  The other columns are neither read nor written.
struct StridedSel {
    long inner = 0;
    int keep = 0, nouter = 1, o1 = 1, o2 = 1;
    int gap_lo = 0, gap_hi = 0;
};

// The same as the kernels see it: tpr tiles of ct columns per row.
struct SelK {
    long inner;
    int keep, tpr, o1, o2, gap_lo, gap_hi;
};
// Checks a selection (nullptr: all ncols columns) of a strided pass of length
// n over `planes` planes and forms *sk and the CTAs per plane (0: nothing
// selected).
cudaError_t strided_selection(long ncols, int planes, int n, int ct, const StridedSel *sel, SelK *sk,
                              unsigned *tiles);

// Batched FFT along a strided axis.  Element e (< pl.n) of column c (< ncols)
// of plane b (< planes) sits at base + b * plane_stride + e * es + c (in
// complex units); columns are contiguous.  dir = -1 forward, +1 inverse.
// in == out is allowed (in place).  ct = columns per CTA.  sel (optional):
// only the selected columns and rows.
template <typename T>
cudaError_t fft_strided(const typename Cx<T>::type *in, typename Cx<T>::type *out, long ncols,
                        long es, long ps_in, long ps_out, int planes, int dir, const Plan &pl,
                        const typename Cx<T>::type *tw, int ntab, int ct, cudaStream_t s,
                        const StridedSel *sel = nullptr);

// Real-to-complex transform along z (contiguous) of nlines lines of N reals
// into nlines lines of N/2+1 complex values; pl is the plan of length N/2 (one
// line per transform) or N (two), tw the table of length N.  kzk in
// [0, N/2+1]: only the entries kz < kzk are written (-1: all).
template <typename T>
cudaError_t fft_z_r2c(const T *in, typename Cx<T>::type *out, int N, long nlines, const Plan &pl,
                      const typename Cx<T>::type *tw, cudaStream_t s, int kzk = -1);

// Complex-to-real transform along z: nlines lines of N/2+1 complex values into
// nlines lines of N reals (real parts of the kz = 0 and N/2 entries only).
// kzk: the entries kz >= kzk are taken as zero and not read (-1: all read).
template <typename T>
cudaError_t fft_z_c2r(const typename Cx<T>::type *in, T *out, int N, long nlines,
                      const Plan &pl, const typename Cx<T>::type *tw, cudaStream_t s, int kzk = -1);

// Columns per CTA of the FP32 strided pass for a length.
int default_ct(int n);

// A plan of the FP64 transforms with its stage twiddles on the device, in the
// fixed-point format of fft_fix.cuh.
struct FixPlan {
    Plan pl{};
    const int4 *tab = nullptr;
};
// The stage twiddles of length n for every E that suits it, in one device
// array: tab[E] points at those of make_plan_e(n, E) (nullptr: no such plan), *tw
// at a table of the n doubles exp(-2 pi i t / n).  *buf receives the array
// (freed with dev_free).
cudaError_t make_fix_tables(int n, int4 **buf, const int4 *tab[17], void **tw);

// The FP64 passes (fft_fix_strided.cuh, fft_fix_z.cu).  Arrays of complex
// values hold doubles, or fixed-point integers in the same 16 bytes with one
// exponent per line in an array of their own.
enum { kIoDouble = 0, kIoCurl = 1, kIoFixed = 2 };
// Input and output of a strided pass.  Input exponents: those of the lines
// that the pass before went along; element e of column (.., kz) of plane b
// belongs to tin[(b / pdiv) eps + e estride + (ecol ? kz : 0)], kz = column mod
// nzh.  Output exponents: tout[b ncols + column].
// kIoCurl (x pass, dir +1, planes = the 3 components, ps apart): transforms
// i k x a of the doubles a, formed on load; the plane is ny rows of nzh columns
// and ix, iy, iz are the wavenumbers per index.  both: planes 0 .. 2 transform a
// itself, planes 3 .. 5 its curl.
struct FixIo {
    int in = kIoDouble, out = kIoDouble;
    const int *tin = nullptr;
    int *tout = nullptr;
    int pdiv = 1, estride = 0, ecol = 0, nzh = 1, both = 0;
    long eps = 0;
    int ny = 0;
    double ix = 1.0, iy = 1.0, iz = 1.0;
};
// Arguments as those of fft_strided.  ct: a power of two up to 32,
// fix_threads(n, E, ct) <= 256.
int fix_threads(int n, int E, int ct);
cudaError_t fix_strided(const void *in, void *out, long ncols, long es, long ps, int planes, int dir,
                        const FixPlan &fp, int ct, cudaStream_t s, const StridedSel *sel, const FixIo &io);
// The input of the r2c pass: f[0] (kind 0), or products of 3-component fields of
// V points each, formed on load: f[0] x f[1] (kind 1), f[0] x f[1] + f[2] x f[3]
// (kind 2; nlines then covers the three components, a multiple of 6).
struct FixProduct {
    const double *f[4] = {nullptr, nullptr, nullptr, nullptr};
    long V = 0;
    int kind = 0;
};
// As fft_z_r2c and fft_z_c2r, with plans of length N (two lines, of the same x,
// per transform; an even number of lines).  The spectra are in fixed point:
// r2c writes the exponent of every line to tout[line]; c2r reads that of
// entry kz of a line from tin[(line / ny) (N/2 + 1) + kz].
cudaError_t fix_z_r2c(const FixProduct &in, void *out, int *tout, int N, long nlines, const FixPlan &fp,
                      cudaStream_t s, int kzk = -1);
cudaError_t fix_z_c2r(const void *in, const int *tin, int ny, double *out, int N, long nlines, const FixPlan &fp,
                      cudaStream_t s, int kzk = -1);
cudaError_t prepare_fix_strided();
cudaError_t prepare_fix_z();

// Opt a kernel into more than 48 KB of dynamic shared memory (once per
// device); fails if bytes exceeds the device's opt-in maximum.
cudaError_t allow_smem(const void *kernel, size_t bytes);
// The library's device allocations (devmem.cu): plain cudaMalloc, or with
// guard bands when NS_GUARD=1.
cudaError_t dev_malloc(void **p, size_t bytes);
void dev_free(void *p);
bool dev_guards();
// A context's error word: zeroed host memory that kernels write through *dev.
// Given back (nullptr is accepted) when nothing that could write it is queued.
cudaError_t error_word_take(int **host, int **dev);
void error_word_give(int *host);

// Launch a kernel that begins with grid_dep(): it may become resident while
// the kernel ahead of it in the stream drains (a programmatic dependency),
// which hides the launch latency between a transform's small passes: 18.4 ->
// 12.0 us for ns_fft_c2r_noalloc on three components of 64^3, 147 -> 126 on six of
// 128^3.  Under capture the launch is an ordinary one: as edges of the step's
// graph, programmatic dependencies made the 48-run ensemble 2 % and 256^3
// MHD 3.5 % slower.
cudaError_t launch_dep(const void *kernel, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t s);

// Opt every transform kernel in up front (called by ns_init, so that nothing
// of the kind happens while a step is being captured into a graph).
cudaError_t prepare_fft_kernels();

}  // namespace nsk
