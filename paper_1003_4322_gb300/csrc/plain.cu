// plain.cu -- the unfused, unpruned ("plain") form of the solver's pointwise
// steps on full half-layout arrays [3][N_x][N_y][N_z/2+1] (Sec. 2, Eqs. 1-2):
// the vorticity i k x a, the cross product u x w on the grid, and the
// projected, dealiased, forced integrating-factor RK2 update; plus the
// deterministic FP64 reductions for energy, enstrophy and the shell spectrum
// (the global quantities and spectra of Sec. 3).  Grids of N_x x N_y x N_z
// points on boxes of sides 2 pi l_i (the domains of aspect ratio other than
// one of Sec. 5) go through the same kernels: index m along axis i is the
// wavenumber m / l_i, and the 2/3 rule holds per axis in grid indices.
#include <math.h>

#include <algorithm>

#include "ns_internal.h"
#include "plain.h"
#include "reduce.cuh"

namespace nsk {

static long gcd_l(long a, long b) { return b ? gcd_l(b, a % b) : a; }

Grid make_grid(int nx, int ny, int nz, double lx, double ly, double lz) {
    Grid g;
    g.nx = nx;
    g.ny = ny;
    g.nz = nz;
    g.lx = lx;
    g.ly = ly;
    g.lz = lz;
    g.ilx = 1.0 / lx;
    g.ily = 1.0 / ly;
    g.ilz = 1.0 / lz;
    long D = nx;
    D = D / gcd_l(D, ny) * ny;
    D = D / gcd_l(D, nz) * nz;
    g.D = D;
    g.qx = D / nx;
    g.qy = D / ny;
    g.qz = D / nz;
    g.unit = lx == 1.0 && ly == 1.0 && lz == 1.0;
    g.m32 = g.M() < (1L << 31);
    g.cube = g.unit && nx == ny && ny == nz;
    const double lm = fmax(lx, fmax(ly, lz));
    g.lmax = 1.0 / (1.0 / lm);   // as the shell width 1 / k_min, k_min = 1 / max l
    return g;
}

int grid_nbins(const Grid &g) {
    if (g.cube) return (int)ceil(sqrt(3.0) * g.nx / 2.0) + 1;
    const double cx = g.nx / 2 / g.lx, cy = g.ny / 2 / g.ly, cz = g.nz / 2 / g.lz;
    const double kmin = 1.0 / fmax(g.lx, fmax(g.ly, g.lz));
    return (int)ceil(sqrt(cx * cx + cy * cy + cz * cz) / kmin) + 1;
}

long grid_max_k2(const Grid &g) {
    const long hx = g.nx / 2, hy = g.ny / 2, hz = g.nz / 2;
    return hx * hx + hy * hy + hz * hz;
}

// The pointwise kernels give one warp a row (kx, ky) of the half layout, or
// of the rectangle that holds the kept modes, with the lanes along kz: the
// wavenumbers and the rule's terms of x and y are formed once per row, where
// one thread per mode spent integer divisions and FP64 conversions on each.
// They are bound by the FP64 pipe (2 instructions per SM and clock), so their
// figures below count FP64 instructions per mode.
struct RowIdx {
    long m0;       // position of the row's kz = 0
    int x, y;      // signed indices
    int px, py;    // array positions
};
__host__ __device__ __forceinline__ int rect_rows(const Rect &r, const Grid &g) {
    return r.on ? (2 * r.kx + 1) * (2 * r.ky + 1) : g.nx * g.ny;
}
__device__ __forceinline__ int rect_kz(const Rect &r, const Grid &g) { return r.on ? r.kz + 1 : g.nz / 2 + 1; }
__device__ __forceinline__ RowIdx row_at(int row, const Rect &r, const Grid &g) {
    RowIdx q;
    const int my = r.on ? 2 * r.ky + 1 : g.ny, ix = row / my, iy = row - ix * my;
    q.px = r.on && ix > r.kx ? ix - (2 * r.kx + 1) + g.nx : ix;
    q.py = r.on && iy > r.ky ? iy - my + g.ny : iy;
    q.x = wavenum(q.px, g.nx);
    q.y = wavenum(q.py, g.ny);
    q.m0 = ((long)q.px * g.ny + q.py) * g.nzh();
    return q;
}

// Wavevector of a row's modes in precision T and |k|^2.  On the unit box
// (UNIT) the wavenumbers are the integer indices and |k|^2 an integer (the
// index of the factor table); elsewhere k = m / l is formed from the
// reciprocals in FP64.
template <typename T, bool UNIT> struct RowWave {
    T kx, ky, exy;   // exy: the factors of x and y (boxes)
    double r2;
    int i2;
    __device__ __forceinline__ RowWave(const RowIdx &q, const Grid &g, const T *etab) {
        i2 = q.x * q.x + q.y * q.y;
        if constexpr (UNIT) {
            kx = (T)q.x;
            ky = (T)q.y;
            r2 = 0.0;
            exy = (T)1;
        } else {
            const double dx = kmul(q.x, g.ilx), dy = kmul(q.y, g.ily);
            kx = (T)dx;
            ky = (T)dy;
            r2 = dx * dx + dy * dy;
            exy = etab ? etab[q.px] * etab[g.nx + q.py] : (T)1;
        }
    }
    __device__ __forceinline__ T kz(int z, const Grid &g) const {
        if constexpr (UNIT) return (T)z;
        else return (T)kmul(z, g.ilz);
    }
    // exp(-c |k|^2) from the run's table of `stride` entries per |k|^2: by
    // integer |k|^2 on the unit box; elsewhere the product of the per-axis
    // factors, tabulated by array position ([N_x | N_y | N_z/2+1]).
    template <int STRIDE> __device__ __forceinline__ T factor(int z, const T *etab, const Grid &g) const {
        if constexpr (UNIT) return etab[STRIDE * (i2 + z * z)];
        else return exy * etab[g.nx + g.ny + z];
    }
};

// Is every mode of the rectangle kept?  (the cubic rule's rectangle is its
// kept set)
__device__ __forceinline__ bool all_kept(const Rect &rc, int dealias) { return rc.on && dealias == 0; }

// x / 2 through the exponent: an FP64 multiplication costs this pipe as much as
// 32 integer instructions.  False (x left as it is) where the exponent does not
// give it.  halve3 keeps those multiplications in one branch, as predicated ones
// occupy the FP64 pipe of a warp that needs none.
__device__ __forceinline__ bool halves(double &x) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const unsigned e = ((unsigned)hi >> 20) & 0x7ffu;
    const bool fast = e - 2u < 0x7fdu - 1u, zero = ((hi & 0x7fffffff) | lo) == 0;
    x = __hiloint2double(fast ? hi - 0x100000 : hi, lo);
    return fast || zero;
}
__device__ __forceinline__ void halve3(float2 &a, float2 &b, float2 &c) {
    a = cscale(a, 0.5f);
    b = cscale(b, 0.5f);
    c = cscale(c, 0.5f);
}
__device__ __forceinline__ void halve3(double2 &a, double2 &b, double2 &c) {
    const bool f0 = halves(a.x), f1 = halves(a.y), f2 = halves(b.x), f3 = halves(b.y), f4 = halves(c.x),
               f5 = halves(c.y);
    if (__builtin_expect(!(f0 && f1 && f2 && f3 && f4 && f5), 0)) {
        if (!f0) a.x *= 0.5;
        if (!f1) a.y *= 0.5;
        if (!f2) b.x *= 0.5;
        if (!f3) b.y *= 0.5;
        if (!f4) c.x *= 0.5;
        if (!f5) c.y *= 0.5;
    }
}

// ---------------------------------------------------------------- curl

// Bits of the six parts of a complex vector OR-ed together: zero exactly when
// every part is +0 (an integer test, which keeps the FP64 pipe free).
__device__ __forceinline__ unsigned long long cbits(double2 a, double2 b, double2 c) {
    return (unsigned long long)(__double_as_longlong(a.x) | __double_as_longlong(a.y) |
                                __double_as_longlong(b.x) | __double_as_longlong(b.y) |
                                __double_as_longlong(c.x) | __double_as_longlong(c.y));
}
__device__ __forceinline__ unsigned long long cbits(float2 a, float2 b, float2 c) {
    return (unsigned long long)(__float_as_uint(a.x) | __float_as_uint(a.y) | __float_as_uint(b.x) |
                                __float_as_uint(b.y) | __float_as_uint(c.x) | __float_as_uint(c.y));
}

// w = i k x a (12 FP64 instructions per mode and one conversion; 0.67 -> 0.63 ms at
// 512^3, FP64 pipe 85 % busy).  The
// state is zero outside the kept set (every dealiasing rule); there the curl
// is written as zeros without arithmetic.  With the rectangle on, only its
// modes are read and written (the transforms that follow read no others).
template <typename T, bool UNIT>
__global__ void __launch_bounds__(256)
k_curl(const typename Cx<T>::type *__restrict__ a, typename Cx<T>::type *__restrict__ w, Grid g, long M, Rect rc) {
    typedef typename Cx<T>::type C;
    const int row = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (row >= rect_rows(rc, g)) return;
    const RowIdx q = row_at(row, rc, g);
    const RowWave<T, UNIT> k(q, g, nullptr);
    const T kx = k.kx, ky = k.ky;
    const int nk = rect_kz(rc, g);
    for (int z = threadIdx.x & 31; z < nk; z += 32) {
        const long m = q.m0 + z;
        const C ax = a[m], ay = a[M + m], az = a[2 * M + m];
        if (cbits(ax, ay, az) == 0) {
            w[m] = w[M + m] = w[2 * M + m] = czero<C>();
            continue;
        }
        const T kz = k.kz(z, g);
        w[m] = mkc(kz * ay.y - ky * az.y, ky * az.x - kz * ay.x);
        w[M + m] = mkc(kx * az.y - kz * ax.y, kz * ax.x - kx * az.x);
        w[2 * M + m] = mkc(ky * ax.y - kx * ay.y, kx * ay.x - ky * ax.x);
    }
}

// ---------------------------------------------------------------- cross product

// c = u x w at every grid point; c may alias u.
template <typename T>
__global__ void k_cross(T *u, const T *__restrict__ w, long V) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < V; i += (long)gridDim.x * blockDim.x) {
        const T ux = u[i], uy = u[V + i], uz = u[2 * V + i];
        const T wx = w[i], wy = w[V + i], wz = w[2 * V + i];
        u[i] = uy * wz - uz * wy;
        u[V + i] = uz * wx - ux * wz;
        u[2 * V + i] = ux * wy - uy * wx;
    }
}

// MHD products on the grid: g = [u, w, b, j] (3 components each, V points
// per component); on return g[0..3V) = u x w + j x b and g[3V..6V) = u x b.
template <typename T>
__global__ void k_cross_mhd(T *g, long V) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < V; i += (long)gridDim.x * blockDim.x) {
        const T ux = g[i], uy = g[V + i], uz = g[2 * V + i];
        const T wx = g[3 * V + i], wy = g[4 * V + i], wz = g[5 * V + i];
        const T bx = g[6 * V + i], by = g[7 * V + i], bz = g[8 * V + i];
        const T jx = g[9 * V + i], jy = g[10 * V + i], jz = g[11 * V + i];
        g[i] = uy * wz - uz * wy + (jy * bz - jz * by);
        g[V + i] = uz * wx - ux * wz + (jz * bx - jx * bz);
        g[2 * V + i] = ux * wy - uy * wx + (jx * by - jy * bx);
        g[3 * V + i] = uy * bz - uz * by;
        g[4 * V + i] = uz * bx - ux * bz;
        g[5 * V + i] = ux * by - uy * bx;
    }
}

// ---------------------------------------------------------------- update

// Can a mode of the row (kx, ky) be forced?  The same for a whole warp, so that the rows
// that cannot branch around the additions.
__device__ __forceinline__ bool forced_row(const RowIdx &q, const UpdateArgs &ua) {
    return ua.force_k > 0 && ((q.x == 0 && (q.y == 0 || q.y == ua.mfy || q.y == -ua.mfy)) ||
                              (q.y == 0 && (q.x == ua.mfx || q.x == -ua.mfx)));
}

// ABC forcing coefficients at signed grid index k (closed form of
// f = F (sin kf z + cos kf y, sin kf x + cos kf z, sin kf y + cos kf x));
// kf sits at grid index kf l_i along axis i (mfx, mfy, mfz).
template <typename C, typename T>
__device__ __forceinline__ void abc_forcing(const Idx &k, const UpdateArgs &ua, T F, C &fx, C &fy, C &fz) {
    const T h = F * (T)0.5;
    if (k.x == 0 && k.y == 0 && k.z == ua.mfz) {   // e^{i kf z}: sin -> -i/2, cos -> 1/2
        fx = cadd(fx, mkc((T)0, -h));
        fy = cadd(fy, mkc(h, (T)0));
    }
    if (k.x == 0 && k.z == 0 && (k.y == ua.mfy || k.y == -ua.mfy)) {
        fx = cadd(fx, mkc(h, (T)0));
        fz = cadd(fz, mkc((T)0, k.y > 0 ? -h : h));
    }
    if (k.y == 0 && k.z == 0 && (k.x == ua.mfx || k.x == -ua.mfx)) {
        fy = cadd(fy, mkc((T)0, k.x > 0 ? -h : h));
        fz = cadd(fz, mkc(h, (T)0));
    }
}


// Stage 1: a1 = E (a + dt N);  stage 2: a = E a / 2 + (a1 + dt N) / 2, with
// N = P Pi (nl / N^3) + f_hat; every mode outside Pi (and k = 0) set to 0.
// The projection is applied to nl itself (it is linear) and dt / N^3 joins the
// stage's weights; the forcing enters as dt f_hat at the forced modes only.
// On the unit box the table holds pairs (E, 1/|k|^2) by integer |k|^2, and a
// mode takes 26 FP64 instructions in either stage and one conversion (60 with a
// division, the conversions of k and the halvings as multiplications).  Stage 2
// also sums the new state's energy and enstrophy (9 more a mode; a lane adds
// its modes in order, the block in a fixed tree, the last block the partials),
// which spares a pass of 0.56 ms over the state and a launch (32^3: 747 -> 724 us
// for ten steps).  The forcing and the halvings' rare multiplications sit behind
// branches: predicated, they kept the FP64 pipe busy in every warp (forced 512^3:
// 1.87 -> 1.37 ms in stage 1, 2.53 -> 1.76 in stage 2).
template <typename T, bool UNIT>
__global__ void __launch_bounds__(256)
k_update(typename Cx<T>::type *__restrict__ a, typename Cx<T>::type *__restrict__ a1,
         const typename Cx<T>::type *__restrict__ nl, const T *__restrict__ etab, Grid g, long M, UpdateArgs ua,
         Rect rc, double *part, EnergyOut eo) {
    typedef typename Cx<T>::type C;
    __shared__ double sh[512];
    double en = 0.0, om = 0.0;   // stage 2: energy and enstrophy of the new state
    const int rows = rect_rows(rc, g);
    for (int row = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); row < rows;
         row += (int)(gridDim.x * blockDim.x) >> 5) {
        const RowIdx q = row_at(row, rc, g);
        const RowWave<T, UNIT> k(q, g, etab);
        double er = 0.0, zr = 0.0;   // sums of w |a|^2 and k_z^2 w |a|^2 of the row
        const T gdt = (T)ua.gdt, dt = (T)ua.dt, F = (T)ua.force_amp;
        const T rn = (T)ua.rn;   // the Coriolis factor in the units of nl
        const T kx = k.kx, ky = k.ky;
        const bool every = all_kept(rc, ua.dealias), forced = forced_row(q, ua);
        const int nk = rect_kz(rc, g);
        for (int z = threadIdx.x & 31; z < nk; z += 32) {
            const long m = q.m0 + z;
            const Idx id{q.x, q.y, z};
            C o0 = czero<C>(), o1 = czero<C>(), o2 = czero<C>();
            if ((every || kept(id, g, ua.dealias)) && (q.x | q.y | z) != 0) {
                // v = N^3 (nl / N^3 + Coriolis), in the units of nl
                C vx = nl[m], vy = nl[M + m], vz = nl[2 * M + m];
                if (ua.rot != 0.0) {   // Coriolis -2 rot z x u of the stage's state, before P
                    const C *cur = ua.stage == 1 ? a : a1;
                    vx = cadd(vx, cscale(cur[M + m], rn));
                    vy = csub(vy, cscale(cur[m], rn));
                }
                const T kz = k.kz(z, g);
                T ik2;
                if constexpr (UNIT) ik2 = etab[2 * (k.i2 + z * z) + 1];
                else {
                    const double dz = kmul(z, g.ilz);
                    ik2 = (T)1 / (T)(k.r2 + dz * dz);
                }
                const T e = k.template factor<UNIT ? 2 : 1>(z, etab, g);
                const C s = cscale(mkc(vx.x * kx + vy.x * ky + vz.x * kz, vx.y * kx + vy.y * ky + vz.y * kz), ik2);
                vx = mkc(vx.x - kx * s.x, vx.y - kx * s.y);   // P(k) v = v - k (k.v) / k^2
                vy = mkc(vy.x - ky * s.x, vy.y - ky * s.y);
                vz = mkc(vz.x - kz * s.x, vz.y - kz * s.y);
                const C f0 = a[m], f1 = a[M + m], f2 = a[2 * M + m];
                if (ua.stage == 1) {   // E (a + (dt/N^3) v + dt f)
                    C t0 = mkc(f0.x + gdt * vx.x, f0.y + gdt * vx.y);
                    C t1 = mkc(f1.x + gdt * vy.x, f1.y + gdt * vy.y);
                    C t2 = mkc(f2.x + gdt * vz.x, f2.y + gdt * vz.y);
                    if (__builtin_expect(forced, 0)) abc_forcing(id, ua, F * dt, t0, t1, t2);
                    o0 = cscale(t0, e);
                    o1 = cscale(t1, e);
                    o2 = cscale(t2, e);
                } else {               // (E a + a1 + (dt/N^3) v + dt f) / 2
                    const C g0 = a1[m], g1 = a1[M + m], g2 = a1[2 * M + m];
                    o0 = mkc(e * f0.x + g0.x + gdt * vx.x, e * f0.y + g0.y + gdt * vx.y);
                    o1 = mkc(e * f1.x + g1.x + gdt * vy.x, e * f1.y + g1.y + gdt * vy.y);
                    o2 = mkc(e * f2.x + g2.x + gdt * vz.x, e * f2.y + g2.y + gdt * vz.y);
                    if (__builtin_expect(forced, 0)) abc_forcing(id, ua, F * dt, o0, o1, o2);
                    halve3(o0, o1, o2);
                }
            }
            C *dst = ua.stage == 1 ? a1 : a;
            dst[m] = o0;
            dst[M + m] = o1;
            dst[2 * M + m] = o2;
            if (ua.stage == 2) {
                double a2 = (double)o0.x * o0.x;
                a2 = fma((double)o0.y, (double)o0.y, a2);
                a2 = fma((double)o1.x, (double)o1.x, a2);
                a2 = fma((double)o1.y, (double)o1.y, a2);
                a2 = fma((double)o2.x, (double)o2.x, a2);
                a2 = fma((double)o2.y, (double)o2.y, a2);
                if ((z == 0 || 2 * z == g.nz) && __builtin_expect(!halves(a2), 0)) a2 *= 0.5;   // 1/2 * multiplicity
                const double kz = UNIT ? (double)z : kmul(z, g.ilz);
                er += a2;
                zr = fma(kz * kz, a2, zr);
            }
        }
        en += er;
        om += fma(UNIT ? (double)k.i2 : k.r2, er, zr);
    }
    if (ua.stage == 2) {
        block_sum2(en, om, sh);
        energy_publish(en, om, part, gridDim.x, 0, blockIdx.x, eo);
    }
}

// Induction update of the magnetic field: N_b = Pi (i k x nb / N^3) with nb
// the transform of u x b, then the IF-RK2 stage with the factor of eta.  The
// mean field b(k = 0) has N_b = 0 and factor 1, so it is carried unchanged.
template <typename T, bool UNIT>
__global__ void __launch_bounds__(256)
k_update_b(typename Cx<T>::type *__restrict__ b, typename Cx<T>::type *__restrict__ b1,
           const typename Cx<T>::type *__restrict__ nb, const T *__restrict__ etab, Grid g, long M, int stage,
           double gdt_, int dealias, Rect rc) {
    typedef typename Cx<T>::type C;
    const int row = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (row >= rect_rows(rc, g)) return;
    const RowIdx q = row_at(row, rc, g);
    const RowWave<T, UNIT> k(q, g, etab);
    const T gdt = (T)gdt_;
    const T kx = k.kx, ky = k.ky;
    const bool every = all_kept(rc, dealias);
    const int nk = rect_kz(rc, g);
    for (int z = threadIdx.x & 31; z < nk; z += 32) {
        const long m = q.m0 + z;
        C o0 = czero<C>(), o1 = czero<C>(), o2 = czero<C>();
        if (every || kept(Idx{q.x, q.y, z}, g, dealias)) {
            const C vx = nb[m], vy = nb[M + m], vz = nb[2 * M + m];
            const T kz = k.kz(z, g), e = k.template factor<1>(z, etab, g);
            // i k x v
            const C nx = mkc(kz * vy.y - ky * vz.y, ky * vz.x - kz * vy.x);
            const C ny = mkc(kx * vz.y - kz * vx.y, kz * vx.x - kx * vz.x);
            const C nz = mkc(ky * vx.y - kx * vy.y, kx * vy.x - ky * vx.x);
            const C f0 = b[m], f1 = b[M + m], f2 = b[2 * M + m];
            if (stage == 1) {
                o0 = cscale(mkc(f0.x + gdt * nx.x, f0.y + gdt * nx.y), e);
                o1 = cscale(mkc(f1.x + gdt * ny.x, f1.y + gdt * ny.y), e);
                o2 = cscale(mkc(f2.x + gdt * nz.x, f2.y + gdt * nz.y), e);
            } else {
                const C g0 = b1[m], g1 = b1[M + m], g2 = b1[2 * M + m];
                o0 = mkc(e * f0.x + g0.x + gdt * nx.x, e * f0.y + g0.y + gdt * nx.y);
                o1 = mkc(e * f1.x + g1.x + gdt * ny.x, e * f1.y + g1.y + gdt * ny.y);
                o2 = mkc(e * f2.x + g2.x + gdt * nz.x, e * f2.y + g2.y + gdt * nz.y);
                halve3(o0, o1, o2);
            }
        }
        C *dst = stage == 1 ? b1 : b;
        dst[m] = o0;
        dst[M + m] = o1;
        dst[2 * M + m] = o2;
    }
}

// Phase-shift dealiasing: dst = src exp(i k.D), D half a grid spacing along
// every axis (k.D = pi sum_i m_i / N_i), the coefficients of the field on the
// shifted grid (three components).  The factor is the product of the per-axis
// factors exp(i pi m_i / N_i), tabulated in FP64 by array position
// ([N_x | N_y | N_z/2+1], rounded once to T).  By rows; modes that are zero
// take no arithmetic (16 FP64 instructions for the others: with the average
// below 0.403 -> 0.246 ms on average at 256^3).
template <typename T>
__global__ void __launch_bounds__(256)
k_phase(const typename Cx<T>::type *__restrict__ src, typename Cx<T>::type *__restrict__ dst,
        const typename Cx<T>::type *__restrict__ ph, Grid g, long M, Rect rc) {
    typedef typename Cx<T>::type C;
    const int row = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (row >= rect_rows(rc, g)) return;
    const RowIdx q = row_at(row, rc, g);
    const C fr = cmul(ph[q.px], ph[g.nx + q.py]);
    const int nk = rect_kz(rc, g);
    for (int z = threadIdx.x & 31; z < nk; z += 32) {
        const long m = q.m0 + z;
        C a = src[m], b = src[M + m], c = src[2 * M + m];
        if (cbits(a, b, c) != 0) {
            const C f = cmul(fr, ph[g.nx + g.ny + z]);
            a = cmul(a, f);
            b = cmul(b, f);
            c = cmul(c, f);
        }
        dst[m] = a;
        dst[M + m] = b;
        dst[2 * M + m] = c;
    }
}

// acc = (acc + sh exp(-i k.D)) / 2: the product on the grid and, shifted
// back, on the shifted grid, averaged (three components), for the kept modes,
// which alone the update reads.
template <typename T>
__global__ void __launch_bounds__(256)
k_phase_avg(typename Cx<T>::type *__restrict__ acc, const typename Cx<T>::type *__restrict__ sh,
            const typename Cx<T>::type *__restrict__ ph, Grid g, long M, Rect rc) {
    typedef typename Cx<T>::type C;
    const int row = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (row >= rect_rows(rc, g)) return;
    const RowIdx q = row_at(row, rc, g);
    const C fr = cmul(ph[q.px], ph[g.nx + q.py]);
    const int nk = rect_kz(rc, g);
    for (int z = threadIdx.x & 31; z < nk; z += 32) {
        if (!kept(Idx{q.x, q.y, z}, g, 2)) continue;
        const long m = q.m0 + z;
        const C f = cconj(cmul(fr, ph[g.nx + g.ny + z]));
        C a = cadd(acc[m], cmul(sh[m], f)), b = cadd(acc[M + m], cmul(sh[M + m], f)),
          c = cadd(acc[2 * M + m], cmul(sh[2 * M + m], f));
        halve3(a, b, c);
        acc[m] = a;
        acc[M + m] = b;
        acc[2 * M + m] = c;
    }
}

// ---------------------------------------------------------------- reductions

template <typename T> struct HalfAcc {
    const typename Cx<T>::type *a;
    int n;
    long M;
    __device__ double operator()(int kx, int ky, int kz) const {
        const long m = ((long)((kx + n) % n) * n + (ky + n) % n) * (n / 2 + 1) + kz;
        double s = 0.0;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double re = (double)a[c * M + m].x, im = (double)a[c * M + m].y;
            s += re * re + im * im;
        }
        return s;
    }
};

template <typename T> struct HalfHelAcc {
    const typename Cx<T>::type *a;
    int n;
    long M;
    __device__ double operator()(int kx, int ky, int kz) const {
        const long m = ((long)((kx + n) % n) * n + (ky + n) % n) * (n / 2 + 1) + kz;
        return helicity_density(kx, ky, kz, a[m].x, a[m].y, a[M + m].x, a[M + m].y, a[2 * M + m].x,
                                a[2 * M + m].y);
    }
};

// Per-mode sums for grids other than the cube: signed indices and their
// wavenumbers -> |a|^2 summed over components, or the helicity density.
template <typename T> struct GridAcc {
    const typename Cx<T>::type *a;
    Grid g;
    __device__ double operator()(int mx, int my, int mz, double, double, double) const {
        const long m = ((long)((mx + g.nx) % g.nx) * g.ny + (my + g.ny) % g.ny) * g.nzh() + mz;
        const long M = g.M();
        double s = 0.0;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double re = (double)a[c * M + m].x, im = (double)a[c * M + m].y;
            s += re * re + im * im;
        }
        return s;
    }
};

template <typename T> struct GridHelAcc {
    const typename Cx<T>::type *a;
    Grid g;
    __device__ double operator()(int mx, int my, int mz, double kx, double ky, double kz) const {
        const long m = ((long)((mx + g.nx) % g.nx) * g.ny + (my + g.ny) % g.ny) * g.nzh() + mz;
        const long M = g.M();
        return helicity_density(kx, ky, kz, a[m].x, a[m].y, a[M + m].x, a[M + m].y, a[2 * M + m].x,
                                a[2 * M + m].y);
    }
};

// Shell spectrum on any grid and box: block K sums the modes whose shell
// round-half-up(|k| lmax) is K.  Threads take the (m_x, m_y) pairs that can
// reach the shell; for each, every m_z of a slightly widened interval is
// tested with the shell formula itself, in FP64 with each operation rounded
// as written (no contraction), so that the binning is the definition's.
// Fixed per-thread order and a fixed tree: deterministic.
template <class Acc>
__global__ void __launch_bounds__(256)
k_grid_spectrum(Acc acc, Grid g, int nbins, double *spec, double *aux) {
    __shared__ double sh[512];
    const int K = blockIdx.x, part = blockIdx.y;   // pairs part, part + kShellParts, ... (blocks)
    if (K >= nbins) return;
    const double hi = (K + 0.5) / g.lmax, lo = (K - 0.5) / g.lmax;
    const int bx = (int)(hi * g.lx) + 1, by = (int)(hi * g.ly) + 1;
    const int x0 = max(-bx, -g.nx / 2), x1 = min(bx, g.nx / 2 - 1);
    const int y0 = max(-by, -g.ny / 2), y1 = min(by, g.ny / 2 - 1);
    const long sy = y1 - y0 + 1, pairs = (long)(x1 - x0 + 1) * sy;
    const double hi2 = hi * hi * (1.0 + 1e-9) + 1e-12;
    double e = 0.0, om = 0.0;
    for (long p = (long)part * blockDim.x + threadIdx.x; p < pairs; p += (long)blockDim.x * gridDim.y) {
        const int mx = x0 + (int)(p / sy), my = y0 + (int)(p % sy);
        const double kx = kof(mx, g.lx), ky = kof(my, g.ly);
        const double r2 = __dadd_rn(__dmul_rn(kx, kx), __dmul_rn(ky, ky));
        if (r2 > hi2) continue;
        const double zlo = lo > 0.0 && lo * lo > r2 ? sqrt(lo * lo - r2) : 0.0;
        const double zhi = sqrt(fmax(0.0, hi2 - r2));
        const int z0 = max(0, (int)floor(zlo * g.lz) - 1);
        const int z1 = min(g.nz / 2, (int)ceil(zhi * g.lz) + 1);
        for (int mz = z0; mz <= z1; mz++) {
            const double kz = kof(mz, g.lz);
            const double k2 = __dadd_rn(r2, __dmul_rn(kz, kz));
            if ((long)floor(__dadd_rn(__dmul_rn(__dsqrt_rn(k2), g.lmax), 0.5)) != K) continue;
            const double w = (mz == 0 || 2 * mz == g.nz) ? 0.5 : 1.0;
            const double de = w * acc(mx, my, mz, kx, ky, kz);
            e += de;
            om += de * k2;
        }
    }
    block_sum2(e, om, sh);
    if (threadIdx.x == 0) {
        spec[nbins + K * kShellParts + part] = e;
        aux[nbins + K * kShellParts + part] = om;
    }
}

// ---------------------------------------------------------------- launchers

static unsigned grid_for(long work, int threads) {
    long b = (work + threads - 1) / threads;
    if (b > 152L * 32) b = 152L * 32;
    return (unsigned)(b < 1 ? 1 : b);
}

static unsigned rows_grid(const Rect &rc, const Grid &g) { return (unsigned)((rect_rows(rc, g) + 7) / 8); }

template <typename T>
cudaError_t plain_curl(const typename Cx<T>::type *a, typename Cx<T>::type *w, const Grid &g, const Rect &rc,
                       cudaStream_t s) {
    if (g.unit) k_curl<T, true><<<rows_grid(rc, g), 256, 0, s>>>(a, w, g, g.M(), rc);
    else k_curl<T, false><<<rows_grid(rc, g), 256, 0, s>>>(a, w, g, g.M(), rc);
    return cudaGetLastError();
}

template <typename T>
cudaError_t plain_cross(T *u, const T *w, const Grid &g, cudaStream_t s) {
    const long V = g.V();
    k_cross<T><<<grid_for(V, 256), 256, 0, s>>>(u, w, V);
    return cudaGetLastError();
}

template <typename T>
cudaError_t plain_cross_mhd(T *f, const Grid &g, cudaStream_t s) {
    const long V = g.V();
    k_cross_mhd<T><<<grid_for(V, 256), 256, 0, s>>>(f, V);
    return cudaGetLastError();
}

template <typename T>
cudaError_t plain_update_b(typename Cx<T>::type *b, typename Cx<T>::type *b1,
                           const typename Cx<T>::type *nb, const T *etab, const Grid &g, int stage,
                           double dt, int dealias, const Rect &rc, cudaStream_t s) {
    const long M = g.M();
    const double gdt = dt / (double)g.V();   // on the host: per thread, the division cost more than a mode
    if (g.unit) k_update_b<T, true><<<rows_grid(rc, g), 256, 0, s>>>(b, b1, nb, etab, g, M, stage, gdt, dealias, rc);
    else k_update_b<T, false><<<rows_grid(rc, g), 256, 0, s>>>(b, b1, nb, etab, g, M, stage, gdt, dealias, rc);
    return cudaGetLastError();
}

template <typename T>
cudaError_t plain_phase(const typename Cx<T>::type *src, typename Cx<T>::type *dst,
                        const typename Cx<T>::type *ph, const Grid &g, const Rect &rc, cudaStream_t s) {
    k_phase<T><<<rows_grid(rc, g), 256, 0, s>>>(src, dst, ph, g, g.M(), rc);
    return cudaGetLastError();
}

template <typename T>
cudaError_t plain_phase_avg(typename Cx<T>::type *acc, const typename Cx<T>::type *sh,
                            const typename Cx<T>::type *ph, const Grid &g, const Rect &rc, cudaStream_t s) {
    k_phase_avg<T><<<rows_grid(rc, g), 256, 0, s>>>(acc, sh, ph, g, g.M(), rc);
    return cudaGetLastError();
}

template <typename T>
cudaError_t plain_update(typename Cx<T>::type *a, typename Cx<T>::type *a1,
                         const typename Cx<T>::type *nl, const T *etab, const Grid &g,
                         const UpdateArgs &args, const Rect &rc, double *part, const EnergyOut &eo,
                         cudaStream_t s) {
    const long M = g.M();
    const unsigned blocks = std::min(rows_grid(rc, g), (unsigned)kEnergyParts);
    UpdateArgs ua = args;
    ua.gdt = ua.dt / (double)g.V();
    ua.rn = 2.0 * ua.rot * (double)g.V();
    if (g.unit) k_update<T, true><<<blocks, 256, 0, s>>>(a, a1, nl, etab, g, M, ua, rc, part, eo);
    else k_update<T, false><<<blocks, 256, 0, s>>>(a, a1, nl, etab, g, M, ua, rc, part, eo);
    return cudaGetLastError();
}

template <typename T>
cudaError_t plain_spectrum(const typename Cx<T>::type *a, const Grid &g, const Reach &rc, int nbins, double *spec,
                           double *ens, cudaStream_t s) {
    const HalfAcc<T> cube{a, g.nx, g.M()};
    const GridAcc<T> any{a, g};
    if (nbins <= kRowBins)
        return g.cube ? shell_rows(cube, CubeShells{g.nx}, rc, nbins, spec, ens, s)
                      : shell_rows(any, GridShells{g}, rc, nbins, spec, ens, s);
    return shell_launch(k_grid_spectrum<GridAcc<T>>, nbins, spec, ens, s, any, g, nbins);
}

template <typename T>
cudaError_t plain_helicity(const typename Cx<T>::type *a, const Grid &g, const Reach &rc, int nbins, double *spec,
                           double *aux, cudaStream_t s) {
    const HalfHelAcc<T> cube{a, g.nx, g.M()};
    const GridHelAcc<T> any{a, g};
    if (nbins <= kRowBins)
        return g.cube ? shell_rows(cube, CubeShells{g.nx}, rc, nbins, spec, aux, s)
                      : shell_rows(any, GridShells{g}, rc, nbins, spec, aux, s);
    return shell_launch(k_grid_spectrum<GridHelAcc<T>>, nbins, spec, aux, s, any, g, nbins);
}

#define NSK_INST(T)                                                                                \
    template cudaError_t plain_curl<T>(const Cx<T>::type *, Cx<T>::type *, const Grid &, const Rect &,   \
                                       cudaStream_t);                                             \
    template cudaError_t plain_cross<T>(T *, const T *, const Grid &, cudaStream_t);              \
    template cudaError_t plain_cross_mhd<T>(T *, const Grid &, cudaStream_t);                     \
    template cudaError_t plain_phase<T>(const Cx<T>::type *, Cx<T>::type *, const Cx<T>::type *,  \
                                        const Grid &, const Rect &, cudaStream_t);                \
    template cudaError_t plain_phase_avg<T>(Cx<T>::type *, const Cx<T>::type *, const Cx<T>::type *, \
                                            const Grid &, const Rect &, cudaStream_t);            \
    template cudaError_t plain_update_b<T>(Cx<T>::type *, Cx<T>::type *, const Cx<T>::type *,     \
                                           const T *, const Grid &, int, double, int, const Rect &,  \
                                           cudaStream_t);                                         \
    template cudaError_t plain_update<T>(Cx<T>::type *, Cx<T>::type *, const Cx<T>::type *,       \
                                         const T *, const Grid &, const UpdateArgs &, const Rect &, \
                                         double *, const EnergyOut &, cudaStream_t);              \
    template cudaError_t plain_spectrum<T>(const Cx<T>::type *, const Grid &, const Reach &, int, double *, \
                                           double *, cudaStream_t);                               \
    template cudaError_t plain_helicity<T>(const Cx<T>::type *, const Grid &, const Reach &, int, double *, \
                                           double *, cudaStream_t);
NSK_INST(float)
NSK_INST(double)
#undef NSK_INST

}  // namespace nsk
