// fused_kA3.cu -- pass A (x inverse of u and of its curl) with shared
// transforms, on constant geometry.
//
// Along an x line k_y and k_z are constants, so the curl's transforms follow
// from those of the velocity and of two products with k_x:
//   w_x = i (k_y U_z - k_z U_y),  w_y = i (k_z U_x - IFFT(k_x u_z)),
//   w_z = i (IFFT(k_x u_y) - k_y U_x).
// A column then takes five transforms and five loads per mode where the six
// independent ones (k_fzk, pass A) take six and nine.  One kind of CTA makes
// U_y, U_z and w_x from u_y and u_z, the other U_x, w_y and w_z; the line kept
// in registers between transforms holds E values.  Bound by latency (six
// fields per column written once, at half of the copy rate); the tuner takes
// it where it is faster than the independent transforms (605 -> 492 us at 512^3,
// 67.8 -> 54.8 at 256^3, 296 -> 238 on 512 x 512 x 256).
#include "fused_k.cuh"

namespace nsk {

template <int NX, int NY, int NZ, int E, int CT>
__global__ void __launch_bounds__(CT *(NX / E))
k_fza3(const float2 *__restrict__ in, float2 *__restrict__ out, const float2 *__restrict__ tw, float3 sc) {
    typedef FzGeom3<NX, NY, NZ, FZ_A> G;
    constexpr int T = NX / E;
    extern __shared__ __align__(16) unsigned char smraw[];
    float2 *sm = reinterpret_cast<float2 *>(smraw);
    const int c = threadIdx.x % CT, slot = threadIdx.x / CT;
    const int kind = blockIdx.x & 1, col = (blockIdx.x >> 1) * CT + c;
    const bool valid = col < G::ncols;
    const int cc = valid ? col : 0, ou = cc / G::Mz, iz = cc - ou * G::Mz;
    const float2 *ib = in + blockIdx.y * G::irun + cc;
    float2 *ob = out + blockIdx.y * G::orun + ou * G::obs + iz;
    const float ky = (float)(ou <= G::Ko ? ou : ou - G::Mo) * (G::box ? sc.y : 1.f);
    const float kz = (float)iz * (G::box ? sc.z : 1.f);
    const float kxs = G::box ? sc.x : 1.f;
    auto load = [&](int f, int e) -> float2 {
        const int r = FzColK<NX, NY, NZ, FZ_A>::compact(e);
        return valid && r >= 0 ? ib[f * G::ifs + r * G::irs] : make_float2(0.f, 0.f);
    };
    auto load_kx = [&](int f, int e) -> float2 {
        return cscale(load(f, e), (float)(2 * e < NX ? e : e - NX) * kxs);
    };
    auto store = [&](int f, int j, float2 v) {
        if (valid) ob[f * G::ofs + (slot + j * T) * G::ors] = v;
    };
    auto sl = [&](int e) -> float2 { return sm[TileIndex<E, CT>::at(e, c)]; };
    auto ss = [&](int e, float2 v) { sm[TileIndex<E, CT>::at(e, c)] = v; };
    float2 X[E], Y[E];
    if (kind == 0) {
        ct_fft_block_reg<NX, E, +1, NX>(X, slot, tw, [&](int e) { return load(1, e); }, sl, ss);
#pragma unroll
        for (int j = 0; j < E; j++) store(1, j, X[j]);
        __syncthreads();   // the transform's last reads of the tile
        ct_fft_block_reg<NX, E, +1, NX>(Y, slot, tw, [&](int e) { return load(2, e); }, sl, ss);
#pragma unroll
        for (int j = 0; j < E; j++) {
            store(2, j, Y[j]);
            store(3, j, make_float2(kz * X[j].y - ky * Y[j].y, ky * Y[j].x - kz * X[j].x));
        }
    } else {
        ct_fft_block_reg<NX, E, +1, NX>(X, slot, tw, [&](int e) { return load(0, e); }, sl, ss);
#pragma unroll
        for (int j = 0; j < E; j++) store(0, j, X[j]);
        __syncthreads();
        ct_fft_block_reg<NX, E, +1, NX>(Y, slot, tw, [&](int e) { return load_kx(2, e); }, sl, ss);
#pragma unroll
        for (int j = 0; j < E; j++)
            store(4, j, make_float2(Y[j].y - kz * X[j].y, kz * X[j].x - Y[j].x));
        __syncthreads();
        ct_fft_block_reg<NX, E, +1, NX>(Y, slot, tw, [&](int e) { return load_kx(1, e); }, sl, ss);
#pragma unroll
        for (int j = 0; j < E; j++)
            store(5, j, make_float2(ky * X[j].y - Y[j].y, Y[j].x - ky * X[j].x));
    }
}

template <int NX, int NY, int NZ, int E, int CT> static bool fza3_fill(FzsKernel *o) {
    o->k = (const void *)k_fza3<NX, NY, NZ, E, CT>;
    o->smem = (size_t)(NX + 1) * TileIndex<E, CT>::rows_stride() * sizeof(float2);
    o->threads = CT * (NX / E);
    return true;
}

bool fza3_lookup(int NX, int NY, int NZ, int E, int CT, FzsKernel *o) {
#define NSK_CASE(n_, e_, ct_) \
    if (NX == n_ && NY == n_ && NZ == n_ && E == e_ && CT == ct_) return fza3_fill<n_, n_, n_, e_, ct_>(o);
    NSK_FZS_SHAPES(NSK_CASE)
#undef NSK_CASE
#define NSK_CASE(nx_, ny_, nz_, e_, ct_) \
    if (NX == nx_ && NY == ny_ && NZ == nz_ && E == e_ && CT == ct_) return fza3_fill<nx_, ny_, nz_, e_, ct_>(o);
    NSK_FZK_GRIDS(NSK_CASE)
#undef NSK_CASE
    return false;
}

}  // namespace nsk
