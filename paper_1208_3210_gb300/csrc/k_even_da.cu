// Adjoint of the even form (even.cuh) with respect to A itself: dL/dA(p, e) of
// L = sum w(q, w_m) X(q, w_m) at a generated A.
//
// A^ is real and even, so each of the four parity parts of the weights (even or
// odd in s_x and in s_y) gives that part of dL/dA alone, on real lines of one
// quadrant: even axes by cosine transforms, odd ones by sine transforms, which
// ride as the imaginary half of the same complex column (k_even_edge.cu):
//
//   k_ev_gen_y, k_ev_x : A^(k, e), k_x <= k_y                           -> Y
//   k_da_w_y           : w at +-s_y, transformed along s_y               -> X [Q][M][2][WS]
//   k_da_w_x           : the same at +-s_x                               -> Z [M][M][4][WS]
//   k_da_corr          : each part with a^, b^ by FFT along energy (as
//                        k_ev_bw): g = corr(w, b) on the occupied cells, h =
//                        conv(w, a) on the empty ones                    -> X [M][M][4][ES]
//   k_da_inv_x         : to every p_x of the grid                        -> Y [N][M][2][ES]
//   k_da_inv_y         : to every p_y                                    -> dL/dA
//
// The parts odd in one axis enter g with the other sign: conj(W^) there against
// W^ in h.  28 GB of traffic at 1024^2 x 512 instead of the general form's 57:
// 19.5 -> 14.1 ms.  Half of it is the energy pass, 13 transforms a line (256^3: 162
// of 333 us); each part's two spectra turned in one visit, the first in the
// registers, the second in shared memory, instead of two visits: 14.8 -> 14.1 ms.
#include "even.cuh"
#include "even_line.cuh"
#include "et_tiles.cuh"

namespace lh {

// Planes of a frequency pair: the parts (even, even), (even, odd), (odd, even),
// (odd, odd) in (x, y).
enum { DA_EE = 0, DA_OY = 1, DA_OX = 2, DA_OO = 3 };

__host__ __device__ inline long long da_s2(int M, int rs) { return 4LL * M * rs + 64; }   // plane strides (floats) of [..][M][4][rs]
__host__ __device__ inline long long da_s1(int M, int rs) { return 2LL * M * rs + 64; }   // and of [..][M][2][rs]
size_t ev_da_x_floats(const Geom &g, const EvGeom &v)
{
    const size_t a = (size_t)g.Q * da_s1(v.M, v.WS), b = (size_t)v.M * da_s2(v.M, v.ES);
    return a > b ? a : b;
}
size_t ev_da_y_floats(const Geom &g, const EvGeom &v) { return (size_t)g.N * da_s1(v.M, v.ES); }
size_t ev_da_z_floats(const EvGeom &v) { return (size_t)v.M * da_s2(v.M, v.WS); }

__device__ __forceinline__ float2 da_load2(const float *p)
{
    float2 q;
    asm("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(q.x), "=f"(q.y) : "l"(p));
    return q;
}

// Rows +-n of the first stage's inputs into even parts (re) and, at M - n, odd
// ones (im); h = half the window: rows n < h above, n <= h below.
template <int M, typename G>
__device__ __forceinline__ void da_fold(Cx2 *z, int u, int h, G &&get)
{
    constexpr int RP = ev_vpt(M) / 2, NBP = M / RP, TPC = M / ev_vpt(M);
    const float2 half = dup2(0.5f);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const int j = b == 0 ? u : (u == 0 ? TPC : NBP - u);
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            const int n = j + r * NBP;
            const float2 p = n < h ? get(n) : dup2(0.f), q = n == 0 ? p : n <= h ? get(-n) : dup2(0.f);
            z[b * RP + r] = {mul2(add2(p, q), half), mul2(sub2(p, q), half)};
        }
    }
    ev_pairs<RP, NBP, TPC>(z, u, [](int n, Cx2 &a, Cx2 &b) {
        const float2 t = a.im;
        a.im = n == 0 ? dup2(0.f) : b.im;
        if (&a != &b) b.im = t;
    });
}
// Frequency rows of a thread after the forward: f(row, cosine part, sine part).
template <int M, typename S>
__device__ __forceinline__ void da_spectrum(const Cx2 *z, int u, S &&store)
{
    constexpr int RL = ev_radix(M, ev_nstages(M) - 1, false), VPT = ev_vpt(M), TPC = M / VPT;
#pragma unroll
    for (int b = 0; b < VPT / RL; ++b)
#pragma unroll
        for (int r = 0; r < RL; ++r) {
            const int k = u + b * TPC + r * (M / RL);
            const bool up = RL % 2 == 0 ? r >= RL / 2 : k >= M / 2;
            store(k, z[b * RL + r].re, up ? neg2(z[b * RL + r].im) : z[b * RL + r].im);
        }
}
// Both signs of every row l of a window of 2h: f(+-l, value) from the inverse's
// even parts (re) and the odd parts of M - l (im).
template <int M, typename S>
__device__ __forceinline__ void da_unfold(const Cx2 *z, int u, int h, S &&store)
{
    constexpr int RP = ev_vpt(M) / 2, NBP = M / RP, TPC = M / ev_vpt(M);
    const bool u0 = u == 0;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const int j = b == 0 ? u : (u0 ? TPC : NBP - u);
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            const int l = j + r * NBP;
            const float2 other = z[(1 - b) * RP + RP - 1 - r].im;
            const float2 self = b == 1 ? z[RP + RP - 1 - r].im : r == 0 ? dup2(0.f) : z[(RP - r) % RP].im;
            const float2 even = z[b * RP + r].re, odd = u0 ? self : other;
            if (l < h) store(l, add2(even, odd));
            if ((b != 0 || r != 0 || !u0) && l <= h) store(-l, sub2(even, odd));
        }
    }
}

// Grid: Q x (column tiles), a pack is two transfers.
template <int M, bool VEC>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_da_w_y(EvGeom v, int Q, int n_omega, const float *__restrict__ w, float *__restrict__ W1,
         const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, false>;
    constexpr int C = F::C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float4)
    after_previous();
    float4 *sm = reinterpret_cast<float4 *>(smem_raw);
    const int row = blockIdx.x / ntile, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;
    const int m = 2 * (ct * C + col);
    const bool on = m < n_omega;
    const float *in = w + ((long long)row * Q + Q / 2) * n_omega + m;
    Cx2 z[F::VPT];
    da_fold<M>(z, u, Q / 2, [&](int n) {
        const float *p = in + (long long)n * n_omega;
        if (!on) return dup2(0.f);
        if constexpr (VEC) return da_load2(p);
        else return make_float2(p[0], m + 1 < n_omega ? p[1] : 0.f);
    });
    ev_pre<M>(z, u, tab);
    F::run(z, sm + col, u, tab);
    if (m >= v.WS) return;
    float *o = W1 + row * da_s1(M, v.WS) + m;
    da_spectrum<M>(z, u, [&](int k, float2 c, float2 s) {
        float *q = o + 2 * k * v.WS;
        *reinterpret_cast<float2 *>(q) = c;
        *reinterpret_cast<float2 *>(q + v.WS) = s;
    });
}

// Grid: M x 2 (even and odd along y) x (column tiles), the tiles of one k_y
// neighbours.
template <int M>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_da_w_x(EvGeom v, int Q, const float *__restrict__ W1, float *__restrict__ W2, const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, false>;
    constexpr int C = F::C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float4)
    after_previous();
    float4 *sm = reinterpret_cast<float4 *>(smem_raw);
    const int kind = blockIdx.x / ntile % 2, ky = blockIdx.x / ntile / 2, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;
    const int m = 2 * (ct * C + col);
    const bool on = m < v.WS;
    const long long s1 = da_s1(M, v.WS), s2 = da_s2(M, v.WS);
    const float *in = W1 + Q / 2 * s1 + (2 * ky + kind) * v.WS + m;
    Cx2 z[F::VPT];
    da_fold<M>(z, u, Q / 2, [&](int n) { return on ? da_load2(in + n * s1) : dup2(0.f); });
    ev_pre<M>(z, u, tab);
    F::run(z, sm + col, u, tab);
    if (!on) return;
    float *o = W2 + (4 * ky + (kind ? DA_OY : DA_EE)) * (long long)v.WS + m;
    da_spectrum<M>(z, u, [&](int k, float2 c, float2 s) {
        float *q = o + k * s2;
        *reinterpret_cast<float2 *>(q) = c;
        *reinterpret_cast<float2 *>(q + 2 * v.WS) = s;   // EE -> OX, OY -> OO
    });
}

// Per line k_x <= k_y: a^, b^ once, kept in the lane's own places in shared
// memory, then the eight parts' weights at (k_x, k_y) and (k_y, k_x), two to a
// transform, each turned into g^ + i h^ and back: 13 transforms.
template <int L, bool THERMAL>
__global__ void __launch_bounds__(32 * EVC_WARPS, 2)
k_da_corr(Geom g, EvGeom v, Band band, const float *__restrict__ B2, const float *__restrict__ W2, float *__restrict__ G3,
          const float2 *__restrict__ tab, int odd)
{
    using E = EvLine<L>;
    constexpr int VPT = E::VPT, TPL = E::TPL, R0 = E::R0, R1 = E::R1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(EVC_WARPS * (E::WARP_ELEMS + 128 * (R1 + 1)) + (THERMAL ? L : 0), float2)
    after_previous();
    const int lane = (int)threadIdx.x % 32, warp = (int)threadIdx.x / 32;
    const int sl = lane / TPL, u = lane % TPL;
    float2 *base = reinterpret_cast<float2 *>(smem_raw);
    float2 *sm = base + warp * E::WARP_ELEMS + sl * E::LP;
    float4 *own_a = reinterpret_cast<float4 *>(base + EVC_WARPS * E::WARP_ELEMS) + warp * 64 * (R1 + 1) + lane;
    float4 *own_w = own_a + 32 * (R1 + 1);
    float2 *wf = base + EVC_WARPS * (E::WARP_ELEMS + 128 * (R1 + 1));
    if constexpr (THERMAL) {
        et_fermi_weights<L>(g, band, wf, (int)threadIdx.x, 32 * EVC_WARPS);
        __syncthreads();
    }
    const int t = (blockIdx.x * EVC_WARPS + warp) * E::LPI + sl;
    const bool live = t < v.M * (v.M + 1) / 2;
    int kx, ky;
    ev_tri(live ? t : 0, v.M, kx, ky);
    float2 x[VPT];
    {
        float raw[VPT];
        const float *p = B2 + (kx * v.s2 + (long long)ky * v.ES + u);
#pragma unroll
        for (int i = 0; i < VPT; ++i) raw[i] = live && u + E::first(i) < v.ne ? __ldcs(p + E::first(i)) : 0.f;
        E::template first_stage<false, THERMAL>(x, raw, u, v.J0, wf);
    }
    E::forward_rest(x, sm, u, tab);
    // the two real lines of Z: Z(k) + conj Z(-k), (Z(k) - conj Z(-k)) / i; slot
    // by slot in the order of ev_pairs
    int slot = 0;
    ev_pairs<R1, R0, TPL>(x, u, [&](int, float2 &zk, float2 &zm) {
        own_a[32 * slot++] = make_float4(zk.x + zm.x, zk.y - zm.y, zk.y + zm.y, zm.x - zk.x);
    });
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
        const int px = c < 2 ? kx : ky, py = c < 2 ? ky : kx;
        // the parts even or odd in both axes, then those odd in one
        const bool mixed = c % 2 != 0;
        const int p0 = mixed ? DA_OY : DA_EE, p1 = mixed ? DA_OX : DA_OO;
        const float *in = W2 + px * da_s2(v.M, v.WS) + 4LL * py * v.WS + u;
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const int n = E::first(i);
            const bool on = live && u + n < g.n_omega;
            x[i] = on ? make_float2(0.5f * __ldcs(in + p0 * v.WS + n), 0.5f * __ldcs(in + p1 * v.WS + n))
                      : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int b = 0; b < VPT / R0; ++b) ev_dft<R0, false>(x + b * R0);
        E::forward_rest(x, sm, u, tab);
        // g^ + i h^ of the first part in place, of the second into the lane's own places
        slot = 0;
        ev_pairs<R1, R0, TPL>(x, u, [&](int, float2 &zk, float2 &zm) {
            float2 w0 = make_float2(zk.x + zm.x, zk.y - zm.y), w1 = make_float2(zk.y + zm.y, zm.x - zk.x);
            if (THERMAL && odd) {   // w(s, m) - w(-s, -m)
                w0 = mixed ? make_float2(w0.x + w0.x, 0.f) : odd_part(w0, true);
                w1 = mixed ? make_float2(w1.x + w1.x, 0.f) : odd_part(w1, true);
            }
            const float4 ab = own_a[32 * slot];
            const float2 a = make_float2(ab.x, ab.y), b = make_float2(ab.z, ab.w);
            const float2 g0 = cmulc(b, w0), h0 = cmul(a, w0), g1 = cmulc(b, w1), h1 = cmul(a, w1);
            own_w[32 * slot++] = make_float4(g1.x - h1.y, g1.y + h1.x, g1.x + h1.y, h1.x - g1.y);
            const bool self = &zk == &zm;
            zk = make_float2(g0.x - h0.y, g0.y + h0.x);               // g^ + i h^
            if (!self) zm = make_float2(g0.x + h0.y, h0.x - g0.y);    // conj g^ + i conj h^
        });
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
            if (q == 1) {
                slot = 0;
                ev_pairs<R1, R0, TPL>(x, u, [&](int, float2 &zk, float2 &zm) {
                    const float4 z = own_w[32 * slot++];
                    const bool self = &zk == &zm;
                    zk = make_float2(z.x, z.y);
                    if (!self) zm = make_float2(z.z, z.w);
                });
            }
            E::inverse(x, sm, u, tab);
            if (live) {
                float *o = G3 + (px * da_s2(v.M, v.ES) + (4LL * py + (q == 0 ? p0 : p1)) * v.ES + u);
                const float sg = mixed ? -1.f : 1.f;
#pragma unroll
                for (int i = 0; i < VPT; ++i) {
                    const int n = u + E::last(i);
                    float r;
                    if constexpr (THERMAL) {
                        const float2 fw = wf[n];
                        r = sg * fw.x * x[i].x + fw.y * x[i].y;
                    } else {
                        r = n < v.J0 ? sg * x[i].x : x[i].y;
                    }
                    if (n < v.ES) o[E::last(i)] = n < v.ne ? r : 0.f;
                }
            }
        }
    }
}

// Grid: M x 2 x (column tiles); a pack is two energies.
template <int M>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_da_inv_x(EvGeom v, int N, const float *__restrict__ G3, float *__restrict__ G4, const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, true>;
    constexpr int C = F::C, VPT = F::VPT, TPC = F::TPC, RF = F::RF;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float4)
    after_previous();
    float4 *sm = reinterpret_cast<float4 *>(smem_raw);
    const int kind = blockIdx.x / ntile % 2, ky = blockIdx.x / ntile / 2, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;
    const int e = 2 * (ct * C + col);
    const bool on = e < v.ES;
    const long long s1 = da_s1(M, v.ES), s2 = da_s2(M, v.ES);
    const float *in = G3 + (4 * ky + (kind ? DA_OY : DA_EE)) * (long long)v.ES + e;
    Cx2 z[VPT];
#pragma unroll
    for (int b = 0; b < VPT / RF; ++b)
#pragma unroll
        for (int r = 0; r < RF; ++r) {
            const int k = u + b * TPC + r * (M / RF);
            const bool up = RF % 2 == 0 ? r >= RF / 2 : k >= M / 2;
            const float2 c = on ? da_load2(in + k * s2) : dup2(0.f), s = on ? da_load2(in + k * s2 + 2 * v.ES) : dup2(0.f);
            z[b * RF + r] = {c, up ? neg2(s) : s};
        }
    F::run(z, sm + col, u, tab);
    ev_post<M>(z, u, tab);
    if (!on) return;
    float *o = G4 + N / 2 * s1 + (2 * ky + kind) * v.ES + e;
    da_unfold<M>(z, u, N / 2, [&](int l, float2 c) { *reinterpret_cast<float2 *>(o + l * s1) = c; });
}

// Grid: N x (column tiles).  Energies [e0, e0 + ne) of rows of n_eps.
template <int M, bool VEC>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_da_inv_y(EvGeom v, int N, int n_eps, const float *__restrict__ G4, float *__restrict__ dA,
           const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, true>;
    constexpr int C = F::C, VPT = F::VPT, TPC = F::TPC, RF = F::RF;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float4)
    after_previous();
    float4 *sm = reinterpret_cast<float4 *>(smem_raw);
    const int row = blockIdx.x / ntile, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;
    const int e = 2 * (ct * C + col);
    const bool on = e < v.ES;
    const float *in = G4 + row * da_s1(M, v.ES) + e;
    const float2 sc = dup2(v.scale);
    Cx2 z[VPT];
#pragma unroll
    for (int b = 0; b < VPT / RF; ++b)
#pragma unroll
        for (int r = 0; r < RF; ++r) {
            const int k = u + b * TPC + r * (M / RF);
            const bool up = RF % 2 == 0 ? r >= RF / 2 : k >= M / 2;
            const float2 c = on ? da_load2(in + 2 * k * v.ES) : dup2(0.f), s = on ? da_load2(in + (2 * k + 1) * v.ES) : dup2(0.f);
            z[b * RF + r] = {mul2(c, sc), mul2(up ? neg2(s) : s, sc)};
        }
    F::run(z, sm + col, u, tab);
    ev_post<M>(z, u, tab);
    if (e >= v.ne) return;
    float *o = dA + ((long long)row * N + N / 2) * n_eps + v.e0 + e;
    da_unfold<M>(z, u, N / 2, [&](int l, float2 c) {
        float *q = o + (long long)l * n_eps;
        if constexpr (VEC) {
            *reinterpret_cast<float2 *>(q) = c;
        } else {
            q[0] = c.x;
            if (e + 1 < v.ne) q[1] = c.y;
        }
    });
}

// Energies outside the window reach no kept transfer.
__global__ void k_da_zero(long long count, int n_eps, int e0, int ne, float *__restrict__ dA)
{
    after_previous();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
        const int e = (int)(i % n_eps);
        if (e < e0 || e >= e0 + ne) dA[i] = 0.f;
    }
}

template <int M>
cudaError_t launch_da_weights_t(const Geom &g, const EvGeom &v, const float *wts, const Work<float> &w, float *Z,
                                cudaStream_t s)
{
    constexpr int C = EvCfg<M>::C;
    const size_t smem = sizeof(float4) * EvFft<M, false>::SMEM_ELEMS;
    static const cudaError_t e0 = smem_attrs(k_da_w_y<M, true>, smem), e1 = smem_attrs(k_da_w_y<M, false>, smem),
                             e2 = smem_attrs(k_da_w_x<M>, smem);
    if (e0 != cudaSuccess) return e0;
    if (e1 != cudaSuccess) return e1;
    if (e2 != cudaSuccess) return e2;
    const int nt = (v.WS / 2 + C - 1) / C;
    auto k = g.n_omega % 2 == 0 && reinterpret_cast<uintptr_t>(wts) % 8 == 0 ? k_da_w_y<M, true> : k_da_w_y<M, false>;
    const cudaError_t e = launch_after(k, g.Q * nt, EvCfg<M>::T, smem, s, v, g.Q, g.n_omega, wts, (float *)w.X,
                                       (const float2 *)w.evt, nt);
    if (e != cudaSuccess) return e;
    return launch_after(k_da_w_x<M>, 2 * M * nt, EvCfg<M>::T, smem, s, v, g.Q, (const float *)w.X, Z,
                        (const float2 *)w.evt, nt);
}
template <int M>
cudaError_t launch_da_inverse_t(const Geom &g, const EvGeom &v, const Work<float> &w, float *dA, cudaStream_t s)
{
    constexpr int C = EvCfg<M>::C;
    const size_t smem = sizeof(float4) * EvFft<M, true>::SMEM_ELEMS;
    static const cudaError_t e0 = smem_attrs(k_da_inv_x<M>, smem), e1 = smem_attrs(k_da_inv_y<M, true>, smem),
                             e2 = smem_attrs(k_da_inv_y<M, false>, smem);
    if (e0 != cudaSuccess) return e0;
    if (e1 != cudaSuccess) return e1;
    if (e2 != cudaSuccess) return e2;
    const int nt = (v.ES / 2 + C - 1) / C;
    cudaError_t e = launch_after(k_da_inv_x<M>, 2 * M * nt, EvCfg<M>::T, smem, s, v, g.N, (const float *)w.X, (float *)w.Y,
                                 (const float2 *)w.evt, nt);
    if (e == cudaSuccess && v.ne < g.n_eps)
        e = launch_after(k_da_zero, 1024, 256, 0, s, (long long)g.N * g.N * g.n_eps, g.n_eps, v.e0, v.ne, dA);
    if (e != cudaSuccess) return e;
    const bool vec = g.n_eps % 2 == 0 && v.ne % 2 == 0 && reinterpret_cast<uintptr_t>(dA + v.e0) % 8 == 0;
    return launch_after(vec ? k_da_inv_y<M, true> : k_da_inv_y<M, false>, g.N * nt, EvCfg<M>::T, smem, s, v, g.N, g.n_eps,
                        (const float *)w.Y, dA, (const float2 *)w.evt, nt);
}
template <int L, bool THERMAL>
cudaError_t launch_da_corr_t(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, const float *Z,
                             cudaStream_t s)
{
    using E = EvLine<L>;
    const size_t smem = sizeof(float2) * (EVC_WARPS * (E::WARP_ELEMS + 128 * (E::R1 + 1)) + (THERMAL ? L : 0));
    static const cudaError_t e = smem_attrs(k_da_corr<L, THERMAL>, smem);
    if (e != cudaSuccess) return e;
    const int n = v.M * (v.M + 1) / 2, per = EVC_WARPS * E::LPI;
    return launch_after(k_da_corr<L, THERMAL>, (n + per - 1) / per, 32 * EVC_WARPS, smem, s, g, v, band,
                        (const float *)w.Y, Z, (float *)w.X, (const float2 *)w.evt + ev_line_table<L>(),
                        (int)(g.quantity == LINDHARD_IMCHI_T));
}
cudaError_t launch_da_weights(const Geom &g, const EvGeom &v, const float *wts, const Work<float> &w, float *Z, cudaStream_t s)
{
#define CALL(M_) launch_da_weights_t<M_>(g, v, wts, w, Z, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}
cudaError_t launch_da_corr(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, const float *Z,
                           cudaStream_t s)
{
    const bool th = g.quantity != LINDHARD_IMCHI;
    switch (v.PE) {
    case 128: return th ? launch_da_corr_t<128, true>(g, v, band, w, Z, s) : launch_da_corr_t<128, false>(g, v, band, w, Z, s);
    case 256: return th ? launch_da_corr_t<256, true>(g, v, band, w, Z, s) : launch_da_corr_t<256, false>(g, v, band, w, Z, s);
    case 384: return th ? launch_da_corr_t<384, true>(g, v, band, w, Z, s) : launch_da_corr_t<384, false>(g, v, band, w, Z, s);
    case 512: return th ? launch_da_corr_t<512, true>(g, v, band, w, Z, s) : launch_da_corr_t<512, false>(g, v, band, w, Z, s);
    default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_da_inverse(const Geom &g, const EvGeom &v, const Work<float> &w, float *dA, cudaStream_t s)
{
#define CALL(M_) launch_da_inverse_t<M_>(g, v, w, dA, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}

}  // namespace lh
