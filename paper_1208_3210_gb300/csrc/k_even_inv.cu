// Inverse momentum passes of the even form (even.cuh): the correlation spectra
// C(k_x, k_y, w_m) back to the lags (Sec. 3's inverse transform).
//
//   k_ev_inv_x : B3 [M][M][WS] (k_x <= k_y, symmetric) -> B4 [nl][M][WS],
//                lags s_x >= 0 for each k_y (and the adjoint's spectra to
//                p_x >= 0)
//   k_ev_inv_y : B4 -> Im chi at the four lags (+-s_x, +-s_y), times the Eq. 9
//                prefactor, out [Q][Q][n_omega]
#include "even.cuh"

namespace lh {

// Grid: M x (column tiles), the tiles of one k_y neighbours.  `rows` outputs;
// planes of RS-float rows, sp floats apart in B3 and dp in B4.
template <int M>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_ev_inv_x(int rows, int RS, long long sp, long long dp, const float *B3, float *__restrict__ B4,
           const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, true>;
    constexpr int C = F::C, VPT = F::VPT, TPC = F::TPC, RP = F::RP, NBP = F::NBP, RF = F::RF;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float4)
    after_previous();
    float4 *sm = reinterpret_cast<float4 *>(smem_raw);
    const int ky = blockIdx.x / ntile, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;
    const int m = 4 * (ct * C + col);
    const bool on = m < RS;
    Cx2 z[VPT];
#pragma unroll
    for (int b = 0; b < VPT / RF; ++b)
#pragma unroll
        for (int r = 0; r < RF; ++r) {
            const int kx = u + b * TPC + r * (M / RF), lo = min(kx, ky), hi = max(kx, ky);
            z[b * RF + r] = on ? ev_load(B3 + lo * sp + hi * RS + m) : Cx2{dup2(0.f), dup2(0.f)};
        }
    F::run(z, sm + col, u, tab);
    ev_post<M>(z, u, tab);
    if (on) {
        float *o = B4 + (long long)ky * RS + m;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int j = F::template butterfly<F::NS - 1>(b, u);
#pragma unroll
            for (int r = 0; r < RP; ++r) {
                const int l = j + r * NBP;
                if (l < rows) F::st(reinterpret_cast<float4 *>(o + l * dp), z[b * RP + r]);
            }
        }
        // lag M of grids that keep it (Q = 2N = 2M): no pair of points is that far apart
        if (u == 0 && rows > M) *reinterpret_cast<float4 *>(o + M * dp) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// Grid: nl x (column tiles), the tiles of one s_x neighbours.  VEC: the four
// transfers of a pack in one 16-byte store (n_omega % 4 == 0, out aligned).
template <int M, bool VEC>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_ev_inv_y(EvGeom v, int Q, int n_omega, const float *B4, float *__restrict__ out,
           const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, true>;
    constexpr int C = F::C, VPT = F::VPT, TPC = F::TPC, RP = F::RP, NBP = F::NBP, RF = F::RF;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float4)
    after_previous();
    float4 *sm = reinterpret_cast<float4 *>(smem_raw);
    const int sx = blockIdx.x / ntile, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;
    const int m = 4 * (ct * C + col);
    const bool on = m < v.WS;
    const float *in = B4 + (long long)sx * v.s4 + m;
    Cx2 z[VPT];
#pragma unroll
    for (int b = 0; b < VPT / RF; ++b)
#pragma unroll
        for (int r = 0; r < RF; ++r) {
            z[b * RF + r] = on ? ev_load(in + (u + b * TPC + r * (M / RF)) * v.WS) : Cx2{dup2(0.f), dup2(0.f)};
        }
    F::run(z, sm + col, u, tab);
    ev_post<M>(z, u, tab);
    if (m >= n_omega) return;
    // rows l = Q/2 - s and Q/2 + s of each axis (the second for 0 < s < Q/2)
    const bool two_x = sx > 0 && sx < Q / 2;
    float *ox = out + (long long)(Q / 2 - sx) * Q * n_omega + m;
    const long long mx = 2LL * sx * Q * n_omega;
    auto put = [&](float *o, float4 c) {
        if constexpr (VEC) {
            *reinterpret_cast<float4 *>(o) = c;
        } else {
            o[0] = c.x;
            if (m + 1 < n_omega) o[1] = c.y;
            if (m + 2 < n_omega) o[2] = c.z;
            if (m + 3 < n_omega) o[3] = c.w;
        }
    };
    auto put_lag = [&](int sy, float4 c) {
        if (sy > Q / 2) return;
        float *o = ox + (long long)(Q / 2 - sy) * n_omega;
        put(o, c);
        if (two_x) put(o + mx, c);
        if (sy > 0 && sy < Q / 2) {
            o += 2LL * sy * n_omega;
            put(o, c);
            if (two_x) put(o + mx, c);
        }
    };
    const float2 sc = dup2(v.scale);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const int j = F::template butterfly<F::NS - 1>(b, u);
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            const float2 a = mul2(z[b * RP + r].re, sc), c = mul2(z[b * RP + r].im, sc);
            put_lag(j + r * NBP, make_float4(a.x, a.y, c.x, c.y));
        }
    }
    if (u == 0 && v.nl > M) put_lag(M, make_float4(0.f, 0.f, 0.f, 0.f));
}

template <int M>
cudaError_t launch_ev_inv_x_t(int rows, int RS, long long sp, long long dp, const Work<float> &w, cudaStream_t s)
{
    const size_t smem = sizeof(float4) * EvFft<M, true>::SMEM_ELEMS;
    static const cudaError_t e = smem_attrs(k_ev_inv_x<M>, smem);
    if (e != cudaSuccess) return e;
    const int ntile = (RS + 4 * EvCfg<M>::C - 1) / (4 * EvCfg<M>::C);
    return launch_after(k_ev_inv_x<M>, M * ntile, EvCfg<M>::T, smem, s, rows, RS, sp, dp, (const float *)w.X,
                        (float *)w.Y, (const float2 *)w.evt, ntile);
}
template <int M>
cudaError_t launch_ev_inv_y_t(const Geom &g, const EvGeom &v, const Work<float> &w, float *out, cudaStream_t s)
{
    const size_t smem = sizeof(float4) * EvFft<M, true>::SMEM_ELEMS;
    static const cudaError_t e0 = smem_attrs(k_ev_inv_y<M, true>, smem);
    static const cudaError_t e1 = smem_attrs(k_ev_inv_y<M, false>, smem);
    if (e0 != cudaSuccess) return e0;
    if (e1 != cudaSuccess) return e1;
    const int ntile = (v.WS + 4 * EvCfg<M>::C - 1) / (4 * EvCfg<M>::C);
    auto k = g.n_omega % 4 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0 ? k_ev_inv_y<M, true> : k_ev_inv_y<M, false>;
    return launch_after(k, v.nl * ntile, EvCfg<M>::T, smem, s, v, g.Q, g.n_omega, (const float *)w.Y, out,
                        (const float2 *)w.evt, ntile);
}
cudaError_t launch_ev_inv_x(const EvGeom &v, const Work<float> &w, cudaStream_t s)
{
#define CALL(M_) launch_ev_inv_x_t<M_>(v.nl, v.WS, v.s3, v.s4, w, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}
// The adjoint's: X [M][M][ES] (k_x <= k_y) -> Y [Nh][M][ES].
cudaError_t launch_ev_inv_x_bw(const EvGeom &v, const Work<float> &w, cudaStream_t s)
{
#define CALL(M_) launch_ev_inv_x_t<M_>(v.Nh, v.ES, v.s2, v.s1, w, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}
cudaError_t launch_ev_inv_y(const Geom &g, const EvGeom &v, const Work<float> &w, float *out, cudaStream_t s)
{
#define CALL(M_) launch_ev_inv_y_t<M_>(g, v, w, out, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}

}  // namespace lh
