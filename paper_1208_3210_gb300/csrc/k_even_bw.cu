// Adjoint of the even form (even.cuh): dL/d(t, t', t'', mu, gamma) of
// L = sum w(q, w_m) X(q, w_m) for a generated A.
//
// dA/dtheta is even in p_x and p_y and symmetric under their exchange, like A,
// so only that part of dL/dA counts, and with it only the same part of the
// weights: the four lags (+-s_x, +-s_y) of w are added, and the rest of the
// adjoint (Eq. 9 is bilinear in the occupied part a and the empty part b:
// g = correlation of w with b on the occupied cells, h = convolution of w with
// a on the empty ones) runs on real cosine spectra of one quadrant, the
// forward's passes in turn:
//
//   k_ev_gen_y, k_ev_x : A^(k, e), k_x <= k_y (as the forward call)      -> Y
//   k_ev_w_y           : w folded to s >= 0, transformed along s_y       -> X
//   k_ev_x             : W^(k, w_m) along s_x, every k_x                 -> Z
//   k_ev_bw            : per k_x <= k_y, W^(k_x, k_y) + W^(k_y, k_x) against
//                        a^, b^ by FFT along energy: G(k, e)             -> X
//   k_ev_inv_x         : G along k_x, p_x >= 0                           -> Y
//   k_ev_chain         : G along k_y, times dA/dtheta, summed
//
// The transposes: the DCT-II's is the DCT-III and the other way round, with
// row 0 of the input weighted 2 (row 0 of the output weighted 1/2).
#include "even.cuh"
#include "even_line.cuh"
#include "et_tiles.cuh"

namespace lh {

// Grid: min(nl, M) x (column tiles), the tiles of one s_x neighbours.  VEC: four
// transfers of a row in one 16-byte load.
template <int M, bool VEC>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_ev_w_y(EvGeom v, int Q, int n_omega, const float *w, float *__restrict__ W1,
         const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, false>;
    constexpr int C = F::C, VPT = F::VPT, TPC = F::TPC, RP = F::RP, NBP = F::NBP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float4)
    after_previous();
    float4 *sm = reinterpret_cast<float4 *>(smem_raw);
    const int sx = blockIdx.x / ntile, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;
    const int m = 4 * (ct * C + col);
    const bool on = m < n_omega;
    // rows Q/2 - s and Q/2 + s of each axis (the second for 0 < s < Q/2)
    const bool two_x = sx > 0 && sx < Q / 2;
    const float *in = w + (long long)(Q / 2 - sx) * Q * n_omega + m;
    const long long mx = 2LL * sx * Q * n_omega;
    auto get = [&](const float *p) {
        if constexpr (VEC) {
            return ev_load(p);
        } else {
            return Cx2{make_float2(p[0], m + 1 < n_omega ? p[1] : 0.f),
                       make_float2(m + 2 < n_omega ? p[2] : 0.f, m + 3 < n_omega ? p[3] : 0.f)};
        }
    };
    const float2 cx = dup2(sx == 0 ? 2.f * v.scale : v.scale);
    Cx2 z[VPT];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const int j = F::template butterfly<0>(b, u);
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            const int s = j + r * NBP;
            Cx2 a = {dup2(0.f), dup2(0.f)};
            if (on && s <= Q / 2) {
                const float *p = in + (long long)(Q / 2 - s) * n_omega;
                a = get(p);
                if (two_x) a = add(a, get(p + mx));
                if (s == 0) {
                    a = add(a, a);
                } else if (s < Q / 2) {
                    p += 2LL * s * n_omega;
                    a = add(a, get(p));
                    if (two_x) a = add(a, get(p + mx));
                }
            }
            z[b * RP + r] = {mul2(a.re, cx), mul2(a.im, cx)};
        }
    }
    ev_pre<M>(z, u, tab);
    F::run(z, sm + col, u, tab);
    if (m < v.WS) {
        float *o = W1 + sx * v.s4 + m;
        constexpr int RL = ev_radix(M, F::NS - 1, false);
#pragma unroll
        for (int b = 0; b < VPT / RL; ++b)
#pragma unroll
            for (int r = 0; r < RL; ++r)
                F::st(reinterpret_cast<float4 *>(o + (u + b * TPC + r * (M / RL)) * v.WS), z[b * RL + r]);
    }
}

// Per pair of lines k (k_x <= k_y): their weights share one transform, which
// waits in shared memory (each lane's own values) while each line's a^, b^ are
// formed, turned in place into g^ + i h^ (g^ = conj(W^) b^, h^ = W^ a^) and
// transformed back.  2.5 transforms a line.
template <int L, bool FULL, bool THERMAL>
__global__ void __launch_bounds__(32 * EVC_WARPS, 2)
k_ev_bw(Geom g, EvGeom v, Band band, const float *B2, const float *W2,
        float *__restrict__ G3, const float2 *__restrict__ tab, int iters, int odd)
{
    using E = EvLine<L>;
    constexpr int VPT = E::VPT, TPL = E::TPL, R0 = E::R0, R1 = E::R1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(EVC_WARPS * (E::WARP_ELEMS + 64 * (R1 + 1)) + (THERMAL ? L : 0), float2)
    after_previous();
    const int lane = (int)threadIdx.x % 32, warp = (int)threadIdx.x / 32;
    const int sl = lane / TPL, u = lane % TPL;
    float2 *sm = reinterpret_cast<float2 *>(smem_raw) + warp * E::WARP_ELEMS + sl * E::LP;
    float4 *own = reinterpret_cast<float4 *>(reinterpret_cast<float2 *>(smem_raw) + EVC_WARPS * E::WARP_ELEMS) +
                  warp * 32 * (R1 + 1) + lane;
    float2 *wf = reinterpret_cast<float2 *>(smem_raw) + EVC_WARPS * (E::WARP_ELEMS + 64 * (R1 + 1));
    if constexpr (THERMAL) {
        et_fermi_weights<L>(g, band, wf, (int)threadIdx.x, 32 * EVC_WARPS);
        __syncthreads();
    }
    const int npairs = v.M / 2 * (v.M + 1) / 2;

    for (int it = 0; it < iters; ++it) {
        const int f = ((blockIdx.x * EVC_WARPS + warp) * iters + it) * E::LPI + sl;
        const bool live = f < npairs;
        float2 x[VPT];
        {
            // both lines' symmetrised weights as one complex line; 1/4: the
            // mean of the two halves and the 1/2 of the separation
            const float *p[2], *q[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                int kx, ky;
                ev_tri(live ? 2 * f + h : 0, v.M, kx, ky);
                p[h] = W2 + kx * v.s3 + (long long)ky * v.WS + u;
                q[h] = W2 + ky * v.s3 + (long long)kx * v.WS + u;
            }
#pragma unroll
            for (int i = 0; i < VPT; ++i) {
                const int n = E::first(i);
                const bool on = live && u + n < g.n_omega;
                x[i] = on ? make_float2(0.25f * (p[0][n] + q[0][n]), 0.25f * (p[1][n] + q[1][n]))
                          : make_float2(0.f, 0.f);
            }
        }
#pragma unroll
        for (int b = 0; b < VPT / R0; ++b) ev_dft<R0, false>(x + b * R0);
        E::forward_rest(x, sm, u, tab);
        // W0^ = Z(k) + conj Z(-k), W1^ = (Z(k) - conj Z(-k)) / i; slot by slot
        // in the order in which ev_pairs visits them below
        int slot = 0;
        auto keep = [&](int, float2 &zk, float2 &zm) {
            float2 w0 = make_float2(zk.x + zm.x, zk.y - zm.y), w1 = make_float2(zk.y + zm.y, zm.x - zk.x);
            if (THERMAL) {
                w0 = odd_part(w0, odd != 0);
                w1 = odd_part(w1, odd != 0);
            }
            own[32 * slot++] = make_float4(w0.x, w0.y, w1.x, w1.y);
        };
        ev_pairs<R1, R0, TPL>(x, u, keep);
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
            int kx, ky;
            ev_tri(live ? 2 * f + q : 0, v.M, kx, ky);
            float raw[VPT];
            const float *p = B2 + (kx * v.s2 + (long long)ky * v.ES + u);
#pragma unroll
            for (int i = 0; i < VPT; ++i)
                raw[i] = live && (FULL || u + E::first(i) < v.ne) ? __ldcs(p + E::first(i)) : 0.f;
            E::template first_stage<FULL, THERMAL>(x, raw, u, v.J0, wf);
            E::forward_rest(x, sm, u, tab);
            slot = 0;
            auto turn = [&](int, float2 &zk, float2 &zm) {
                const float4 ww = own[32 * slot++];
                const float2 w = q == 0 ? make_float2(ww.x, ww.y) : make_float2(ww.z, ww.w);
                const float2 a = make_float2(zk.x + zm.x, zk.y - zm.y), b = make_float2(zk.y + zm.y, zm.x - zk.x);
                const float2 gk = cmulc(b, w), hk = cmul(a, w);
                const bool self = &zk == &zm;
                zk = make_float2(gk.x - hk.y, gk.y + hk.x);               // g^ + i h^
                if (!self) zm = make_float2(gk.x + hk.y, hk.x - gk.y);    // conj g^ + i conj h^
            };
            ev_pairs<R1, R0, TPL>(x, u, turn);
            E::inverse(x, sm, u, tab);
            if (live) {
                float *o = G3 + (kx * v.s2 + (long long)ky * v.ES + u);
#pragma unroll
                for (int i = 0; i < VPT; ++i) {
                    const int n = u + E::last(i);
                    float r;
                    if constexpr (THERMAL) {
                        const float2 fw = wf[n];
                        r = fw.x * x[i].x + fw.y * x[i].y;
                    } else {
                        r = n < v.J0 ? x[i].x : x[i].y;
                    }
                    if (n < v.ES) o[E::last(i)] = n < v.ne ? r : 0.f;
                }
            }
        }
    }
}

// Grid: Nh x (column tiles).  partial[blockIdx.x][5] receives this CTA's sums.
template <int M>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_ev_chain(Geom g, EvGeom v, Band band, const AxisTab *axis, const float2 *eps,
           const InstState *st, const float *G4, double *__restrict__ partial,
           const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, true>;
    constexpr int C = F::C, T = F::T, VPT = F::VPT, TPC = F::TPC, RP = F::RP, NBP = F::NBP, RF = F::RF;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float4)
    after_previous();
    float4 *sm = reinterpret_cast<float4 *>(smem_raw);
    const int jx = blockIdx.x / ntile, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;
    const int e = 4 * (ct * C + col);
    const bool on = e < v.ES;
    const float *in = G4 + (long long)jx * v.s1 + e;
    Cx2 z[VPT];
#pragma unroll
    for (int b = 0; b < VPT / RF; ++b)
#pragma unroll
        for (int r = 0; r < RF; ++r)
            z[b * RF + r] = on ? ev_load(in + (u + b * TPC + r * (M / RF)) * v.ES) : Cx2{dup2(0.f), dup2(0.f)};
    F::run(z, sm + col, u, tab);
    ev_post<M>(z, u, tab);

    // per row p_y: band energy, amplitude (with the transposes' 1/2 at p = 0),
    // cos p_y and cos 2 p_y, in the exchange buffer (24 Nh bytes: Nh < M rows of
    // at least two packs)
    __syncthreads();
    float4 *rows = sm;
    float2 *cy = reinterpret_cast<float2 *>(sm + v.Nh);
    const AxisTab ax = axis[g.N / 2 + jx];
    for (int i = threadIdx.x; i < v.Nh; i += T) {
        const AxisTab ay = axis[g.N / 2 + i];
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        band_point_f32(band, ax, ay, st, q.x, q.y, q.z);
        q.z *= (jx == 0 ? 0.5f : 1.f) * (i == 0 ? 0.5f : 1.f);
        rows[i] = q;
        cy[i] = make_float2(ay.c1h, ay.c2h);
    }
    __syncthreads();
    float2 eh[2], el[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int k = min(e + 2 * h, v.ne - 1), k1 = min(e + 2 * h + 1, v.ne - 1);   // past the window G is 0
        const float2 a = eps[v.e0 + k], b = eps[v.e0 + k1];
        eh[h] = make_float2(a.x, b.x);
        el[h] = make_float2(a.y, b.y);
    }
    // G dA/dxi = G amp 2 d / D^2 and G dA/dgamma = G (amp / gamma) (d^2 - gamma^2) / D^2
    const float2 g2 = dup2(band.gam2);
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;   // sums of G amp d / D^2 times 1, cos p_y, cos 2 p_y
    float2 sg = dup2(0.f);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const int j = F::template butterfly<F::NS - 1>(b, u);
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            const int n = j + r * NBP;
            if (n < v.Nh) {
                const float4 q = rows[n];
                const float2 c = cy[n];
                float2 sum = dup2(0.f);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 d = add2(sub2(eh[h], dup2(q.x)), sub2(el[h], dup2(q.y)));
                    const float2 d2 = mul2(d, d), D = add2(d2, g2);
                    const float2 iD = make_float2(rcp_approx(D.x), rcp_approx(D.y));
                    const float2 t = mul2(mul2(h ? z[b * RP + r].im : z[b * RP + r].re, dup2(q.z)), mul2(iD, iD));
                    sum = fma2(t, d, sum);
                    sg = fma2(t, sub2(d2, g2), sg);
                }
                const float a = sum.x + sum.y;
                s0 += a;
                s1 = fmaf(a, c.x, s1);
                s2 = fmaf(a, c.y, s2);
            }
        }
    }
    double val[4] = {s0, s1, s2, (double)sg.x + (double)sg.y};
    // the last warp may be a part of one (T = 144)
    constexpr int NWP = (T + 31) / 32;
    const int lane = threadIdx.x % 32, wp = threadIdx.x / 32, nl = min(32, T - 32 * wp);
    const unsigned mask = nl == 32 ? 0xffffffffu : (1u << nl) - 1u;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        for (int o = 16; o > 0; o >>= 1) {
            const double other = __shfl_down_sync(mask, val[q], o);
            if (lane + o < nl) val[q] += other;
        }
    __syncthreads();   // the rows have been read
    double *red = reinterpret_cast<double *>(smem_raw);
    if (lane == 0)
        for (int q = 0; q < 4; ++q) red[wp * 4 + q] = val[q];
    __syncthreads();
    if (threadIdx.x == 0) {
        double t[4] = {0, 0, 0, 0};
        for (int i = 0; i < NWP; ++i)
            for (int q = 0; q < 4; ++q) t[q] += red[i * 4 + q];
        const bool tb = band.band_kind != 1;
        double *o = partial + 5LL * blockIdx.x;
        o[0] = tb ? -4.0 * (ax.c1 * t[0] + t[1]) : 0.0;        // 2 x dxi/dt = -2 (cos p_x + cos p_y)
        o[1] = tb ? -8.0 * ax.c1 * t[1] : 0.0;                 // dxi/dt' = -4 cos p_x cos p_y
        o[2] = tb ? -4.0 * (ax.c2 * t[0] + t[2]) : 0.0;        // dxi/dt'' = -2 (cos 2p_x + cos 2p_y)
        o[3] = -2.0 * t[0];                                    // dxi/dmu = -1
        o[4] = t[3] / band.gamma;
    }
}

template <int M>
cudaError_t launch_ev_w_y_t(const Geom &g, const EvGeom &v, const float *wts, const Work<float> &w, cudaStream_t s)
{
    const size_t smem = sizeof(float4) * EvFft<M, false>::SMEM_ELEMS;
    static const cudaError_t e0 = smem_attrs(k_ev_w_y<M, true>, smem);
    static const cudaError_t e1 = smem_attrs(k_ev_w_y<M, false>, smem);
    if (e0 != cudaSuccess) return e0;
    if (e1 != cudaSuccess) return e1;
    const int ntile = (v.WS + 4 * EvCfg<M>::C - 1) / (4 * EvCfg<M>::C), rows = v.nl < M ? v.nl : M;
    auto k = g.n_omega % 4 == 0 && reinterpret_cast<uintptr_t>(wts) % 16 == 0 ? k_ev_w_y<M, true> : k_ev_w_y<M, false>;
    return launch_after(k, rows * ntile, EvCfg<M>::T, smem, s, v, g.Q, g.n_omega, wts, (float *)w.X,
                        (const float2 *)w.evt, ntile);
}
template <int M>
cudaError_t launch_ev_chain_t(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, double *partial,
                              cudaStream_t s)
{
    const size_t smem = sizeof(float4) * EvFft<M, true>::SMEM_ELEMS;
    static const cudaError_t e = smem_attrs(k_ev_chain<M>, smem);
    if (e != cudaSuccess) return e;
    const int ntile = (v.ES + 4 * EvCfg<M>::C - 1) / (4 * EvCfg<M>::C);
    return launch_after(k_ev_chain<M>, v.Nh * ntile, EvCfg<M>::T, smem, s, g, v, band, w.axis, (const float2 *)w.eps,
                        w.state, (const float *)w.Y, partial, (const float2 *)w.evt, ntile);
}
// CTAs of k_ev_chain (rows of its partial sums).
int ev_chain_blocks(const EvGeom &v)
{
#define CALL(M_) v.Nh * ((v.ES + 4 * EvCfg<M_>::C - 1) / (4 * EvCfg<M_>::C))
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}
template <int L, bool FULL, bool THERMAL>
cudaError_t launch_ev_bw_t(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, const float *W2,
                           int sms, cudaStream_t s)
{
    using E = EvLine<L>;
    const size_t smem = sizeof(float2) * (EVC_WARPS * (E::WARP_ELEMS + 64 * (E::R1 + 1)) + (THERMAL ? L : 0));
    static const cudaError_t e = smem_attrs(k_ev_bw<L, FULL, THERMAL>, smem);
    if (e != cudaSuccess) return e;
    const int npairs = v.M / 2 * (v.M + 1) / 2, iters = ev_corr_iters(npairs, E::LPI, sms);
    const int per = EVC_WARPS * iters * E::LPI;
    return launch_after(k_ev_bw<L, FULL, THERMAL>, (npairs + per - 1) / per, 32 * EVC_WARPS, smem, s, g, v, band,
                        (const float *)w.Y, W2, (float *)w.X, (const float2 *)w.evt + ev_line_table<L>(), iters,
                        g.quantity == LINDHARD_IMCHI_T);
}
template <int L>
cudaError_t launch_ev_bw_l(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, const float *W2,
                           int sms, cudaStream_t s)
{
    if (g.quantity != LINDHARD_IMCHI) return launch_ev_bw_t<L, false, true>(g, v, band, w, W2, sms, s);
    if (v.ne == L && v.J0 == L / 2) return launch_ev_bw_t<L, true, false>(g, v, band, w, W2, sms, s);
    return launch_ev_bw_t<L, false, false>(g, v, band, w, W2, sms, s);
}
// Whether the adjoint has this form: the two-stage energy lengths.
bool ev_bw_applies(const EvGeom &v) { return v.M != 0 && v.PE <= 512; }
cudaError_t launch_ev_w_y(const Geom &g, const EvGeom &v, const float *wts, const Work<float> &w, cudaStream_t s)
{
#define CALL(M_) launch_ev_w_y_t<M_>(g, v, wts, w, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}
cudaError_t launch_ev_bw(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, const float *W2,
                         int sms, cudaStream_t s)
{
    switch (v.PE) {
    case 128: return launch_ev_bw_l<128>(g, v, band, w, W2, sms, s);
    case 256: return launch_ev_bw_l<256>(g, v, band, w, W2, sms, s);
    case 384: return launch_ev_bw_l<384>(g, v, band, w, W2, sms, s);
    case 512: return launch_ev_bw_l<512>(g, v, band, w, W2, sms, s);
    default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_ev_chain(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, double *partial,
                            cudaStream_t s)
{
#define CALL(M_) launch_ev_chain_t<M_>(g, v, band, w, partial, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}

}  // namespace lh
