// The even form (even.cuh) with the edge row and column p = -N/2 dp, which have
// no mirror on the grid, for bands whose form factor does not make them
// negligible (few zones, small or no ff_a).
//
// With half of the edge's weight put on either end of an axis, A = E + O: E
// even, and O odd but on the edge alone.  With theta = 2 pi (k + 1/2) / P,
// s_k = sin(N theta_k / 2), a(k_y, e) the cosine transform of the edge column
// and c(e) the corner,
//
//   A^(k_x, k_y, e) = R + i I,  R = E^ - C,  I = X + Y,
//   C = s_x s_y c(e), X = s_x a(k_y, e), Y = s_y a(k_x, e),
//
// so the edge adds M + 1 energy lines, transformed once (k_ev_edge), and no
// second momentum transform forward.  A^ at the mirrored frequency (-k_x, k_y)
// is the same with C and X negated.  The energy correlation at both,
// Re = R (x) R + I (x) I and Im = R (x) I - I (x) R ((x): occupied conjugated
// times empty, Eq. 9), gives the four parity parts of the spectrum at k_x <=
// k_y, which the inverse takes by cosine transforms along the axes on which a
// part is even and by sine transforms along the others:
//
//   C(+-s_x, +-s_y) = EE +- OX +- OY (+-)(+-) OO.
//
// A sine transform is the cosine transform of the values with every second
// sign changed, read backwards, S_j = D_{M-j}: in this form's order the upper
// half of the rows changes sign, and rows j and M - j end in one thread.  So
// one complex column carries a cosine part (re) and a sine part (im).
//
// Against the general form (full grid, complex): half of the energy
// transforms, no transform of A's mirror images, and B2 and B3, B4 of M^2
// instead of P^2 frequencies.  Measured us a call without form factor, general
// (tuned) -> this: 128^2 x 128 69 -> 54, 256^2 x 256 290 -> 145, all lags of
// 150^2 x 201 276 -> 125, Im chi_T of 288^2 x 200 697 -> 259, 1024^2 x 512 8185
// -> 3740; no grid was found on which the general form is the faster one.
#include "even.cuh"
#include "even_line.cuh"
#include "et_tiles.cuh"

namespace lh {

// Energy spectra of the edge lines, separated (occupied re, im, empty re, im),
// line t < M: a(k_t, e), line M: c(e).  A lane's values in the order of the
// correlation's registers, [line][R1 + 1][TPL]: its frequencies k <= L/2.
template <int L, bool THERMAL>
__global__ void __launch_bounds__(32 * EVC_WARPS, EvLine<L>::MINB)
k_ev_edge(Geom g, EvGeom v, Band band, const AxisTab *__restrict__ axis, const float2 *__restrict__ eps,
          const InstState *__restrict__ st, const float *__restrict__ B1, float4 *__restrict__ lines,
          const float2 *__restrict__ tab)
{
    using E = EvLine<L>;
    constexpr int VPT = E::VPT, TPL = E::TPL, R1 = E::R1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(EVC_WARPS * E::WARP_ELEMS + (THERMAL ? L : 0), float2)
    after_previous();
    const int lane = (int)threadIdx.x % 32, warp = (int)threadIdx.x / 32;
    const int sl = lane / TPL, u = lane % TPL;
    float2 *sm = reinterpret_cast<float2 *>(smem_raw) + warp * E::WARP_ELEMS + sl * E::LP;
    float2 *wf = reinterpret_cast<float2 *>(smem_raw) + EVC_WARPS * E::WARP_ELEMS;
    if constexpr (THERMAL) {
        et_fermi_weights<L>(g, band, wf, (int)threadIdx.x, 32 * EVC_WARPS);
        __syncthreads();
    }
    // sin(N theta_k / 2) of row n: k = 2n below M/2, 2 (M - 1 - n) + 1 above
    float *sines = reinterpret_cast<float *>(lines) + ev_edge_lines(v);
    for (int n = blockIdx.x * 32 * EVC_WARPS + threadIdx.x; n < v.M; n += gridDim.x * 32 * EVC_WARPS) {
        const int k = n < v.M / 2 ? 2 * n : 2 * (v.M - 1 - n) + 1;
        const long long q = (long long)g.N * (2 * k + 1) % (8LL * v.M);
        sines[n] = (float)sinpi((double)q / (4.0 * v.M));
    }
    const int t = (blockIdx.x * EVC_WARPS + warp) * E::LPI + sl;
    float raw[VPT];
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t == v.M) band_point_f32(band, axis[0], axis[0], st, q.x, q.y, q.z);
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int n = u + E::first(i);
        raw[i] = 0.f;
        if (t < v.M && n < v.ne) raw[i] = 2.f * B1[(v.Nh - 1) * v.s1 + (long long)t * v.ES + n];
        if (t == v.M && n < v.ne) {
            const float2 e = __ldg(&eps[v.e0 + n]);
            const float d = (e.x - q.x) + (e.y - q.y);
            raw[i] = q.z * ev_rcp(fmaf(d, d, band.gam2));
        }
    }
    float2 x[VPT];
    E::template first_stage<false, THERMAL>(x, raw, u, v.J0, wf);
    E::forward_rest(x, sm, u, tab);
    if (t > v.M) return;
    const bool u0 = u == 0;
    float4 *o = lines + (long long)t * (R1 + 1) * TPL + u;
    auto sep = [](float2 zk, float2 zm) { return make_float4(zk.x + zm.x, zk.y - zm.y, zk.y + zm.y, zm.x - zk.x); };
#pragma unroll
    for (int r = 0; r < R1 / 2; ++r) {
        o[r * TPL] = sep(x[r], u0 ? x[(R1 - r) % R1] : x[R1 + R1 - 1 - r]);
        o[(R1 / 2 + r) * TPL] = sep(x[R1 + r], u0 ? x[R1 + R1 - 1 - r] : x[R1 - 1 - r]);
    }
    o[R1 * TPL] = sep(x[R1 / 2], x[R1 / 2]);
}

// The four parity parts' spectra at one energy frequency from E^ and the edge
// lines there: (EE, OY) and (OX, OO), twice each (in v.scale).
struct EdgeParts { float2 ee, oo, ox, oy; };
template <bool THERMAL>
__device__ __forceinline__ EdgeParts ev_edge_parts(float4 e, float4 ay, float4 ax, float4 c, float sx, float sy, bool odd)
{
    const float t = sx * sy;
    const float2 eo = make_float2(e.x, e.y), eu = make_float2(e.z, e.w);
    const float2 co = make_float2(t * c.x, t * c.y), cu = make_float2(t * c.z, t * c.w);
    const float2 xo = make_float2(sx * ay.x, sx * ay.y), xu = make_float2(sx * ay.z, sx * ay.w);
    const float2 yo = make_float2(sy * ax.x, sy * ax.y), yu = make_float2(sy * ax.z, sy * ax.w);
    const float2 r1o = csub(eo, co), r1u = csub(eu, cu), r2o = cadd(eo, co), r2u = cadd(eu, cu);
    const float2 i1o = cadd(yo, xo), i1u = cadd(yu, xu), i2o = csub(yo, xo), i2u = csub(yu, xu);
    const float2 re1 = cadd(cmulc(r1u, r1o), cmulc(i1u, i1o)), re2 = cadd(cmulc(r2u, r2o), cmulc(i2u, i2o));
    const float2 im1 = csub(cmulc(r1u, i1o), cmulc(i1u, r1o)), im2 = csub(cmulc(r2u, i2o), cmulc(i2u, r2o));   // -Im
    EdgeParts p = {cadd(re1, re2), csub(re2, re1), csub(im1, im2), cadd(im1, im2)};
    if (THERMAL && odd) {
        // C(s, w) - C(-s, -w): the parts odd in one axis change sign with s
        p.ee = make_float2(0.f, p.ee.y + p.ee.y);
        p.oo = make_float2(0.f, p.oo.y + p.oo.y);
        p.ox = make_float2(p.ox.x + p.ox.x, 0.f);
        p.oy = make_float2(p.oy.x + p.oy.x, 0.f);
    }
    return p;
}

// Energy correlation of each line k_x <= k_y: one transform forward and two
// inverse, of EE + i OY and OX + i OO.  The second waits in the lane's own
// places in shared memory (a second set of VPT registers halved the warps).
// HALF: WS <= L/2, the upper half of the lags is not formed.
template <int L>
__host__ __device__ constexpr int ev_edge_smem()   // float2 of a warp
{
    return EvLine<L>::WARP_ELEMS + 32 * EvLine<L>::VPT;
}
template <int L, bool THERMAL, bool HALF>
__global__ void __launch_bounds__(32 * EVC_WARPS, EvLine<L>::MINB)
k_ev_edge_corr(Geom g, EvGeom v, Band band, const float *__restrict__ B2, const float4 *__restrict__ lines,
               float4 *__restrict__ B3, const float2 *__restrict__ tab, int iters, int odd)
{
    using E = EvLine<L>;
    constexpr int VPT = E::VPT, TPL = E::TPL, R0 = E::R0, R1 = E::R1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(EVC_WARPS * ev_edge_smem<L>() + (THERMAL ? L : 0), float2)
    after_previous();
    const int lane = (int)threadIdx.x % 32, warp = (int)threadIdx.x / 32;
    const int sl = lane / TPL, u = lane % TPL;
    float2 *sm = reinterpret_cast<float2 *>(smem_raw) + warp * ev_edge_smem<L>() + sl * E::LP;
    float2 *own = reinterpret_cast<float2 *>(smem_raw) + warp * ev_edge_smem<L>() + E::WARP_ELEMS + lane;   // stride 32
    float2 *wf = reinterpret_cast<float2 *>(smem_raw) + EVC_WARPS * ev_edge_smem<L>();
    if constexpr (THERMAL) {
        et_fermi_weights<L>(g, band, wf, (int)threadIdx.x, 32 * EVC_WARPS);
        __syncthreads();
    }
    const float *sines = reinterpret_cast<const float *>(lines) + ev_edge_lines(v);
    const int nlines = v.M * (v.M + 1) / 2;
    const bool u0 = u == 0;
    auto w_of = [](float2 x1, float2 x2) { return make_float2(x1.x - x2.y, x1.y + x2.x); };      // P1 + i P2
    auto w_conj = [](float2 x1, float2 x2) { return make_float2(x1.x + x2.y, x2.x - x1.y); };    // conj P1 + i conj P2
    auto sep = [](float2 zk, float2 zm) { return make_float4(zk.x + zm.x, zk.y - zm.y, zk.y + zm.y, zm.x - zk.x); };

    for (int it = 0; it < iters; ++it) {
        const int t = ((blockIdx.x * EVC_WARPS + warp) * iters + it) * E::LPI + sl;
        const bool live = t < nlines;
        int kx, ky;
        ev_tri(live ? t : 0, v.M, kx, ky);
        float raw[VPT];
        const float *p = B2 + (kx * v.s2 + (long long)ky * v.ES + u);
#pragma unroll
        for (int i = 0; i < VPT; ++i) raw[i] = live && u + E::first(i) < v.ne ? __ldcs(p + E::first(i)) : 0.f;
        const float sx = __ldg(sines + kx), sy = __ldg(sines + ky);
        const float4 *ly = lines + (long long)ky * (R1 + 1) * TPL + u, *lx = lines + (long long)kx * (R1 + 1) * TPL + u,
                     *lc = lines + (long long)v.M * (R1 + 1) * TPL + u;
        float2 x[VPT];
        E::template first_stage<false, THERMAL>(x, raw, u, v.J0, wf);
        E::forward_rest(x, sm, u, tab);
        auto parts = [&](int j, float2 zk, float2 zm) {
            return ev_edge_parts<THERMAL>(sep(zk, zm), __ldg(ly + j * TPL), __ldg(lx + j * TPL), __ldg(lc + j * TPL), sx, sy,
                                          odd != 0);
        };
        // Frequencies k <= L/2 and their mirrors, in place: row r of the first
        // butterfly mirrors row R1 - r (u = 0) or the second's R1 - 1 - r, row r
        // of the second its own R1 - 1 - r (u = 0) or the first's.
#pragma unroll
        for (int r = 0; r < R1 / 2; ++r) {
            const EdgeParts a = parts(r, x[r], u0 ? x[(R1 - r) % R1] : x[R1 + R1 - 1 - r]);
            const EdgeParts b = parts(R1 / 2 + r, x[R1 + r], u0 ? x[R1 + R1 - 1 - r] : x[R1 - 1 - r]);
            const float2 ac = w_conj(a.ee, a.oy), bc = w_conj(b.ee, b.oy);
            x[r] = w_of(a.ee, a.oy);
            x[R1 + r] = w_of(b.ee, b.oy);
            x[R1 + R1 - 1 - r] = u0 ? bc : ac;
            if (r > 0) x[R1 - r] = u0 ? ac : x[R1 - r];
            x[R1 - 1 - r] = u0 ? x[R1 - 1 - r] : bc;
            own[32 * (u0 ? (R1 - r) % R1 : R1 + R1 - 1 - r)] = w_conj(a.ox, a.oo);
            own[32 * (u0 ? R1 + R1 - 1 - r : R1 - 1 - r)] = w_conj(b.ox, b.oo);
            own[32 * r] = w_of(a.ox, a.oo);
            own[32 * (R1 + r)] = w_of(b.ox, b.oo);
        }
        if (u0) {   // k = L/2
            const EdgeParts a = parts(R1, x[R1 / 2], x[R1 / 2]);
            x[R1 / 2] = w_of(a.ee, a.oy);
            own[32 * (R1 / 2)] = w_of(a.ox, a.oo);
        }
        E::inverse(x, sm, u, tab);
#pragma unroll
        for (int i = 0; i < VPT; ++i) {
            const float2 w = own[32 * i];
            own[32 * i] = x[i];
            x[i] = w;
        }
        E::inverse(x, sm, u, tab);
        if (live) {
            float4 *o = B3 + (kx * (v.s3 / 4) + (long long)ky * v.WS + u);
#pragma unroll
            for (int i = 0; i < VPT; ++i) {
                const int m = E::last(i);
                if ((!HALF || i % R0 < R0 / 2) && u + m < v.WS) {   // the row's padding too: finite values (WS <= L)
                    const float2 w = own[32 * i];
                    o[m] = make_float4(w.x, w.y, x[i].x, x[i].y);
                }
            }
        }
    }
}

// B3 (EE, OY, OX, OO of k_x <= k_y) -> B4 [Q][M][WS]: the even and the odd part
// along y (x, y of a value) at every lag s_x of the window.  Grid: M x (column
// tiles), a pack is one transfer.
template <int M>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_ev_edge_inv_x(EvGeom v, int Q, const float *__restrict__ B3, float2 *__restrict__ B4,
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
    const int m = ct * C + col;
    const bool on = m < v.WS;
    Cx2 z[VPT];
#pragma unroll
    for (int b = 0; b < VPT / RF; ++b)
#pragma unroll
        for (int r = 0; r < RF; ++r) {
            const int kx = u + b * TPC + r * (M / RF), lo = min(kx, ky), hi = max(kx, ky);
            // (EE, OY) even in x, (OX, OO) odd; above the diagonal the axes change places
            const Cx2 q = on ? ev_load(B3 + lo * v.s3 + 4LL * (hi * v.WS + m)) : Cx2{dup2(0.f), dup2(0.f)};
            const float oy = kx <= ky ? q.re.y : q.im.x, ox = kx <= ky ? q.im.x : q.re.y;
            z[b * RF + r] = {make_float2(q.re.x, oy), kx < M / 2 ? make_float2(ox, q.im.y) : make_float2(-ox, -q.im.y)};
        }
    F::run(z, sm + col, u, tab);
    ev_post<M>(z, u, tab);
    if (!on) return;
    float2 *o = B4 + ((long long)ky * v.WS + m);
    const long long s4 = v.s4 / 2;
    auto put = [&](int l, float2 even, float2 oddv) {
        if (l < Q / 2) o[(Q / 2 + l) * s4] = add2(even, oddv);
        if (l > 0 && l <= Q / 2) o[(Q / 2 - l) * s4] = sub2(even, oddv);
    };
    ev_pairs<RP, NBP, TPC>(z, u, [&](int n, Cx2 &a, Cx2 &b) {
        put(n, a.re, n == 0 ? make_float2(0.f, 0.f) : b.im);
        if (&a != &b) put(M - n, b.re, a.im);
    });
    // lag -M of grids that keep it (Q = 2N = 2M): no pair of points is that far apart
    if (u == 0 && Q / 2 == M) o[0] = make_float2(0.f, 0.f);
}

// B4 -> Im chi at the lags (s_x, +-s_y), times the Eq. 9 prefactor.  Grid: Q x
// (column tiles), a pack is two transfers.  VEC: both in one 8-byte store.
template <int M, bool VEC>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_ev_edge_inv_y(EvGeom v, int Q, int n_omega, const float *__restrict__ B4, float *__restrict__ out,
                const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, true>;
    constexpr int C = F::C, VPT = F::VPT, TPC = F::TPC, RP = F::RP, NBP = F::NBP, RF = F::RF;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float4)
    after_previous();
    float4 *sm = reinterpret_cast<float4 *>(smem_raw);
    const int row = blockIdx.x / ntile, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;
    const int m = 2 * (ct * C + col);
    const bool on = m < v.WS;
    const float *in = B4 + row * v.s4 + 2 * m;
    Cx2 z[VPT];
#pragma unroll
    for (int b = 0; b < VPT / RF; ++b)
#pragma unroll
        for (int r = 0; r < RF; ++r) {
            const int ky = u + b * TPC + r * (M / RF);
            const Cx2 q = on ? ev_load(in + 2 * ky * v.WS) : Cx2{dup2(0.f), dup2(0.f)};
            z[b * RF + r] = {make_float2(q.re.x, q.im.x),
                             ky < M / 2 ? make_float2(q.re.y, q.im.y) : make_float2(-q.re.y, -q.im.y)};
        }
    F::run(z, sm + col, u, tab);
    ev_post<M>(z, u, tab);
    if (m >= n_omega) return;
    float *o = out + ((long long)row * Q + Q / 2) * n_omega + m;
    const float2 sc = dup2(v.scale);
    auto store = [&](int l, float2 c) {
        float *q = o + (long long)l * n_omega;
        if constexpr (VEC) {
            *reinterpret_cast<float2 *>(q) = c;
        } else {
            q[0] = c.x;
            if (m + 1 < n_omega) q[1] = c.y;
        }
    };
    auto put = [&](int l, float2 even, float2 oddv) {
        if (l < Q / 2) store(l, mul2(add2(even, oddv), sc));
        if (l > 0 && l <= Q / 2) store(-l, mul2(sub2(even, oddv), sc));
    };
    ev_pairs<RP, NBP, TPC>(z, u, [&](int n, Cx2 &a, Cx2 &b) {
        put(n, a.re, n == 0 ? make_float2(0.f, 0.f) : b.im);
        if (&a != &b) put(M - n, b.re, a.im);
    });
    if (u == 0 && Q / 2 == M) store(-M, make_float2(0.f, 0.f));
}

template <int L, bool THERMAL>
cudaError_t launch_ev_edge_t(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, cudaStream_t s)
{
    using E = EvLine<L>;
    const size_t smem = sizeof(float2) * (EVC_WARPS * E::WARP_ELEMS + (THERMAL ? L : 0));
    static const cudaError_t e = smem_attrs(k_ev_edge<L, THERMAL>, smem);
    if (e != cudaSuccess) return e;
    const int per = EVC_WARPS * E::LPI;
    return launch_after(k_ev_edge<L, THERMAL>, (v.M + 1 + per - 1) / per, 32 * EVC_WARPS, smem, s, g, v, band, w.axis,
                        (const float2 *)w.eps, w.state, (const float *)w.X, (float4 *)((float *)w.Y + v.M * v.s2),
                        (const float2 *)w.evt + ev_line_table<L>());
}
template <int L, bool THERMAL, bool HALF>
cudaError_t launch_ev_edge_corr_t(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, int sms,
                                  cudaStream_t s)
{
    using E = EvLine<L>;
    const size_t smem = sizeof(float2) * (EVC_WARPS * ev_edge_smem<L>() + (THERMAL ? L : 0));
    static const cudaError_t e = smem_attrs(k_ev_edge_corr<L, THERMAL, HALF>, smem);
    if (e != cudaSuccess) return e;
    const int nlines = v.M * (v.M + 1) / 2, iters = ev_corr_iters(nlines, E::LPI, sms);
    const int per = EVC_WARPS * iters * E::LPI;
    return launch_after(k_ev_edge_corr<L, THERMAL, HALF>, (nlines + per - 1) / per, 32 * EVC_WARPS, smem, s, g, v, band,
                        (const float *)w.Y, (const float4 *)((const float *)w.Y + v.M * v.s2), (float4 *)w.X,
                        (const float2 *)w.evt + ev_line_table<L>(), iters, (int)(g.quantity == LINDHARD_IMCHI_T));
}
template <int L>
cudaError_t launch_ev_edge_corr_l(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, int sms,
                                  cudaStream_t s)
{
    const bool half = v.WS <= L / 2;
    if (g.quantity != LINDHARD_IMCHI)
        return half ? launch_ev_edge_corr_t<L, true, true>(g, v, band, w, sms, s)
                    : launch_ev_edge_corr_t<L, true, false>(g, v, band, w, sms, s);
    return half ? launch_ev_edge_corr_t<L, false, true>(g, v, band, w, sms, s)
                : launch_ev_edge_corr_t<L, false, false>(g, v, band, w, sms, s);
}
template <int M>
cudaError_t launch_ev_edge_inv_x_t(const Geom &g, const EvGeom &v, const Work<float> &w, cudaStream_t s)
{
    const size_t smem = sizeof(float4) * EvFft<M, true>::SMEM_ELEMS;
    static const cudaError_t e = smem_attrs(k_ev_edge_inv_x<M>, smem);
    if (e != cudaSuccess) return e;
    const int ntile = (v.WS + EvCfg<M>::C - 1) / EvCfg<M>::C;
    return launch_after(k_ev_edge_inv_x<M>, M * ntile, EvCfg<M>::T, smem, s, v, g.Q, (const float *)w.X, (float2 *)w.Y,
                        (const float2 *)w.evt, ntile);
}
template <int M>
cudaError_t launch_ev_edge_inv_y_t(const Geom &g, const EvGeom &v, const Work<float> &w, float *out, cudaStream_t s)
{
    const size_t smem = sizeof(float4) * EvFft<M, true>::SMEM_ELEMS;
    static const cudaError_t e0 = smem_attrs(k_ev_edge_inv_y<M, true>, smem);
    static const cudaError_t e1 = smem_attrs(k_ev_edge_inv_y<M, false>, smem);
    if (e0 != cudaSuccess) return e0;
    if (e1 != cudaSuccess) return e1;
    const int ntile = (v.WS / 2 + EvCfg<M>::C - 1) / EvCfg<M>::C;
    auto k = g.n_omega % 2 == 0 && reinterpret_cast<uintptr_t>(out) % 8 == 0 ? k_ev_edge_inv_y<M, true>
                                                                              : k_ev_edge_inv_y<M, false>;
    return launch_after(k, g.Q * ntile, EvCfg<M>::T, smem, s, v, g.Q, g.n_omega, (const float *)w.Y, out,
                        (const float2 *)w.evt, ntile);
}

cudaError_t launch_ev_edge(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, cudaStream_t s)
{
    const bool th = g.quantity != LINDHARD_IMCHI;
    switch (v.PE) {
    case 128: return th ? launch_ev_edge_t<128, true>(g, v, band, w, s) : launch_ev_edge_t<128, false>(g, v, band, w, s);
    case 256: return th ? launch_ev_edge_t<256, true>(g, v, band, w, s) : launch_ev_edge_t<256, false>(g, v, band, w, s);
    case 384: return th ? launch_ev_edge_t<384, true>(g, v, band, w, s) : launch_ev_edge_t<384, false>(g, v, band, w, s);
    case 512: return th ? launch_ev_edge_t<512, true>(g, v, band, w, s) : launch_ev_edge_t<512, false>(g, v, band, w, s);
    default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_ev_edge_corr(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, int sms,
                                cudaStream_t s)
{
    switch (v.PE) {
    case 128: return launch_ev_edge_corr_l<128>(g, v, band, w, sms, s);
    case 256: return launch_ev_edge_corr_l<256>(g, v, band, w, sms, s);
    case 384: return launch_ev_edge_corr_l<384>(g, v, band, w, sms, s);
    case 512: return launch_ev_edge_corr_l<512>(g, v, band, w, sms, s);
    default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_ev_edge_inv_x(const Geom &g, const EvGeom &v, const Work<float> &w, cudaStream_t s)
{
#define CALL(M_) launch_ev_edge_inv_x_t<M_>(g, v, w, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}
cudaError_t launch_ev_edge_inv_y(const Geom &g, const EvGeom &v, const Work<float> &w, float *out, cudaStream_t s)
{
#define CALL(M_) launch_ev_edge_inv_y_t<M_>(g, v, w, out, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}

}  // namespace lh
