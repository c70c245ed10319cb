// The even form (even.cuh) with the edge row and column p = -N/2 dp, which have
// no mirror on the grid, for bands whose form factor does not make them
// negligible (few zones, small or no ff_a; free electrons always).
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
// (tuned) -> this: 128^2 x 128 69 -> 53, 256^2 x 256 290 -> 126, all lags of
// 150^2 x 201 276 -> 105, 320^2 x 400 929 -> 309, 1024^2 x 512 8185 -> 3540; no
// grid was found on which the general form is the faster one.  The correlation
// there went from 1118 to 1039 us, at 512^2 x 256 from 247 to 139 us, with its
// products packed over two frequencies, the corner's spectrum in shared memory
// and the edge lines' loaded a step ahead.
#include "even.cuh"
#include "even_line.cuh"
#include "et_tiles.cuh"

namespace lh {

// A line's occupied and empty spectra at two frequencies k <= L/2 at once: row r
// of a lane's first and of its second butterfly (packed, one in each half).
struct EdgeLine { Cx2 occ, emp; };
__device__ __forceinline__ EdgeLine edge_separate(Cx2 k, Cx2 m)   // Z(k), Z(L - k); z holds the 1/2
{
    return {{add2(k.re, m.re), sub2(k.im, m.im)}, {add2(k.im, m.im), sub2(m.re, k.re)}};
}
// Z(L - k) for these: row r of the first butterfly mirrors row R1 - r (u = 0) or
// the second's R1 - 1 - r, row r of the second its own R1 - 1 - r (u = 0) or the
// first's.
template <int R1>
__device__ __forceinline__ Cx2 edge_mirror(const float2 *x, int r, bool u0)
{
    const float2 a = u0 ? x[(R1 - r) % R1] : x[R1 + R1 - 1 - r], b = u0 ? x[R1 + R1 - 1 - r] : x[R1 - 1 - r];
    return {make_float2(a.x, b.x), make_float2(a.y, b.y)};
}

// Energy spectra of the edge lines, separated; line t < M: a(k_t, e), line M:
// c(e).  A lane's values in the order of the correlation's registers: per line
// [R1 / 2][occupied, empty][TPL] packs, then [TPL] (occupied, empty) at L/2.
template <int L, bool THERMAL>
__global__ void __launch_bounds__(32 * EVC_WARPS, EvLine<L>::MINB)
k_ev_edge(Geom g, EvGeom v, Band band, const AxisTab *axis, const float2 *eps,
          const InstState *st, const float *B1, float4 *__restrict__ lines,
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
            const float2 e = eps[v.e0 + n];
            const float d = (e.x - q.x) + (e.y - q.y);
            raw[i] = q.z * rcp_approx(fmaf(d, d, band.gam2));
        }
    }
    float2 x[VPT];
    E::template first_stage<false, THERMAL>(x, raw, u, v.J0, wf);
    E::forward_rest(x, sm, u, tab);
    if (t > v.M) return;
    const bool u0 = u == 0;
    float4 *o = lines + (long long)t * (R1 + 1) * TPL + u;
#pragma unroll
    for (int r = 0; r < R1 / 2; ++r) {
        const EdgeLine q = edge_separate({make_float2(x[r].x, x[R1 + r].x), make_float2(x[r].y, x[R1 + r].y)},
                                         edge_mirror<R1>(x, r, u0));
        EvFft<16, false>::st(o + 2 * r * TPL, q.occ);
        EvFft<16, false>::st(o + (2 * r + 1) * TPL, q.emp);
    }
    const EdgeLine h = edge_separate({dup2(x[R1 / 2].x), dup2(x[R1 / 2].y)}, {dup2(x[R1 / 2].x), dup2(x[R1 / 2].y)});
    o[R1 * TPL] = make_float4(h.occ.re.x, h.occ.im.x, h.emp.re.x, h.emp.im.x);
}

// The four parity parts' spectra, twice each (in v.scale), from E^ and the edge
// lines there.  Packed over two frequencies: 80 instructions instead of 160.
struct EdgeParts { Cx2 ee, oo, ox, oy; };
__device__ __forceinline__ Cx2 edge_scaled(Cx2 a, float2 s) { return {mul2(a.re, s), mul2(a.im, s)}; }
__device__ __forceinline__ Cx2 edge_fma(Cx2 a, float2 s, Cx2 b) { return {fma2(a.re, s, b.re), fma2(a.im, s, b.im)}; }
// In program order (volatile): these are loaded a step ahead of their use.
// Loaded where they are used, each step waits for them (512^2 x 256 of two
// zones: 250 us instead of 149).
__device__ __forceinline__ Cx2 edge_load(const float4 *p)
{
    float4 q;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(q.x), "=f"(q.y), "=f"(q.z), "=f"(q.w) : "l"(p) : "memory");
    return {make_float2(q.x, q.y), make_float2(q.z, q.w)};
}
// conj(a) b + conj(c) d and conj(a) b - conj(c) d
__device__ __forceinline__ Cx2 edge_sum(Cx2 a, Cx2 b, Cx2 c, Cx2 d)
{
    return {fma2(c.im, d.im, fma2(c.re, d.re, fma2(a.im, b.im, mul2(a.re, b.re)))),
            sub2(fma2(c.re, d.im, mul2(a.re, b.im)), fma2(c.im, d.re, mul2(a.im, b.re)))};
}
__device__ __forceinline__ Cx2 edge_diff(Cx2 a, Cx2 b, Cx2 c, Cx2 d)
{
    return {sub2(fma2(a.im, b.im, mul2(a.re, b.re)), fma2(c.im, d.im, mul2(c.re, d.re))),
            sub2(fma2(c.im, d.re, mul2(a.re, b.im)), fma2(c.re, d.im, mul2(a.im, b.re)))};
}
template <bool THERMAL>
__device__ __forceinline__ EdgeParts edge_parts(EdgeLine e, EdgeLine ay, EdgeLine ax, EdgeLine c, float sx, float sy,
                                                bool odd)
{
    const float2 t = dup2(sx * sy), nt = neg2(t), px = dup2(sx), nx = neg2(px), py = dup2(sy);
    const Cx2 r1o = edge_fma(c.occ, nt, e.occ), r1u = edge_fma(c.emp, nt, e.emp);   // R at (k_x, k_y) and (-k_x, k_y)
    const Cx2 r2o = edge_fma(c.occ, t, e.occ), r2u = edge_fma(c.emp, t, e.emp);
    const Cx2 yo = edge_scaled(ax.occ, py), yu = edge_scaled(ax.emp, py);
    const Cx2 i1o = edge_fma(ay.occ, px, yo), i1u = edge_fma(ay.emp, px, yu);       // I there
    const Cx2 i2o = edge_fma(ay.occ, nx, yo), i2u = edge_fma(ay.emp, nx, yu);
    const Cx2 re1 = edge_sum(r1o, r1u, i1o, i1u), re2 = edge_sum(r2o, r2u, i2o, i2u);
    const Cx2 im1 = edge_diff(i1o, r1u, r1o, i1u), im2 = edge_diff(i2o, r2u, r2o, i2u);   // -Im
    EdgeParts p = {add(re1, re2), sub(re2, re1), sub(im1, im2), add(im1, im2)};
    if (THERMAL && odd) {
        // C(s, w) - C(-s, -w): the parts odd in one axis change sign with s
        p.ee = {dup2(0.f), add2(p.ee.im, p.ee.im)};
        p.oo = {dup2(0.f), add2(p.oo.im, p.oo.im)};
        p.ox = {add2(p.ox.re, p.ox.re), dup2(0.f)};
        p.oy = {add2(p.oy.re, p.oy.re), dup2(0.f)};
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
template <int L>
__host__ __device__ constexpr int ev_edge_corner()   // float2 of the corner's spectrum, one copy a CTA
{
    return 2 * (EvLine<L>::R1 + 1) * EvLine<L>::TPL;
}
template <int L, bool THERMAL, bool HALF>
__global__ void __launch_bounds__(32 * EVC_WARPS, EvLine<L>::MINB)
k_ev_edge_corr(Geom g, EvGeom v, Band band, const float *B2, const float4 *lines,
               float4 *__restrict__ B3, const float2 *__restrict__ tab, int iters, int odd)
{
    using E = EvLine<L>;
    constexpr int VPT = E::VPT, TPL = E::TPL, R0 = E::R0, R1 = E::R1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(EVC_WARPS * ev_edge_smem<L>() + ev_edge_corner<L>() + (THERMAL ? L : 0), float2)
    after_previous();
    const int lane = (int)threadIdx.x % 32, warp = (int)threadIdx.x / 32;
    const int sl = lane / TPL, u = lane % TPL;
    float2 *sm = reinterpret_cast<float2 *>(smem_raw) + warp * ev_edge_smem<L>() + sl * E::LP;
    float2 *own = reinterpret_cast<float2 *>(smem_raw) + warp * ev_edge_smem<L>() + E::WARP_ELEMS + lane;   // stride 32
    float4 *corner = reinterpret_cast<float4 *>(reinterpret_cast<float2 *>(smem_raw) + EVC_WARPS * ev_edge_smem<L>());
    float2 *wf = reinterpret_cast<float2 *>(smem_raw) + EVC_WARPS * ev_edge_smem<L>() + ev_edge_corner<L>();
    for (int i = threadIdx.x; i < (R1 + 1) * TPL; i += 32 * EVC_WARPS) corner[i] = lines[(long long)v.M * (R1 + 1) * TPL + i];
    if constexpr (THERMAL) et_fermi_weights<L>(g, band, wf, (int)threadIdx.x, 32 * EVC_WARPS);
    __syncthreads();
    const float *sines = reinterpret_cast<const float *>(lines) + ev_edge_lines(v);
    const int nlines = v.M * (v.M + 1) / 2;
    const bool u0 = u == 0;
    // (one wave of CTAs with an equal share each: 320^2 x 400 138 us instead of 121)
    for (int it = 0; it < iters; ++it) {
        const int t = ((blockIdx.x * EVC_WARPS + warp) * iters + it) * E::LPI + sl;
        const bool live = t < nlines;
        int kx, ky;
        ev_tri(live ? t : 0, v.M, kx, ky);
        float raw[VPT];
        const float *p = B2 + (kx * v.s2 + (long long)ky * v.ES + u);
#pragma unroll
        for (int i = 0; i < VPT; ++i) raw[i] = live && u + E::first(i) < v.ne ? __ldcs(p + E::first(i)) : 0.f;
        const float sx = sines[kx], sy = sines[ky];
        const float4 *ly = lines + (long long)ky * (R1 + 1) * TPL + u, *lx = lines + (long long)kx * (R1 + 1) * TPL + u;
        float2 x[VPT];
        E::template first_stage<false, THERMAL>(x, raw, u, v.J0, wf);
        E::forward_rest(x, sm, u, tab);
        auto line = [&](const float4 *l, int r) { return EdgeLine{edge_load(l + 2 * r * TPL), edge_load(l + (2 * r + 1) * TPL)}; };
        auto line_c = [&](int r) {
            return EdgeLine{EvFft<16, false>::ld(corner + 2 * r * TPL + u), EvFft<16, false>::ld(corner + (2 * r + 1) * TPL + u)};
        };
        auto half = [&](float4 q) { return EdgeLine{{dup2(q.x), dup2(q.y)}, {dup2(q.z), dup2(q.w)}}; };
        // P1 + i P2 at k, conj P1 + i conj P2 at L - k
        auto w_of = [](Cx2 p, Cx2 q) { return Cx2{sub2(p.re, q.im), add2(p.im, q.re)}; };
        auto w_conj = [](Cx2 p, Cx2 q) { return Cx2{add2(p.re, q.im), sub2(q.re, p.im)}; };
        // frequencies k <= L/2 and their mirrors, in place (edge_mirror's rows)
        EdgeLine ny = line(ly, 0), nx = line(lx, 0);
#pragma unroll
        for (int r = 0; r < R1 / 2; ++r) {
            const EdgeLine e = edge_separate({make_float2(x[r].x, x[R1 + r].x), make_float2(x[r].y, x[R1 + r].y)},
                                             edge_mirror<R1>(x, r, u0));
            const EdgeLine cy = ny, cx = nx;
            if (r + 1 < R1 / 2) { ny = line(ly, r + 1); nx = line(lx, r + 1); }
            const EdgeParts p = edge_parts<THERMAL>(e, cy, cx, line_c(r), sx, sy, odd != 0);
            const Cx2 k1 = w_of(p.ee, p.oy), m1 = w_conj(p.ee, p.oy), k2 = w_of(p.ox, p.oo), m2 = w_conj(p.ox, p.oo);
            const float2 ac = make_float2(m1.re.x, m1.im.x), bc = make_float2(m1.re.y, m1.im.y);
            x[r] = make_float2(k1.re.x, k1.im.x);
            x[R1 + r] = make_float2(k1.re.y, k1.im.y);
            x[R1 + R1 - 1 - r] = u0 ? bc : ac;
            if (r > 0) x[R1 - r] = u0 ? ac : x[R1 - r];
            x[R1 - 1 - r] = u0 ? x[R1 - 1 - r] : bc;
            own[32 * (u0 ? (R1 - r) % R1 : R1 + R1 - 1 - r)] = make_float2(m2.re.x, m2.im.x);
            own[32 * (u0 ? R1 + R1 - 1 - r : R1 - 1 - r)] = make_float2(m2.re.y, m2.im.y);
            own[32 * r] = make_float2(k2.re.x, k2.im.x);
            own[32 * (R1 + r)] = make_float2(k2.re.y, k2.im.y);
        }
        if (u0) {   // k = L/2
            const Cx2 z = {dup2(x[R1 / 2].x), dup2(x[R1 / 2].y)};
            const EdgeParts p = edge_parts<THERMAL>(edge_separate(z, z), half(ly[R1 * TPL]), half(lx[R1 * TPL]),
                                                    half(corner[R1 * TPL + u]), sx, sy, odd != 0);
            const Cx2 k1 = w_of(p.ee, p.oy), k2 = w_of(p.ox, p.oo);
            x[R1 / 2] = make_float2(k1.re.x, k1.im.x);
            own[32 * (R1 / 2)] = make_float2(k2.re.x, k2.im.x);
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

// Both signs of every lag l of the window from the even parts D_l (re) and the
// odd S_l = D_{M-l} (im; S_0 = 0), out at o + (Q/2 +- l) stride.  One code for
// all units of a warp: unit 0's mirrors lie in its own butterflies (ev_pairs),
// selected, where a branch had each such warp run both sides.
template <int M, typename T, typename F>
__device__ __forceinline__ void edge_lags(const Cx2 *z, int u, int Q, T *o, long long stride, F &&store)
{
    constexpr int RP = ev_vpt(M) / 2, NBP = M / RP, TPC = M / ev_vpt(M);
    const bool u0 = u == 0;
    const int h = Q / 2;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const int j = b == 0 ? u : (u0 ? TPC : NBP - u);
        T *pp = o + (h + j) * stride, *pm = o + (h - j) * stride;
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            const int l = j + r * NBP;
            const float2 other = z[(1 - b) * RP + RP - 1 - r].im;
            const float2 self = b == 1 ? z[RP + RP - 1 - r].im : r == 0 ? make_float2(0.f, 0.f) : z[(RP - r) % RP].im;
            const float2 even = z[b * RP + r].re, odd = u0 ? self : other;
            if (l < h) store(pp + r * NBP * stride, add2(even, odd));
            if ((b != 0 || r != 0 || !u0) && l <= h) store(pm - r * NBP * stride, sub2(even, odd));
        }
    }
}

// B3 (EE, OY, OX, OO of k_x <= k_y) -> B4 [Q][M][WS]: the even and the odd part
// along y (x, y of a value) at every lag s_x of the window.  Grid: M x (column
// tiles), a pack is one transfer.
template <int M>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_ev_edge_inv_x(EvGeom v, int Q, const float *B3, float2 *__restrict__ B4,
                const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, true>;
    constexpr int C = F::C, VPT = F::VPT, TPC = F::TPC, RF = F::RF;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float4)
    after_previous();
    float4 *sm = reinterpret_cast<float4 *>(smem_raw);
    const int ky = blockIdx.x / ntile, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;
    const int m = ct * C + col;
    const bool on = m < v.WS;
    const unsigned S3 = (unsigned)(v.s3 / 4);   // M S3 < 2^32 for every length and transfer count
    Cx2 z[VPT];
#pragma unroll
    for (int b = 0; b < VPT / RF; ++b)
#pragma unroll
        for (int r = 0; r < RF; ++r) {
            // (EE, OY) even in x, (OX, OO) odd; above the diagonal the axes change places
            const int kx = u + b * TPC + r * (M / RF);
            const bool below = kx <= ky;
            const Cx2 q = on ? ev_load(B3 + 4 * (size_t)(below ? kx * S3 + (ky * v.WS + m) : ky * S3 + (kx * v.WS + m)))
                             : Cx2{dup2(0.f), dup2(0.f)};
            const float oy = below ? q.re.y : q.im.x, ox = below ? q.im.x : q.re.y;
            const bool up = RF % 2 == 0 ? r >= RF / 2 : kx >= M / 2;
            z[b * RF + r] = {make_float2(q.re.x, oy), up ? make_float2(-ox, -q.im.y) : make_float2(ox, q.im.y)};
        }
    F::run(z, sm + col, u, tab);
    ev_post<M>(z, u, tab);
    if (!on) return;
    const long long s4 = v.s4 / 2;
    float2 *o = B4 + ((long long)ky * v.WS + m);
    edge_lags<M>(z, u, Q, o, s4, [](float2 *p, float2 c) { *p = c; });
    // lag -M of grids that keep it (Q = 2N = 2M): no pair of points is that far apart
    if (u == 0 && Q / 2 == M) o[0] = make_float2(0.f, 0.f);
}

// B4 -> Im chi at the lags (s_x, +-s_y), times the Eq. 9 prefactor.  Grid: Q x
// (column tiles), a pack is two transfers.  VEC: both in one 8-byte store.
template <int M, bool VEC>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_ev_edge_inv_y(EvGeom v, int Q, int n_omega, const float *B4, float *__restrict__ out,
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
            const bool up = RF % 2 == 0 ? r >= RF / 2 : ky >= M / 2;
            z[b * RF + r] = {make_float2(q.re.x, q.im.x), up ? make_float2(-q.re.y, -q.im.y) : make_float2(q.re.y, q.im.y)};
        }
    F::run(z, sm + col, u, tab);
    ev_post<M>(z, u, tab);
    if (m >= n_omega) return;
    float *o = out + ((long long)row * Q + Q / 2) * n_omega + m;
    const float2 sc = dup2(v.scale);
    auto store = [&](float *q, float2 c) {
        if constexpr (VEC) {
            *reinterpret_cast<float2 *>(q) = c;
        } else {
            q[0] = c.x;
            if (m + 1 < n_omega) q[1] = c.y;
        }
    };
#pragma unroll
    for (int i = 0; i < VPT; ++i) z[i] = {mul2(z[i].re, sc), mul2(z[i].im, sc)};
    edge_lags<M>(z, u, Q, o - (long long)(Q / 2) * n_omega, n_omega, store);
    if (u == 0 && Q / 2 == M) store(o - (long long)M * n_omega, make_float2(0.f, 0.f));
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
    const size_t smem = sizeof(float2) * (EVC_WARPS * ev_edge_smem<L>() + ev_edge_corner<L>() + (THERMAL ? L : 0));
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
