// The even form of the correlation: geometry, buffers and the column engine of
// its momentum passes (k_even_fwd.cu, k_even_corr.cu, k_even_inv.cu).
//
// A generated A(p, e) (Eqs. 4-5) is real, even in p_x and in p_y and symmetric
// under their exchange: both bands depend on p through cos p and cos 2p, or
// p^2.  So instead of complex transforms over all of (p, e) with the energy
// axis first, this form transforms the momentum axes first, as cosine
// transforms of one quadrant, and does the energy correlation of Eq. 9 on the
// real spectra that come out:
//
//   A(p_x, p_y, e)  p >= 0          generated      N/2 x N/2 x n_eps reals
//   -> cosine transform along p_y, then p_x        M x M x n_eps, k_x <= k_y kept
//   -> energy correlation per (k_x, k_y), k_x <= k_y  (FFT along e)  x n_omega
//   -> inverse cosine transform along k_x, k_y     lags s >= 0
//   -> Im chi at the four lags (+-s_x, +-s_y)
//
// with M >= (N + Q/2) / 2 frequencies per axis.  At 1024^2 x 512 the buffers
// move 5.3 GB instead of the general form's 33.4 GB and the momentum
// transforms take 0.38 G complex points (two real columns a point) instead of
// 3.4 G: 8.19 -> 1.50 ms a call (256^3: 0.279 -> 0.065 ms; Im chi_T there
// 0.412 -> 0.074 ms).
//
// Transform.  The frequencies are theta_k = pi (2k + 1) / (2M), the
// half-shifted grid of length P = 2M: it turns the circular correlation of
// length P into the one whose wrapped terms change sign, which is as good
// here (P >= N + Q/2: no wrapped term reaches a kept lag) and makes both
// directions square: x_j -> y_k = x_0 + 2 sum_{j=1}^{M-1} x_j cos(j theta_k)
// (DCT-III), y_k -> x_j = (1/M) sum_k y_k cos(j theta_k) (DCT-II).  Two real
// columns make one complex column z, and with w_j = e^{i pi j / 2M}
//
//   V_j = w_j (z_j - i z_{M-j}),  v_n = sum_j V_j e^{2 pi i j n / M}
//
// gives y_{2n} = v_n, y_{2n+1} = v_{M-1-n} (Makhoul 1980's reordering): one
// complex FFT of M points for two real columns of 2M.  The order v_n is kept
// (any order of the frequencies serves as long as every pass uses the same),
// and the inverse is V = FFT(v), z_j = (conj(w_j) V_j + w_j V_{M-j}) / 2.
//
// The edge.  The grid p_i = (i - N/2) dp holds p = -N/2 dp without its mirror.
// This form leaves that row and column of A out where their part of Im chi is
// below the rounding of its FP32 sums (ev_band_applies).  Otherwise
// k_even_edge.cu carries them.
#pragma once

#include "kernels.cuh"

namespace lh {

// Lengths M of the cosine transforms: 16, 32, ..., 2048; 24, 48, ..., 1536; and
// 72, 144, ..., 1152, 432 and 864, so that no axis is padded by more than a third.
__host__ __device__ constexpr int ev_len(int i)
{
    return i < 8 ? 16 << i : i < 15 ? 24 << (i - 8) : i < 20 ? 72 << (i - 15) : i == 20 ? 432 : i == 21 ? 864 : 0;
}
// Smallest length >= x, 0 past the last.
inline int ev_len_for(long long x)
{
    int best = 0;
    for (int i = 0; ev_len(i); ++i)
        if (ev_len(i) >= x && (best == 0 || ev_len(i) < best)) best = ev_len(i);
    return best;
}
// Energy transform lengths of the correlation (the warp-per-line schedules).
inline int ev_energy_len(int n)
{
    return n <= 128 ? 128 : n <= 256 ? 256 : n <= 384 ? 384 : n <= 512 ? 512 : n <= 768 ? 768 : 0;
}

struct EvGeom {
    int M;            // frequencies per momentum axis
    int Nh;           // momentum rows p >= 0 kept (N / 2)
    int nl;           // lag rows s >= 0 (Q / 2 + 1)
    int e0, ne, J0;   // energy window [e0, e0 + ne) that reaches the kept transfers; occupied: j < J0
    int PE;           // energy FFT length
    int ES, WS;       // row strides (floats) of energies and transfers
    long long s1;     // plane strides (floats) of B1 [Nh][M][ES],
    long long s2;     //   B2 [M][M][ES] (k_x <= k_y),
    long long s3;     //   B3 [M][M][WS] (k_x <= k_y),
    long long s4;     //   B4 [nl][M][WS]
    float scale;      // Eq. 9 prefactor and transform norms
};

// Geometry of the even form, false where it does not apply (the grid's part of
// the rule; the band's is ev_band_applies).
inline bool ev_geom(const Geom &g, EvGeom &v)
{
    if (g.periodic) return false;
    v.M = ev_len_for((g.N + g.Q / 2 + 1) / 2);
    v.Nh = g.N / 2;
    v.nl = g.Q / 2 + 1;
    v.e0 = 0;
    v.ne = g.n_eps;
    if (g.quantity == LINDHARD_IMCHI) {
        // e_j < 0 <= e_{j+m}, m < n_omega: J0 - n_omega < j, j + m < J0 + n_omega
        const int lo = g.J0 - g.n_omega > 0 ? g.J0 - g.n_omega : 0;
        const int hi = g.J0 + g.n_omega < g.n_eps ? g.J0 + g.n_omega : g.n_eps;
        v.e0 = lo;
        v.ne = hi - lo;
    }
    v.J0 = g.J0 - v.e0;
    v.PE = ev_energy_len(g.quantity == LINDHARD_IMCHI ? v.ne : g.n_eps + g.n_omega - 1);
    if (v.M == 0 || v.PE == 0 || v.Nh < 2) return false;
    v.ES = (v.ne + 7) / 8 * 8;
    v.WS = (g.n_omega + 7) / 8 * 8;
    // 256 bytes of padding per plane: rows one plane apart then fall on
    // different memory channels
    v.s1 = (long long)v.M * v.ES + 64;
    v.s2 = v.s1;
    v.s3 = (long long)v.M * v.WS + 64;
    v.s4 = v.s3;
    // g.scale holds 1 / (P^2 PE); here 1 / M per axis, the 1/2 of each
    // inverse's last step and 1 / PE
    v.scale = (float)(g.scale * ((double)g.P * g.P * g.PE) / (4.0 * (double)v.M * v.M * v.PE));
    return true;
}
// Floats of the two work buffers: X holds B1, then B3; Y holds B2, then B4.
inline long long ev_x_floats(const EvGeom &v)
{
    const long long a = v.Nh * v.s1, b = v.M * v.s3;
    return a > b ? a : b;
}
inline long long ev_y_floats(const EvGeom &v)
{
    const long long a = v.M * v.s2, b = v.nl * v.s4;
    return a > b ? a : b;
}
// The same with the edge row and column (k_even_edge.cu): one row more, four
// volumes B3 (of k_x <= k_y) and two B4 of every lag s_x, and after B2 the edge
// lines' energy spectra and the M values sin(N theta_k / 2).
inline bool ev_edge_geom(const Geom &g, EvGeom &v)
{
    if (!ev_geom(g, v) || v.PE > 512) return false;
    v.Nh = g.N / 2 + 1;
    v.s3 = 4LL * v.M * v.WS + 64;
    v.s4 = 2LL * v.M * v.WS + 64;
    v.scale *= 0.5f;
    return true;
}
__host__ __device__ inline long long ev_edge_lines(const EvGeom &v) { return 4LL * (v.M + 1) * (v.PE / 2 + 16); }
inline long long ev_edge_x_floats(const EvGeom &v)
{
    const long long a = v.Nh * v.s1, b = v.M * v.s3;
    return a > b ? a : b;
}
inline long long ev_edge_y_floats(const Geom &g, const EvGeom &v)
{
    const long long a = v.M * v.s2 + ev_edge_lines(v) + v.M, b = g.Q * v.s4;
    return a > b ? a : b;
}
// Whether the edge row may be left out: its weight exp(-p^2 ff_a^2 / 8) must lie
// below 2^-24, half a unit in the last place of an FP32 sum, of the weight of the
// row with the same band energies that is nearest to the centre.  A tight-binding
// band of Z zones has that row at p_x = 0 (Z even) or pi (Z odd).  Free electrons
// have none: with mu at the edge's energy (Z pi)^2 / 2 the edge is what carries
// the spectral weight (4 zones of 12 points, ff_a 0.92, gamma 0.05: without it Im
// chi is off by 1.4e-3 of its maximum at mu = 79), so theirs is always carried.
inline bool ev_band_applies(const Geom &g, const Band &b)
{
    const double Z = g.N / g.npz, near = g.N / g.npz % 2, pa = 3.14159265358979323846 * b.ff_a;
    return b.band_kind != 1 && (Z * Z - near) * (pa * pa) >= 8.0 * 24.0 * 0.69314718055994530942;
}

// ---------------------------------------------------------------------------
// Packed arithmetic.  A thread carries two complex columns at once, one in each
// half of every register pair: four neighbouring floats x0..x3 of a row are the
// columns x0 + i x2 and x1 + i x3, so a row's 16 bytes are (re, im) as they
// lie, every complex operation is the same FP32x2 instruction for both columns
// with no swap of register halves, and every twiddle, address and predicate
// serves both.  Against one complex column a thread (75 instructions a point,
// issue slots 70% busy) this issues half the instructions; what bounds the
// passes now is the L1 data pipe (60-65%, the two exchanges) and the wait for
// loads.  1024^2 x 512, us, one column -> two: generation 338 -> 289, p_x 440
// -> 396, inverse k_x 250 -> 244, inverse k_y 280 -> 267 (5.5 TB/s).
struct Cx2 { float2 re, im; };

__device__ __forceinline__ float2 dup2(float c) { return make_float2(c, c); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return psub<true>(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ Cx2 add(Cx2 a, Cx2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ Cx2 sub(Cx2 a, Cx2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
// a + i b and a - i b
__device__ __forceinline__ Cx2 add_i(Cx2 a, Cx2 b) { return {sub2(a.re, b.im), add2(a.im, b.re)}; }
__device__ __forceinline__ Cx2 sub_i(Cx2 a, Cx2 b) { return {add2(a.re, b.im), sub2(a.im, b.re)}; }
// a times w or conj(w)
template <bool CONJ>
__device__ __forceinline__ Cx2 mul_w(Cx2 a, float2 w)
{
    const float2 wr = dup2(w.x), wi = dup2(w.y);
    if constexpr (CONJ) return {fma2(a.re, wr, mul2(a.im, wi)), fma2(a.im, wr, neg2(mul2(a.re, wi)))};
    else return {fma2(a.re, wr, neg2(mul2(a.im, wi))), fma2(a.im, wr, mul2(a.re, wi))};
}

// Small DFTs, positive exponent with INV.  The multiplications by sqrt(1/2)
// and sqrt(3/4) ride on the sums that follow as fused multiply-adds; 12 = 3 x 4
// by the prime-factor map (Good 1958), which needs no twiddles.
template <bool INV>
__device__ __forceinline__ void dft3(Cx2 &a, Cx2 &b, Cx2 &c)
{
    const float2 h = dup2(-0.5f), s = dup2(INV ? -0.86602540378443864676f : 0.86602540378443864676f), n = neg2(s);
    const Cx2 t = add(b, c), d = sub(b, c), m = {fma2(t.re, h, a.re), fma2(t.im, h, a.im)};
    a = add(a, t);
    b = {fma2(d.im, s, m.re), fma2(d.re, n, m.im)};   // m - i s d
    c = {fma2(d.im, n, m.re), fma2(d.re, s, m.im)};   // m + i s d
}
template <bool INV>
__device__ __forceinline__ void dft4(Cx2 &a, Cx2 &b, Cx2 &c, Cx2 &d)
{
    const Cx2 p = add(a, c), m = sub(a, c), q = add(b, d), r = sub(b, d);
    a = add(p, q);
    c = sub(p, q);
    b = INV ? add_i(m, r) : sub_i(m, r);
    d = INV ? sub_i(m, r) : add_i(m, r);
}
// (e + w o, e - w o) for w = e^{-+ i pi/4} (K = 1) or e^{-+ 3 i pi/4} (K = 3)
template <bool INV, int K>
__device__ __forceinline__ void combine45x(Cx2 e, Cx2 o, Cx2 &lo, Cx2 &hi)
{
    const float2 c = dup2(0.70710678118654752440f), n = dup2(-0.70710678118654752440f);
    const float2 s = add2(o.re, o.im), d = sub2(o.im, o.re);
    // forward: w1 o = c (s + i d), w3 o = c (d - i s); inverse: w1 o = c (-d + i s), w3 o = c (-s - i d)
    if constexpr (K == 1 && !INV) {
        lo = {fma2(s, c, e.re), fma2(d, c, e.im)};
        hi = {fma2(s, n, e.re), fma2(d, n, e.im)};
    } else if constexpr (K == 3 && !INV) {
        lo = {fma2(d, c, e.re), fma2(s, n, e.im)};
        hi = {fma2(d, n, e.re), fma2(s, c, e.im)};
    } else if constexpr (K == 1) {
        lo = {fma2(d, n, e.re), fma2(s, c, e.im)};
        hi = {fma2(d, c, e.re), fma2(s, n, e.im)};
    } else {
        lo = {fma2(s, n, e.re), fma2(d, n, e.im)};
        hi = {fma2(s, c, e.re), fma2(d, c, e.im)};
    }
}
template <bool INV>
__device__ __forceinline__ void dft8(Cx2 *v)
{
    Cx2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<INV>(e0, e1, e2, e3);
    dft4<INV>(o0, o1, o2, o3);
    v[0] = add(e0, o0);
    v[4] = sub(e0, o0);
    v[2] = INV ? add_i(e2, o2) : sub_i(e2, o2);
    v[6] = INV ? sub_i(e2, o2) : add_i(e2, o2);
    combine45x<INV, 1>(e1, o1, v[1], v[5]);
    combine45x<INV, 3>(e3, o3, v[3], v[7]);
}
template <int R, bool INV>
__device__ __forceinline__ void dft(Cx2 *v)
{
    if constexpr (R == 2) {
        const Cx2 a = v[0], b = v[1];
        v[0] = add(a, b);
        v[1] = sub(a, b);
    } else if constexpr (R == 3) {
        dft3<INV>(v[0], v[1], v[2]);
    } else if constexpr (R == 4) {
        dft4<INV>(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 6) {
        // inputs n = 3 i + 2 j, outputs k = 3 k2 + 4 k3 (mod 6)
        Cx2 a[3] = {add(v[0], v[3]), add(v[2], v[5]), add(v[4], v[1])};
        Cx2 b[3] = {sub(v[0], v[3]), sub(v[2], v[5]), sub(v[4], v[1])};
        dft3<INV>(a[0], a[1], a[2]);
        dft3<INV>(b[0], b[1], b[2]);
        v[0] = a[0]; v[4] = a[1]; v[2] = a[2];
        v[3] = b[0]; v[1] = b[1]; v[5] = b[2];
    } else if constexpr (R == 8) {
        dft8<INV>(v);
    } else if constexpr (R == 12) {
        // inputs n = 3 i + 4 j, outputs k = 9 k4 + 4 k3 (mod 12)
        Cx2 t[3][4];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
#pragma unroll
            for (int i = 0; i < 4; ++i) t[j][i] = v[(3 * i + 4 * j) % 12];
            dft4<INV>(t[j][0], t[j][1], t[j][2], t[j][3]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            dft3<INV>(t[0][k], t[1][k], t[2][k]);
#pragma unroll
            for (int q = 0; q < 3; ++q) v[(9 * k + 4 * q) % 12] = t[q][k];
        }
    } else {
        static_assert(R == 16, "radices of the schedules");
        Cx2 e[8], o[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) { e[i] = v[2 * i]; o[i] = v[2 * i + 1]; }
        dft8<INV>(e);
        dft8<INV>(o);
        v[0] = add(e[0], o[0]);
        v[8] = sub(e[0], o[0]);
        v[4] = INV ? add_i(e[4], o[4]) : sub_i(e[4], o[4]);
        v[12] = INV ? sub_i(e[4], o[4]) : add_i(e[4], o[4]);
        combine45x<INV, 1>(e[2], o[2], v[2], v[10]);
        combine45x<INV, 3>(e[6], o[6], v[6], v[14]);
#pragma unroll
        for (int k = 1; k < 8; k += 2) {
            const float c = (float)cos48(3 * k), s = (float)sin48(3 * k);
            const Cx2 w = mul_w<!INV>(o[k], make_float2(c, s));
            v[k] = add(e[k], w);
            v[k + 8] = sub(e[k], w);
        }
    }
}

// ---------------------------------------------------------------------------
// Radix schedules of the cosine transform's FFT (DCT-III order; DCT-II runs
// them reversed).  The first radix R0 is half of the values per thread, so
// that a thread owns butterflies j and M/R0 - j and with them rows n and M - n.
__host__ __device__ constexpr int ev_vpt(int M) { return M % 3 == 0 ? 24 : 16; }
__host__ __device__ constexpr int ev_nstages(int M)
{
    return M <= 144 ? 2 : M == 1536 ? 4 : 3;
}
__host__ __device__ constexpr int ev_radix_f(int M, int s)
{
    return s == 0 ? ev_vpt(M) / 2
         : M == 16 || M == 24 ? 2
         : M == 32 || M == 48 ? 4
         : M == 64 || M == 96 ? 8
         : M == 72 ? 6
         : M == 128 ? 16
         : M == 144 ? 12
         : M == 288 ? (s == 1 ? 8 : 3)
         : M == 432 || M == 576 || M == 864 || M == 1152 ? (s == 1 ? 12 : M / 144)
         : M == 192 ? 4
         : M == 256 ? (s == 1 ? 8 : 4)
         : M == 384 ? (s == 1 ? 8 : 4)
         : M == 512 || M == 768 ? 8
         : M == 1024 ? (s == 1 ? 8 : 16)
         : M == 1536 ? (s == 1 ? 8 : 4)
         : 16;
}
__host__ __device__ constexpr int ev_radix(int M, int s, bool rev) { return ev_radix_f(M, rev ? ev_nstages(M) - 1 - s : s); }
__host__ __device__ constexpr int ev_ns(int M, int s, bool rev)
{
    return s == 0 ? 1 : ev_ns(M, s - 1, rev) * ev_radix(M, s - 1, rev);
}
// Tables (float2): per length M the values w_j = e^{i pi j / 2M}, j < M, then
// per direction and stage s >= 1 rows k < Ns of w, w^2 (and for radices above 4
// w^3, w^4), w = e^{-2 pi i k / (Ns Rs)}; the higher powers are products of
// these, one rounding deep up to w^8.  (All powers from a table, as register
// pairs ready for the packed products, loaded no slower per value but took a
// third of the L1 data pipe: a 16-byte load costs four wavefronts however many
// lanes share its address.)
__host__ __device__ constexpr int ev_row(int R) { return R > 4 ? 4 : 2; }
__host__ __device__ constexpr int ev_table_offset(int M, int s, bool rev)   // s = 0: the w_j
{
    int o = 0;
    for (int i = 0; ev_len(i) != 0; ++i) {
        const int L = ev_len(i);
        if (L == M && s == 0) return o;
        o += L;
        for (int d = 0; d < 2; ++d)
            for (int st = 1; st < ev_nstages(L); ++st) {
                if (L == M && s == st && rev == (d != 0)) return o;
                o += ev_ns(L, st, d != 0) * ev_row(ev_radix(L, st, d != 0));
            }
    }
    return o;
}
__host__ __device__ constexpr int ev_table_entries() { return ev_table_offset(0, 0, false); }
// w^1..w^(R-1) from a table row
template <int R>
__device__ __forceinline__ void ev_powers(float2 *w, const float2 *__restrict__ row)
{
    const float4 q = __ldg(reinterpret_cast<const float4 *>(row));
    w[1] = make_float2(q.x, q.y);
    if constexpr (R > 2) w[2] = make_float2(q.z, q.w);   // radices 2, 3 and 4: two powers a row
    if constexpr (R == 4) w[3] = cmul(w[1], w[2]);
    if constexpr (R > 4) {
        const float4 p = __ldg(reinterpret_cast<const float4 *>(row) + 1);
        w[3] = make_float2(p.x, p.y);
        w[4] = make_float2(p.z, p.w);
#pragma unroll
        for (int r = 5; r < R; ++r) w[r] = r <= 8 ? cmul(w[4], w[r - 4]) : cmul(w[8], w[r - 8]);
    }
}

// Tiles: C packs of two complex columns (4C floats, 64 to 512 bytes of a row).
// Per SM 512 threads at 16 values each and 384 at 24: a load in flight holds its
// place in L1, and a fourth tile of 53 KB per SM left so little of it that the
// passes that load slowed down (k_ev_x at 1024^2 x 512 0.40 -> 0.52 ms); the
// generating pass, which loads nothing, runs four (0.31 -> 0.29 ms).
template <int M> struct EvCfg {
    static constexpr int C = M <= 24 || M == 72 ? 32 : M <= 48 || M == 144 ? 16 : M <= 256 || M == 288 || M == 432 ? 8 : M <= 1536 ? 4 : 2;
    static constexpr int T = C * M / ev_vpt(M);
    static constexpr int MINB_GEN = 512 / T > 0 ? 512 / T : 1;
    static constexpr int MINB = ev_vpt(M) == 16 ? 512 / T : 384 / T > 0 ? 384 / T : 1;
};

// One tile of C packs, VPT values per thread.  REV = false: DCT-III (positive
// exponent), the first stage on the butterfly pairs; REV = true: DCT-II
// (negative exponent), the last stage on the pairs.  Thread: pack tid % C,
// unit u = tid / C.
template <int M, bool REV>
struct EvFft {
    static constexpr int C = EvCfg<M>::C, T = EvCfg<M>::T, VPT = ev_vpt(M), TPC = M / VPT, NS = ev_nstages(M);
    static constexpr int RF = ev_radix(M, 0, REV), RP = ev_vpt(M) / 2, NBP = M / RP;   // RP, NBP: the paired stage
    // rows of C packs (16 bytes each); rows narrower than 128 bytes get one
    // empty row after every RF rows, so that the first exchange's writes (rows
    // RF apart) fall into different banks
    static constexpr bool PAD = C < 8;
    static constexpr int SMEM_ELEMS = (PAD ? M + M / RF : M) * C;   // packs
    static_assert(NBP == 2 * TPC, "a thread owns one butterfly pair");

    __device__ __forceinline__ static int srow(int row) { return (PAD ? row + row / RF : row) * C; }
    // offset of `step` further rows (a multiple of RF, or inside a block of RF)
    __host__ __device__ static constexpr int soff(int step) { return (PAD ? step + step / RF : step) * C; }
    __device__ __forceinline__ static void st(float4 *p, Cx2 v) { *p = make_float4(v.re.x, v.re.y, v.im.x, v.im.y); }
    __device__ __forceinline__ static Cx2 ld(const float4 *p)
    {
        const float4 q = *p;
        return {make_float2(q.x, q.y), make_float2(q.z, q.w)};
    }
    template <int S>
    __device__ __forceinline__ static int butterfly(int b, int u)
    {
        constexpr bool paired = REV ? S == NS - 1 : S == 0;
        if constexpr (paired) return b == 0 ? u : (u == 0 ? TPC : NBP - u);
        else return u + b * TPC;
    }
    template <int S>
    __device__ __forceinline__ static void rest(Cx2 *v, float4 *sm, int u, const float2 *__restrict__ tab)
    {
        if constexpr (S < NS) {
            constexpr int Rp = ev_radix(M, S - 1, REV), Nsp = ev_ns(M, S - 1, REV);
            constexpr int Rs = ev_radix(M, S, REV), Ns = ev_ns(M, S, REV);
            static_assert(VPT % Rp == 0 && VPT % Rs == 0, "values per thread");
            static_assert(!PAD || ((M / Rs) % RF == 0 && (Nsp == 1 || Nsp % RF == 0)), "compile-time padded offsets");
            if (S > 1) __syncthreads();   // the previous exchange has been read
#pragma unroll
            for (int b = 0; b < VPT / Rp; ++b) {
                const int j = butterfly<S - 1>(b, u);
                float4 *p = sm + srow((j / Nsp) * (Nsp * Rp) + j % Nsp);
#pragma unroll
                for (int r = 0; r < Rp; ++r) st(p + soff(r * Nsp), v[b * Rp + r]);
            }
            __syncthreads();
#pragma unroll
            for (int b = 0; b < VPT / Rs; ++b) {
                const int j = butterfly<S>(b, u);
                const float4 *p = sm + srow(j);
                float2 w[Rs];
                ev_powers<Rs>(w, tab + ev_table_offset(M, S, REV) + j % Ns * ev_row(Rs));
                v[b * Rs] = ld(p);
#pragma unroll
                for (int r = 1; r < Rs; ++r) v[b * Rs + r] = mul_w<!REV>(ld(p + soff(r * (M / Rs))), w[r]);
                dft<Rs, !REV>(v + b * Rs);
            }
            rest<S + 1>(v, sm, u, tab);
        }
    }
    // sm: this thread's pack of the tile's exchange buffer (base + tid % C);
    // v: first-stage inputs on entry, last-stage outputs on exit
    __device__ __forceinline__ static void run(Cx2 *v, float4 *sm, int u, const float2 *__restrict__ tab)
    {
#pragma unroll
        for (int b = 0; b < VPT / RF; ++b) dft<RF, !REV>(v + b * RF);
        rest<1>(v, sm, u, tab);
    }
};

// A pack from global memory, read once: not kept in L1, whose few KB beside the
// exchange buffers hold the tables.  Volatile and not through the read-only
// path: the kernel before may have written it (after_previous).
__device__ __forceinline__ Cx2 ev_load(const float *p)
{
    float4 q;
    asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(q.x), "=f"(q.y), "=f"(q.z), "=f"(q.w) : "l"(p) : "memory");
    return {make_float2(q.x, q.y), make_float2(q.z, q.w)};
}

// The pairs (n, M - n) of a thread's two paired butterflies (rows j + r NBP in
// v[b RP + r]): f(row n, value at n, value at M - n) for every pair, with
// M - 0 taken as row 0 itself.
template <int RP, int NBP, int TPC, typename V, typename F>
__device__ __forceinline__ void ev_pairs(V *v, int u, F &&f)
{
    if (u != 0) {
#pragma unroll
        for (int r = 0; r < RP; ++r) f(u + r * NBP, v[r], v[RP + RP - 1 - r]);
    } else {
        f(0, v[0], v[0]);
#pragma unroll
        for (int r = 1; r < RP / 2; ++r) f(r * NBP, v[r], v[RP - r]);
        f(RP / 2 * NBP, v[RP / 2], v[RP / 2]);
#pragma unroll
        for (int r = 0; r < RP / 2; ++r) f(TPC + r * NBP, v[RP + r], v[RP + RP - 1 - r]);
    }
}

// z -> V of the DCT-III, in place: V_n = w (a - i b), V_{M-n} = conj(w) (a + i b)
// for a = z_n, b = z_{M-n} (row 0: V_0 = z_0).
template <int M>
__device__ __forceinline__ void ev_pre(Cx2 *v, int u, const float2 *__restrict__ tab)
{
    constexpr int RP = ev_vpt(M) / 2, NBP = M / RP, TPC = M / ev_vpt(M);
    const float2 *wt = tab + ev_table_offset(M, 0, false);
    ev_pairs<RP, NBP, TPC>(v, u, [&](int n, Cx2 &a, Cx2 &b) {
        if (&a == &b) {   // n = 0: unchanged; n = M/2: w (1 - i) a = sqrt(2) a
            const float2 c = dup2(1.41421356237309505f);
            if (n != 0) a = {mul2(a.re, c), mul2(a.im, c)};
            return;
        }
        const float2 w = __ldg(wt + n);
        const Cx2 s = sub_i(a, b), d = add_i(a, b);
        a = mul_w<false>(s, w);
        b = mul_w<true>(d, w);
    });
}

// V -> 2 z of the DCT-II, in place: 2 z_n = conj(w) V_n + w V_{M-n},
// 2 z_{M-n} = -i (w V_{M-n} - conj(w) V_n).
template <int M>
__device__ __forceinline__ void ev_post(Cx2 *v, int u, const float2 *__restrict__ tab)
{
    constexpr int RP = ev_vpt(M) / 2, NBP = M / RP, TPC = M / ev_vpt(M);
    const float2 *wt = tab + ev_table_offset(M, 0, false);
    ev_pairs<RP, NBP, TPC>(v, u, [&](int n, Cx2 &a, Cx2 &b) {
        if (&a == &b) {
            const float2 c = dup2(n == 0 ? 2.0f : 1.41421356237309505f);
            a = {mul2(a.re, c), mul2(a.im, c)};
            return;
        }
        const float2 w = __ldg(wt + n);
        const Cx2 s = mul_w<true>(a, w), t = mul_w<false>(b, w);
        a = add(s, t);
        b = {sub2(t.im, s.im), sub2(s.re, t.re)};
    });
}

}  // namespace lh

// Dispatch on the cosine-transform length.
#define LH_EV_SWITCH(M_, CALL)                                    \
    switch (M_) {                                                 \
    case 16: return CALL(16);                                     \
    case 24: return CALL(24);                                     \
    case 32: return CALL(32);                                     \
    case 48: return CALL(48);                                     \
    case 64: return CALL(64);                                     \
    case 96: return CALL(96);                                     \
    case 128: return CALL(128);                                   \
    case 192: return CALL(192);                                   \
    case 256: return CALL(256);                                   \
    case 384: return CALL(384);                                   \
    case 512: return CALL(512);                                   \
    case 768: return CALL(768);                                   \
    case 1024: return CALL(1024);                                 \
    case 1536: return CALL(1536);                                 \
    case 72: return CALL(72);                                     \
    case 144: return CALL(144);                                   \
    case 288: return CALL(288);                                   \
    case 432: return CALL(432);                                   \
    case 576: return CALL(576);                                   \
    case 864: return CALL(864);                                   \
    case 1152: return CALL(1152);                                 \
    case 2048: return CALL(2048);                                 \
    default: return cudaErrorInvalidValue;                        \
    }
