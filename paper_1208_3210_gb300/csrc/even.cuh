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
// 3.4 G: 8.19 -> 1.70 ms a call (256^3: 0.279 -> 0.087 ms; Im chi_T there
// 0.412 -> 0.106 ms).
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
// This form leaves that row and column of A out, so it is taken only when
// their weight |M|^2 is below 2^-24 of the centre's (ev_band_applies): their
// part of Im chi is then below the rounding of its FP32 sums.
#pragma once

#include "kernels.cuh"

namespace lh {

// Lengths M of the cosine transforms: 16, 32, ..., 2048 and 24, 48, ..., 1536.
__host__ __device__ constexpr int ev_len(int i)
{
    return i < 8 ? 16 << i : i < 15 ? 24 << (i - 8) : 0;
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
// The edge row's weight against the centre's, exp(-(N dp / 2)^2 ff_a^2 / 8),
// below 2^-24: half a unit in the last place of an FP32 sum of the centre's.
inline bool ev_band_applies(const Geom &g, const Band &b)
{
    const double p = 0.5 * g.N * g.dp * b.ff_a;
    return p * p >= 8.0 * 24.0 * 0.69314718055994530942;
}

// ---------------------------------------------------------------------------
// Radix schedules of the cosine transform's FFT (DCT-III order; DCT-II runs
// them reversed).  The first radix R0 is half of the values per thread, so
// that a thread owns butterflies j and M/R0 - j and with them rows n and M - n.
__host__ __device__ constexpr int ev_vpt(int M) { return M % 3 == 0 ? 24 : 16; }
__host__ __device__ constexpr int ev_nstages(int M)
{
    return M <= 128 ? 2 : M == 1536 ? 4 : 3;
}
__host__ __device__ constexpr int ev_radix_f(int M, int s)
{
    return s == 0 ? ev_vpt(M) / 2
         : M == 16 || M == 24 ? 2
         : M == 32 || M == 48 ? 4
         : M == 64 || M == 96 ? 8
         : M == 128 ? 16
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
// Tables (float2 units): per length M the M values w_j = e^{i pi j / 2M}, then
// per direction and stage s >= 1 rows k < Ns of (w, w^2), w = e^{-2 pi i k / (Ns Rs)}.
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
                o += 2 * ev_ns(L, st, d != 0);
            }
    }
    return o;
}
__host__ __device__ constexpr int ev_table_entries() { return ev_table_offset(0, 0, false); }

// Tiles: C complex columns (2C floats of a row), about 768 threads per SM (up
// to 85 registers each): the loads of one CTA's tile overlap the butterflies
// of another's.
template <int M> struct EvCfg {
    static constexpr int C = M <= 24 ? 64 : M <= 96 ? 32 : M <= 384 ? 16 : M <= 1536 ? 8 : 4;
    static constexpr int T = C * M / ev_vpt(M);
    static constexpr int MINB = M >= 1024 ? 1 : 768 / T;
};

// v[1..R) times the powers of (w, w^2) (conjugated with CONJ).
template <int R, bool CONJ>
__device__ __forceinline__ void ev_twiddle(float2 *v, const float4 *row)
{
    const float4 q = __ldg(row);
    float2 w[R];
    w[1] = make_float2(q.x, q.y);
    if constexpr (R > 2) w[2] = make_float2(q.z, q.w);
#pragma unroll
    for (int r = 3; r < R; ++r) w[r] = cmul(w[r / 2], w[r - r / 2]);
#pragma unroll
    for (int r = 1; r < R; ++r) v[r] = CONJ ? cmulc(v[r], w[r]) : cmul(v[r], w[r]);
}

// One tile of C complex columns, VPT values per thread.  REV = false: DCT-III
// (positive exponent), the first stage on the butterfly pairs; REV = true:
// DCT-II (negative exponent), the last stage on the pairs.  Thread: column
// tid % C, unit u = tid / C.
template <int M, bool REV>
struct EvFft {
    static constexpr int C = EvCfg<M>::C, T = EvCfg<M>::T, VPT = ev_vpt(M), TPC = M / VPT, NS = ev_nstages(M);
    static constexpr int RF = ev_radix(M, 0, REV), RP = ev_vpt(M) / 2, NBP = M / RP;   // RP, NBP: the paired stage
    // rows of C values; narrow rows get one empty row after every RF rows, so
    // that the first exchange's writes (rows RF apart) fall into different banks
    static constexpr bool PAD = C < 16;
    static constexpr int SMEM_ELEMS = (PAD ? M + M / RF : M) * C;
    static_assert(NBP == 2 * TPC, "a thread owns one butterfly pair");

    __device__ __forceinline__ static int srow(int row) { return (PAD ? row + row / RF : row) * C; }
    // offset of `step` further rows (a multiple of RF, or inside a block of RF)
    __host__ __device__ static constexpr int soff(int step) { return (PAD ? step + step / RF : step) * C; }
    template <int S>
    __device__ __forceinline__ static int butterfly(int b, int u)
    {
        constexpr bool paired = REV ? S == NS - 1 : S == 0;
        if constexpr (paired) return b == 0 ? u : (u == 0 ? TPC : NBP - u);
        else return u + b * TPC;
    }
    template <int S>
    __device__ __forceinline__ static void rest(float2 *v, float2 *sm, int u, const float2 *__restrict__ tab)
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
                float2 *p = sm + srow((j / Nsp) * (Nsp * Rp) + j % Nsp);
#pragma unroll
                for (int r = 0; r < Rp; ++r) p[soff(r * Nsp)] = v[b * Rp + r];
            }
            __syncthreads();
#pragma unroll
            for (int b = 0; b < VPT / Rs; ++b) {
                const int j = butterfly<S>(b, u);
                const float2 *p = sm + srow(j);
#pragma unroll
                for (int r = 0; r < Rs; ++r) v[b * Rs + r] = p[soff(r * (M / Rs))];
                ev_twiddle<Rs, !REV>(v + b * Rs, reinterpret_cast<const float4 *>(tab + ev_table_offset(M, S, REV)) + j % Ns);
                Dft<Rs, !REV, float2>::run(v + b * Rs);
            }
            rest<S + 1>(v, sm, u, tab);
        }
    }
    // sm: this thread's column of the tile's exchange buffer (base + tid % C);
    // v: first-stage inputs on entry, last-stage outputs on exit
    __device__ __forceinline__ static void run(float2 *v, float2 *sm, int u, const float2 *__restrict__ tab)
    {
#pragma unroll
        for (int b = 0; b < VPT / RF; ++b) Dft<RF, !REV, float2>::run(v + b * RF);
        rest<1>(v, sm, u, tab);
    }
};

// The pairs (n, M - n) of a thread's two paired butterflies (rows j + r NBP in
// v[b RP + r]): f(row n, value at n, value at M - n) for every pair, with
// M - 0 taken as row 0 itself.
template <int RP, int NBP, int TPC, typename F>
__device__ __forceinline__ void ev_pairs(float2 *v, int u, F &&f)
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
__device__ __forceinline__ void ev_pre(float2 *v, int u, const float2 *__restrict__ tab)
{
    constexpr int RP = ev_vpt(M) / 2, NBP = M / RP, TPC = M / ev_vpt(M);
    const float2 *wt = tab + ev_table_offset(M, 0, false);
    ev_pairs<RP, NBP, TPC>(v, u, [&](int n, float2 &a, float2 &b) {
        if (&a == &b) {
            // n = 0: unchanged; n = M/2: w (1 - i) a = sqrt(2) a
            if (n != 0) a = make_float2(1.41421356237309505f * a.x, 1.41421356237309505f * a.y);
            return;
        }
        const float2 w = __ldg(wt + n);
        const float2 s = make_float2(a.x + b.y, a.y - b.x), d = make_float2(a.x - b.y, a.y + b.x);
        a = cmul(s, w);
        b = cmulc(d, w);
    });
}

// V -> 2 z of the DCT-II, in place: 2 z_n = conj(w) V_n + w V_{M-n},
// 2 z_{M-n} = -i (w V_{M-n} - conj(w) V_n).
template <int M>
__device__ __forceinline__ void ev_post(float2 *v, int u, const float2 *__restrict__ tab)
{
    constexpr int RP = ev_vpt(M) / 2, NBP = M / RP, TPC = M / ev_vpt(M);
    const float2 *wt = tab + ev_table_offset(M, 0, false);
    ev_pairs<RP, NBP, TPC>(v, u, [&](int n, float2 &a, float2 &b) {
        if (&a == &b) {
            const float c = n == 0 ? 2.0f : 1.41421356237309505f;
            a = make_float2(c * a.x, c * a.y);
            return;
        }
        const float2 w = __ldg(wt + n);
        const float2 s = cmulc(a, w), t = cmul(b, w);
        a = cadd(s, t);
        b = make_float2(t.y - s.y, s.x - t.x);
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
    case 2048: return CALL(2048);                                 \
    default: return cudaErrorInvalidValue;                        \
    }
