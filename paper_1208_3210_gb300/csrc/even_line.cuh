// Two-stage energy transforms of the even form (k_even_corr.cu, k_even_bw.cu) and
// of the Kramers-Kronig pass (k_kk.cu): lines of 128,
// 256, 384 or 512 energies, TPL = 8 or 16 lanes a line, VPT = 16, 32 or 48
// values a lane, one exchange through shared memory.  The three-stage schedules
// with 16 values a lane (et_tiles.cuh) were bound by the L1 data pipe here (71%
// at 512 energies, 88% at 128: two exchanges and the twiddle rows of two
// stages); these issue 34 instructions a point instead of 47 with that pipe at
// 37% and the FMA pipe at 45%.  The correlation at 1024^2 x 512: 366 -> 305 us
// (3.0 TB/s), Im chi_T at 256^3: 37 -> 27 us.
//
//   forward : L = R0 R1; stage 0 on butterflies u + b TPL (radix R0), stage 1 on
//             j and R0 - j (radix R1 = VPT / 2; u = 0: 0 and R0/2), so that Z(k)
//             and Z(L - k) end in the same lane
//   inverse : the mirror image, radix R1 on the same pairs first, then R0
#pragma once

#include "even.cuh"

namespace lh {

// cos(2 pi m / 32)
__host__ __device__ constexpr double cos32_q(int m)   // m in [0, 8]
{
    return m == 0 ? 1.0 : m == 1 ? 0.98078528040323044913 : m == 2 ? 0.92387953251128675613
         : m == 3 ? 0.83146961230254523708 : m == 4 ? 0.70710678118654752440 : m == 5 ? 0.55557023301960222474
         : m == 6 ? 0.38268343236508977173 : m == 7 ? 0.19509032201612826785 : 0.0;
}
__host__ __device__ constexpr double cos32(int m)
{
    return (m % 32) <= 8 ? cos32_q(m % 32) : (m % 32) <= 16 ? -cos32_q(16 - m % 32)
         : (m % 32) <= 24 ? -cos32_q(m % 32 - 16) : cos32_q(32 - m % 32);
}
// x exp(-+ 2 pi i K / R)
template <int R, int K, bool INV>
__device__ __forceinline__ float2 ev_twc(float2 x)
{
    if constexpr (R == 32 && K % 2 != 0) {
        constexpr float c = (float)cos32(K), s = (float)cos32(K + 24);   // cos, sin
        return INV ? make_float2(x.x * c - x.y * s, x.x * s + x.y * c) : make_float2(x.x * c + x.y * s, x.y * c - x.x * s);
    } else if constexpr (R == 32) return twc<16, K / 2, INV>(x);
    else return twc<R, K, INV>(x);
}

// Complex sums as packed FP32x2 instructions (padd): these kernels have
// registers to spare (scalar sums: 364 us instead of 319).
constexpr bool EV_PK = true;

// DFT of R values: radix 32 as two halves of 16.
template <int R, bool INV, int K = 0>
__device__ __forceinline__ void ev_dit(float2 *v, const float2 *e, const float2 *o)
{
    if constexpr (K < R / 2) {
        const float2 t = ev_twc<R, K, INV>(o[K]);
        v[K] = padd<EV_PK>(e[K], t);
        v[K + R / 2] = psub<EV_PK>(e[K], t);
        ev_dit<R, INV, K + 1>(v, e, o);
    }
}
template <int R, bool INV>
__device__ __forceinline__ void ev_dft(float2 *v)
{
    if constexpr (R == 32) {
        float2 e[16], o[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) { e[i] = v[2 * i]; o[i] = v[2 * i + 1]; }
        Dft<16, INV, float2, EV_PK>::run(e);
        Dft<16, INV, float2, EV_PK>::run(o);
        ev_dit<32, INV>(v, e, o);
    } else {
        Dft<R, INV, float2, EV_PK>::run(v);
    }
}
// Tables after the cosine transforms': per length, k < 32: (w, w^2), 32 entries
// later (w^3, w^4), 32 later (w^8, w^16), w = e^{-2 pi i k / L}: no power is more
// than two products from an entry.
constexpr int EV_LINE_TABLE = 192;
__host__ __device__ constexpr int ev_line_len(int i) { return i == 0 ? 128 : i == 1 ? 256 : i == 2 ? 384 : i == 3 ? 512 : 0; }
template <int L>
__host__ __device__ constexpr int ev_line_table()
{
    return (ev_table_entries() + 1) / 2 * 2 + (L == 128 ? 0 : L == 256 ? 1 : L == 384 ? 2 : 3) * EV_LINE_TABLE;
}
__host__ __device__ constexpr int ev_all_tables() { return (ev_table_entries() + 1) / 2 * 2 + 4 * EV_LINE_TABLE; }

constexpr int EVC_WARPS = 4;

// Line t of the triangle k_x <= k_y, rows k_x and M - 1 - k_x folded to M + 1
// entries: t = f (M + 1) + c.
__device__ __forceinline__ void ev_tri(int t, int M, int &kx, int &ky)
{
    const int f = t / (M + 1), c = t - f * (M + 1);
    if (c < M - f) {
        kx = f;
        ky = f + c;
    } else {
        kx = M - 1 - f;
        ky = c - 1;   // kx + (c - (M - f))
    }
}

// Rounds per warp: up to 8 while every SM still gets 48 warps' worth.
inline int ev_corr_iters(int npairs, int lpi, int sms)
{
    const int rounds = (npairs + lpi - 1) / lpi, it = rounds / (sms * 48);
    return it < 1 ? 1 : it > 8 ? 8 : it;
}

template <int L>
struct EvLine {
    static constexpr int R0 = L == 512 ? 32 : 16, R1 = L / R0, VPT = 2 * R1, TPL = L / VPT, LPI = 32 / TPL;
    // exchange rows of R0 (forward) or R1 (inverse) values and one empty; a
    // line's start is 8 values off a multiple of 16 from its neighbour's, so
    // that two 8-lane lines use different halves of the banks
    static constexpr int LP = L == 128 ? 152 : L == 256 ? 280 : L == 384 ? 408 : 544;
    static constexpr int WARP_ELEMS = LPI * LP;
    // 168 registers, 255 at 384 energies (48 values; at 168 it spills); two
    // CTAs of 255 registers at 512 energies: 364 us instead of 319
    static constexpr int MINB = L == 384 ? 2 : L == 128 ? 4 : 3;
    static_assert(R0 == 2 * TPL && VPT % R0 == 0, "schedule");
    static_assert(LP >= R1 * (R0 + 1) && LP >= R0 * (R1 + 1), "exchange");

    // energy of x[i] before the forward, transfer of x[i] after the inverse, less u
    __host__ __device__ static constexpr int first(int i) { return (i / R0) * TPL + (i % R0) * R1; }
    __host__ __device__ static constexpr int last(int i) { return first(i); }
    __device__ __forceinline__ static int pair(int b, int u) { return b == 0 ? u : (u == 0 ? TPL : R0 - u); }

    // w^r, 0 < r < R, of row k
    template <int R>
    __device__ __forceinline__ static void powers(float2 *w, const float2 *__restrict__ tab, int k)
    {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(tab) + k), b = __ldg(reinterpret_cast<const float4 *>(tab) + 32 + k);
        w[1] = make_float2(a.x, a.y);
        w[2] = make_float2(a.z, a.w);
        w[3] = make_float2(b.x, b.y);
        w[4] = make_float2(b.z, b.w);
        if constexpr (R > 8) {
            const float4 c = __ldg(reinterpret_cast<const float4 *>(tab) + 64 + k);
            w[8] = make_float2(c.x, c.y);
            if constexpr (R > 16) w[16] = make_float2(c.z, c.w);
        }
#pragma unroll
        for (int r = 5; r < R; ++r) {
            const int p = r < 8 ? 4 : r < 16 ? 8 : 16;
            if (r != p) w[r] = cmul(w[p], w[r - p]);
        }
    }

    // z = a + i b (with the 1/2 of the separation) and the first radix.  FULL:
    // occupied rows n < L/2 are real, the others imaginary, so the first
    // radix-2 level z_r +- z_{r + R0/2} is A_r + i B_r and its conjugate.
    template <bool FULL, bool THERMAL>
    __device__ __forceinline__ static void first_stage(float2 *x, const float *raw, int u, int J0, const float2 *wf)
    {
#pragma unroll
        for (int b = 0; b < VPT / R0; ++b) {
            if constexpr (FULL && !THERMAL) {
                float2 s[R0 / 2], d[R0 / 2];
#pragma unroll
                for (int r = 0; r < R0 / 2; ++r) {
                    s[r] = make_float2(0.5f * raw[b * R0 + r], 0.5f * raw[b * R0 + r + R0 / 2]);
                    d[r] = make_float2(s[r].x, -s[r].y);
                }
                dif<0>(d);
                ev_dft<R0 / 2, false>(s);
                ev_dft<R0 / 2, false>(d);
#pragma unroll
                for (int r = 0; r < R0 / 2; ++r) { x[b * R0 + 2 * r] = s[r]; x[b * R0 + 2 * r + 1] = d[r]; }
            } else {
#pragma unroll
                for (int r = 0; r < R0; ++r) {
                    const int n = u + first(b * R0 + r);
                    const float A = 0.5f * raw[b * R0 + r];
                    if constexpr (THERMAL) {
                        const float2 w = wf[n];
                        x[b * R0 + r] = make_float2(A * w.x, A * w.y);
                    } else {
                        x[b * R0 + r] = n < J0 ? make_float2(A, 0.f) : make_float2(0.f, A);
                    }
                }
                ev_dft<R0, false>(x + b * R0);
            }
        }
    }
    template <int K>
    __device__ __forceinline__ static void dif(float2 *d)
    {
        if constexpr (K < R0 / 2) {
            d[K] = ev_twc<R0, K, false>(d[K]);
            dif<K + 1>(d);
        }
    }
    __device__ __forceinline__ static void forward_rest(float2 *x, float2 *sm, int u, const float2 *__restrict__ tab)
    {
        __syncwarp();   // the previous exchange has been read
#pragma unroll
        for (int b = 0; b < VPT / R0; ++b)
#pragma unroll
            for (int r = 0; r < R0; ++r) sm[(u + b * TPL) * (R0 + 1) + r] = x[b * R0 + r];
        __syncwarp();
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int j = pair(b, u);
            float2 w[R1];
            powers<R1>(w, tab, j);
            x[b * R1] = sm[j];
#pragma unroll
            for (int r = 1; r < R1; ++r) x[b * R1 + r] = cmul(sm[j + r * (R0 + 1)], w[r]);
            ev_dft<R1, false>(x + b * R1);
        }
    }
    __device__ __forceinline__ static void inverse(float2 *x, float2 *sm, int u, const float2 *__restrict__ tab)
    {
        ev_dft<R1, true>(x);
        ev_dft<R1, true>(x + R1);
        __syncwarp();
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            float2 *p = sm + pair(b, u) * (R1 + 1);
#pragma unroll
            for (int r = 0; r < R1; ++r) p[r] = x[b * R1 + r];
        }
        __syncwarp();
#pragma unroll
        for (int b = 0; b < VPT / R0; ++b) {
            const int j = u + b * TPL;
            float2 w[R0];
            powers<R0>(w, tab, j);
            x[b * R0] = sm[j];
#pragma unroll
            for (int r = 1; r < R0; ++r) x[b * R0 + r] = cmulc(sm[j + r * (R1 + 1)], w[r]);
            ev_dft<R0, true>(x + b * R0);   // outputs that the caller drops are not formed
        }
    }
};

}  // namespace lh
