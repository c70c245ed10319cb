// Real part of the Lindhard susceptibility by the Kramers-Kronig relation and
// the RPA susceptibility (Sec. 4: "the real part of the Lindhard
// susceptibility ... by applying Kramers-Kronig relation";
// chi_RPA = chi_L / (1 - V_q chi_L) with V_q decaying as 1 / q^2).
//
// For every lag q the transfers w_m = m de, m < n_omega, carry Im chi; with
// Im chi odd in w (chi(-q) = chi(q) for the inversion-symmetric bands of this
// problem) and zero beyond the computed window, Maclaurin's rule for the
// principal value gives a dense linear map along w:
//
//   Re chi_m = sum_k W(m, k) Im chi_k,  W(m, k) = (4/pi) k / (k^2 - m^2)
//              for k >= 1 with k - m odd, 0 otherwise.
//
//   k_kk_fft  : the sum as a Hilbert transform by FFT (below), two lines per
//               8 or 16 lanes, then chi_RPA.  n_omega <= 256.
//   k_kk_simt : the whole sum in FP32 SIMT (every weight from an FP32 table),
//               then chi_RPA.  n_omega <= 1536.
//
// V_q = v0 / |q|^2 at q = ((l_x - Q/2) dp, (l_y - Q/2) dp); at q = 0 chi_RPA
// takes its limit 0 (v0 = 0: chi_RPA = chi everywhere).  The weight tables
// are built once per plan in FP64 (k_kk_tables).
#include <algorithm>

#include "even_line.cuh"
#include "kernels.cuh"

namespace lh {

constexpr int KK_MAX_FFT = 256;   // longest n_omega of the FFT form
constexpr int KK_MAX_SIMT = 1536;

// Transform length of the FFT form: a multiple of 128 with n_omega <= M / 2
// (the lengths of even_line.cuh).
__host__ __device__ constexpr int kk_len(int nw) { return nw <= 64 ? 128 : nw <= 128 ? 256 : nw <= 192 ? 384 : 512; }
// Weight table of one n_omega: [FFT, n_omega <= 256 only: M FP32, then M / 2
// complex FP32, both in the order in which a lane of the transforms takes
// them], [SIMT: ceil(n_omega / 2) x n_omega FP32].  Byte offsets:
__host__ __device__ constexpr size_t kk_simt_off(int nw) { return nw <= KK_MAX_FFT ? 8ull * kk_len(nw) : 0; }
size_t kk_table_bytes(int nw) { return kk_simt_off(nw) + 4ull * ((nw + 1) / 2) * nw; }

__host__ __device__ inline double kk_weight(int m, int k, int nw)
{
    if (k < 1 || k >= nw || m >= nw || ((k - m) & 1) == 0) return 0.0;
    return 4.0 / 3.14159265358979323846 * (double)k / ((double)k * k - (double)m * m);
}

// Places in the table: H of frequency n = u + last(i) at [i / 4][u][i % 4], and
// w_n = e^{i pi n / 2M} of transfer n = ra + r R0 (or rb + r R0), ra = u, at
// [j / 2][u][j % 2], j = r (or R1 / 2 + r): lanes take 16 bytes side by side.
__device__ inline int kk_slot(int M, int n)
{
    const int R0 = M == 512 ? 32 : 16, R1 = M / R0, TPL = R0 / 2;
    const int r = n / R1, j = n % R1, u = j % TPL, i = j / TPL * R0 + r;
    return (i / 4 * TPL + u) * 4 + i % 4;
}
__device__ inline int kk_wslot(int M, int n)
{
    const int R0 = M == 512 ? 32 : 16, R1 = M / R0, TPL = R0 / 2;
    const int r = n / R0, c = n % R0, h = c >= TPL, u = h ? (c == TPL ? 0 : R0 - c) : c, j = h * (R1 / 2) + r;
    return (j / 2 * TPL + u) * 2 + j % 2;
}

// Transform of the kernel of the FFT form at the n-th frequency as the
// transforms list them (even.cuh: theta_k, k = 2n, then k = 2 (M - 1 - n) + 1),
// one warp per frequency: H(theta) = (4/pi) sum_{j odd < 2 n_omega - 1}
// sin(j theta) / j, with the sign (-1)^k and the 1 / 2M of the transforms.
__global__ void k_kk_tables(int nw, unsigned char *tab)
{
    const int H = (nw + 1) / 2, M = nw <= KK_MAX_FFT ? kk_len(nw) : 0;
    const long long n_simt = (long long)H * nw;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n_simt; i += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(i / nw), m = (int)(i % nw);
        reinterpret_cast<float *>(tab + kk_simt_off(nw))[i] = (float)kk_weight(m, 2 * j + 1 - (m & 1), nw);
    }
    const int lane = threadIdx.x % 32;
    for (int n = (int)((blockIdx.x * blockDim.x + threadIdx.x) / 32); n < M; n += (int)(gridDim.x * blockDim.x / 32)) {
        const int k = n < M / 2 ? 2 * n : 2 * (M - 1 - n) + 1;
        double h = 0.0;
        for (int j = 1 + 2 * lane; j < 2 * nw - 1; j += 64)
            h += sinpi((double)((j * (2 * k + 1)) % (4 * M)) / (double)(2 * M)) / (double)j;
        for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
        h *= 4.0 / 3.14159265358979323846 / (2.0 * M);
        if (lane == 0) reinterpret_cast<float *>(tab)[kk_slot(M, n)] = (float)(n < M / 2 ? h : -h);
    }
    for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < M / 2; n += gridDim.x * blockDim.x) {
        double sn, cs;
        sincospi(0.5 * (double)n / (double)M, &sn, &cs);
        reinterpret_cast<float2 *>(tab + 4 * M)[kk_wslot(M, n)] = make_float2((float)cs, (float)sn);
    }
}

cudaError_t launch_kk_tables(int nw, void *tab, cudaStream_t s)
{
    k_kk_tables<<<64, 256, 0, s>>>(nw, static_cast<unsigned char *>(tab));
    return cudaGetLastError();
}

// chi_RPA from chi = (r, x) at one transfer; V = 0 returns chi unchanged.
// The reciprocal of |1 - V chi|^2 is the hardware approximation (2 ulp),
// far inside the FP32 bar of chi_RPA.
__device__ __forceinline__ float2 kk_rpa(float r, float x, float V, bool zero)
{
    if (zero) return make_float2(0.f, 0.f);
    const float dr = 1.f - V * r, di = -V * x;
    const float inv = __fdividef(1.f, dr * dr + di * di);
    return make_float2((r * dr + x * di) * inv, (x * dr - r * di) * inv);
}
// V_q of lag line l = l_x Q + l_y; *zero when q = 0 with an interaction
__device__ __forceinline__ float kk_vq(long long l, int Q, double dp, double v0, bool *zero)
{
    const double qx = (double)(l / Q - Q / 2) * dp, qy = (double)(l % Q - Q / 2) * dp, q2 = qx * qx + qy * qy;
    *zero = (q2 == 0.0 && v0 != 0.0);
    return (v0 == 0.0 || q2 == 0.0) ? 0.f : (float)(v0 / q2);
}

// ---------------------------------------------------------------------------
// FFT form.  With x odd (x_{-k} = -x_k, x_0 not read) the sum is a convolution,
// Re chi_m = sum_k x_k h(k - m), h(j) = 2 / (pi j) for odd j, else 0: x odd and
// h odd, so on the half-shifted frequencies theta_k = pi (2k + 1) / 2M of
// even.cuh (period 2M with a change of sign) it is
//
//   S(theta) = 2 sum_j x_j sin(j theta),  Re chi_m = (1/M) sum_k S H cos(m theta_k),
//
// H the transform of h, cut at the |j| <= 2 n_omega - 2 that the kept transfers
// reach (M >= 2 n_omega: nothing wraps onto them).  The sine transform is the
// cosine transform of the reversed sequence times (-1)^k (in H's table), so
// V_n = -i w_n x_n and V_{M-n} = i conj(w_n) x_n; both transforms and the
// product by H stay in registers but for one exchange each (EvLine), two lines
// a complex column.
//
// Bound by instruction issue (100 instructions an output, 54% of the slots) and
// the wait for loads; 16 bytes an output, 3.5 TB/s.  It replaces BF16 hi/lo
// products on the tensor cores with an FP32 near band, where the operand split,
// the near band and the transposes around the products took about 145
// instructions an output with one or two CTAs of 8 warps per SM.  1024^2 lags x
// 256 transfers: 2.70 -> 1.24 ms (1.22 without the lines' scales), error 1.2e-6 ->
// 1.5e-7 of the result's norm; 256^2 x 128: 0.069 -> 0.052 ms.  Four lines a group in packed arithmetic (77
// instructions an output, 226 registers, 8 warps per SM): 1.46 ms; this with
// 168 registers: 1.56 ms, with 96: 1.46 ms; transfers' tables in natural order
// (one value a load): 1.26 ms.
//
// Two lines share a transform, and its rounding is that of the larger one: each is
// scaled by a power of two to a maximum in [1, 2) first and back after (exact; a
// line 1e-4 of its neighbour was off by 1e-3 of itself, and one near FP32's largest
// overflowed into it).  An infinity or NaN would still spread over the other line,
// so a group that holds one is summed directly (kk_direct).
constexpr int KKF_WARPS = 4;

// v0 / dp^2 = (h + l) 2^e, |h + l| in [0.05, 4e5] for any v0 (dp is 2 pi / 4096 to
// pi), so that neither a very small nor a very large v0 leaves FP32 before |q|^2
// divides it.
struct KkV {
    float h, l;
    int e;
};

// One pair of lines by the sum itself, FP32.
__device__ __noinline__ void kk_direct(long long l0, long long nlines, int nw, int u, int tpl, int Q, KkV v,
                                       const float *__restrict__ im, float *__restrict__ re, float2 *__restrict__ rpa);

// max(m, |x|), NaN if either is
__device__ __forceinline__ float kk_max(float m, float x)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(m), "f"(fabsf(x)));
    return r;
}

// v0 / |q|^2 of lag line l; *zero when q = 0 with an interaction
__device__ __forceinline__ float kk_v(long long l, int Q, KkV v, bool *zero)
{
    const int x = (int)(l / Q) - Q / 2, y = (int)(l % Q) - Q / 2;
    const float k2 = (float)(x * x + y * y);   // exact: Q <= 4096
    *zero = k2 == 0.f && v.h != 0.f;
    if (k2 == 0.f || v.h == 0.f) return 0.f;
    const float q = v.h / k2;
    return ldexpf(q + (fmaf(-q, k2, v.h) + v.l) / k2, v.e);
}

template <int M>
__global__ void __launch_bounds__(32 * KKF_WARPS, M == 384 ? 2 : 4)
k_kk_fft(long long nlines, int nw, int Q, KkV v0, const float *__restrict__ im, float *__restrict__ re,
         float2 *__restrict__ rpa, const float4 *__restrict__ kt, const float2 *__restrict__ tab)
{
    using E = EvLine<M>;
    constexpr int VPT = E::VPT, TPL = E::TPL, R0 = E::R0, R1 = E::R1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(KKF_WARPS * E::WARP_ELEMS, float2)
    const int lane = (int)threadIdx.x % 32, warp = (int)threadIdx.x / 32;
    const int sl = lane / TPL, u = lane % TPL;
    float2 *sm = reinterpret_cast<float2 *>(smem_raw) + warp * E::WARP_ELEMS + sl * E::LP;
    // this group's two lines, one complex column (Q is even, so Q^2 is too)
    const long long l0 = 2 * (((long long)blockIdx.x * KKF_WARPS + warp) * E::LPI + sl);
    const bool live = l0 < nlines, u0 = u == 0;
    // transfers below M/2 of this lane: ra + r R0 and rb + r R0, r < R1 / 2;
    // their mirrors M - n lie in the other butterfly (u = 0: in the same one)
    const int ra = u, rb = E::pair(1, u);
    const float *row = im + (live ? l0 : 0) * nw;
    float2 raw[2][R1 / 2];
    float top[2] = {0.f, 0.f}, up[2], down[2];   // the lines' maxima, their scales and back
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float *p = row + (h ? rb : ra);
#pragma unroll
        for (int r = 0; r < R1 / 2; ++r) {
            const bool in = live && (h ? rb : ra) + r * R0 < nw && (h + r > 0 || !u0);   // x_0 does not enter
            raw[h][r] = make_float2(in ? __ldg(p + r * R0) : 0.f, in ? __ldg(p + nw + r * R0) : 0.f);
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int r = 0; r < R1 / 2; ++r) {
            top[0] = kk_max(top[0], raw[h][r].x);
            top[1] = kk_max(top[1], raw[h][r].y);
        }
    bool bad = false;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
        for (int o = TPL / 2; o > 0; o >>= 1) top[i] = kk_max(top[i], __shfl_xor_sync(0xffffffffu, top[i], o));
        const unsigned e = __float_as_uint(top[i]) >> 23;   // 255: an infinity or NaN
        bad |= e == 255u;
        const unsigned c = min(max(e, 1u), 253u);
        up[i] = __uint_as_float((254u - c) << 23);
        down[i] = __uint_as_float(c << 23);
    }

    const float4 *ht = kt + u, *wt = kt + M / 4 + u;   // the lane's columns of the tables
    auto w_of = [&](float4 q, int r) { return r % 2 ? make_float2(q.z, q.w) : make_float2(q.x, q.y); };
    // V_n = -i w x, V_{M-n} = i conj(w) x
    float2 x[VPT], prev = make_float2(0.f, 0.f);
    auto sel = [&](float2 a, float2 b) { return make_float2(u0 ? a.x : b.x, u0 ? a.y : b.y); };
#pragma unroll
    for (int r = 0; r < R1 / 2; ++r) {
        float2 hi[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 v = make_float2(raw[h][r].x * up[0], raw[h][r].y * up[1]);
            const float2 w = w_of(__ldg(wt + (h * (R1 / 2) + r) / 2 * TPL), r);
            const float2 a = cmul(v, w), b = cmulc(v, w);
            x[h * R1 + r] = mul_mi(a);
            hi[h] = mul_i(b);
        }
        x[R1 + R1 - 1 - r] = sel(hi[1], hi[0]);
        if (r > 0) x[R1 - r] = sel(hi[0], prev);
        prev = hi[1];
    }
    x[R1 / 2] = sel(make_float2(0.f, 0.f), prev);
    E::inverse(x, sm, u, tab);
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const float4 q = __ldg(ht + i / 4 * TPL);
        const float h = i % 4 == 0 ? q.x : i % 4 == 1 ? q.y : i % 4 == 2 ? q.z : q.w;
        x[i] = make_float2(x[i].x * h, x[i].y * h);
    }
#pragma unroll
    for (int b = 0; b < VPT / R0; ++b) ev_dft<R0, false>(x + b * R0);
    E::forward_rest(x, sm, u, tab);
    if (!live) return;
    if (bad) {
        kk_direct(l0, nlines, nw, u, TPL, Q, v0, im, re, rpa);
        return;
    }
    float V[2];
    bool zero[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) V[i] = kk_v(l0 + i, Q, v0, &zero[i]);
    // Re chi of transfer m = conj(w) V_m + w V_{M-m} (the 1/2 in H)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int rh = h ? rb : ra;
        const float *xi = row + rh;
        float *ro = re + l0 * nw + rh;
        float2 *po = rpa + l0 * nw + rh;
#pragma unroll
        for (int r = 0; r < R1 / 2; ++r) {
            const float2 w = w_of(__ldg(wt + (h * (R1 / 2) + r) / 2 * TPL), r);
            const float2 a = x[h * R1 + r];
            const float2 b = h ? sel(x[R1 + R1 - 1 - r], x[R1 - 1 - r]) : sel(x[(R1 - r) % R1], x[R1 + R1 - 1 - r]);
            const float2 z = cadd(cmulc(a, w), cmul(b, w));
            const float y[2] = {z.x * down[0], z.y * down[1]};
            if (rh + r * R0 < nw) {
#pragma unroll
                for (int i = 0; i < 2; ++i) ro[i * nw + r * R0] = y[i];
                if (rpa) {
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        po[i * nw + r * R0] = kk_rpa(y[i], __ldg(xi + i * nw + r * R0), V[i], zero[i]);
                }
            }
        }
    }
}

__device__ __noinline__ void kk_direct(long long l0, long long nlines, int nw, int u, int tpl, int Q, KkV v,
                                       const float *__restrict__ im, float *__restrict__ re, float2 *__restrict__ rpa)
{
    for (int i = 0; i < 2 && l0 + i < nlines; ++i) {
        const float *row = im + (l0 + i) * nw;
        bool zero;
        const float V = kk_v(l0 + i, Q, v, &zero);
        for (int m = u; m < nw; m += tpl) {
            float s = 0.f;
            for (int k = 1 + (m & 1); k < nw; k += 2)
                s = fmaf(1.27323954473516268615f * (float)k / (float)(k * k - m * m), row[k], s);
            re[(l0 + i) * nw + m] = s;
            if (rpa) rpa[(l0 + i) * nw + m] = kk_rpa(s, row[m], V, zero);
        }
    }
}

// ---------------------------------------------------------------------------
// FP32 SIMT form: LB lines per CTA of 256 threads staged in shared memory
// (rows padded with one zero to nw + 1 floats), V_q per line beside them.
// Warp w takes lines w LPW .. w LPW + LPW - 1 and its lanes run along the
// transfers: each weight W(m, k) is read once per warp step (coalesced) and
// applied to the warp's LPW lines from registers; stores are coalesced.
constexpr int KK_SIMT_LPW = 8;
__host__ __device__ constexpr int kk_simt_lines(int nw)
{
    // 8 warps x up to 8 lines, at most ~96 KB of rows (two CTAs per SM)
    return (96 * 1024) / (4 * (nw + 1)) >= 64 ? 64 : ((96 * 1024) / (4 * (nw + 1))) / 8 * 8 < 8 ? 8
         : ((96 * 1024) / (4 * (nw + 1))) / 8 * 8;
}

__global__ void __launch_bounds__(256)
k_kk_simt(long long nlines, int nw, int Q, double dp, double v0, const float *__restrict__ im, float *__restrict__ re,
          float2 *__restrict__ rpa, const float *__restrict__ hs, int LB)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *rows = reinterpret_cast<float *>(smem_raw);          // [LB][nw + 1]
    float *vS = rows + LB * (nw + 1);                           // [LB] V_q (NaN: chi_RPA = 0)
    if (dyn_smem_bytes() < (unsigned)((LB * (nw + 1) + LB) * 4)) return;
    const long long l0 = (long long)blockIdx.x * LB;
#pragma unroll 8
    for (int i = threadIdx.x; i < LB * (nw + 1); i += blockDim.x) {
        const int l = i / (nw + 1), k = i % (nw + 1);
        rows[i] = (k < nw && l0 + l < nlines) ? im[(l0 + l) * nw + k] : 0.f;
    }
    if (threadIdx.x < LB) {
        bool zero;
        const float V = kk_vq(l0 + threadIdx.x, Q, dp, v0, &zero);
        vS[threadIdx.x] = zero ? __int_as_float(0x7fc00000) : V;
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, ln = threadIdx.x & 31, lpw = LB / 8;
    const int H = (nw + 1) / 2;
    for (int m0 = 0; m0 < nw; m0 += 32) {
        const int m = m0 + ln, k0 = 1 - (m & 1);
        float s[KK_SIMT_LPW];
#pragma unroll
        for (int i = 0; i < KK_SIMT_LPW; ++i) s[i] = 0.f;
#pragma unroll 4
        for (int j = 0; j < H; ++j) {
            const float h = (m < nw) ? __ldg(hs + (size_t)j * nw + m) : 0.f;
            const int k = 2 * j + k0;                           // <= nw: the padding zero
#pragma unroll
            for (int i = 0; i < KK_SIMT_LPW; ++i)
                if (i < lpw) s[i] = fmaf(h, rows[(warp * lpw + i) * (nw + 1) + k], s[i]);
        }
        if (m < nw) {
#pragma unroll
            for (int i = 0; i < KK_SIMT_LPW; ++i) {
                const int l = warp * lpw + i;
                if (i >= lpw || l0 + l >= nlines) continue;
                re[(l0 + l) * nw + m] = s[i];
                if (rpa) {
                    const float V = vS[l];
                    rpa[(l0 + l) * nw + m] = kk_rpa(s[i], rows[l * (nw + 1) + m], isnan(V) ? 0.f : V, isnan(V));
                }
            }
        }
    }
}

// variant 0: FFT (n_omega <= 256); 1: FP32 SIMT (n_omega <= 1536).  evt: the
// tables of even.cuh and even_line.cuh.
template <int M>
static cudaError_t launch_kk_fft_t(const Geom &g, const float *im, float *re, float2 *rpa, const void *tab, double v0,
                                   const float2 *evt, cudaStream_t s)
{
    using E = EvLine<M>;
    const size_t smem = sizeof(float2) * KKF_WARPS * E::WARP_ELEMS;
    static const cudaError_t e0 = smem_attrs(k_kk_fft<M>, smem);
    if (e0 != cudaSuccess) return e0;
    const long long nlines = (long long)g.Q * g.Q, per = 2LL * KKF_WARPS * E::LPI;
    KkV kv;
    const double v = frexp(v0, &kv.e) / (g.dp * g.dp);
    kv.h = (float)v;
    kv.l = (float)(v - (double)kv.h);
    k_kk_fft<M><<<(unsigned)((nlines + per - 1) / per), 32 * KKF_WARPS, smem, s>>>(
        nlines, g.n_omega, g.Q, kv, im, re, rpa, static_cast<const float4 *>(tab),
        evt + ev_line_table<M>());
    return cudaGetLastError();
}

cudaError_t launch_kk_rpa(const Geom &g, const float *im, float *re, float2 *rpa, const void *tab, double v0,
                          int variant, const void *evt, cudaStream_t s)
{
    const int nw = g.n_omega;
    if (variant == 0) {
        if (nw > KK_MAX_FFT) return cudaErrorNotSupported;
        switch (kk_len(nw)) {
        case 128: return launch_kk_fft_t<128>(g, im, re, rpa, tab, v0, (const float2 *)evt, s);
        case 256: return launch_kk_fft_t<256>(g, im, re, rpa, tab, v0, (const float2 *)evt, s);
        case 384: return launch_kk_fft_t<384>(g, im, re, rpa, tab, v0, (const float2 *)evt, s);
        default: return launch_kk_fft_t<512>(g, im, re, rpa, tab, v0, (const float2 *)evt, s);
        }
    }
    if (variant != 1 || nw > KK_MAX_SIMT) return cudaErrorNotSupported;
    const int LB = kk_simt_lines(nw);
    const size_t smem = (size_t)(LB * (nw + 1) + LB) * 4;
    static const cudaError_t e0 = smem_attrs(k_kk_simt, 100 * 1024);
    if (e0 != cudaSuccess) return e0;
    const long long nlines = (long long)g.Q * g.Q;
    const int grid = (int)((nlines + LB - 1) / LB);
    k_kk_simt<<<grid, 256, smem, s>>>(nlines, nw, g.Q, g.dp, v0, im, re, rpa,
                                     reinterpret_cast<const float *>(static_cast<const unsigned char *>(tab) +
                                                                     kk_simt_off(nw)),
                                     LB);
    return cudaGetLastError();
}

}  // namespace lh
