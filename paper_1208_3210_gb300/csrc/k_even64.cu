// The even form with the edge row and column (even.cuh, k_even_edge.cu: the
// transforms, the edge's terms and the four parity parts) in double precision,
// for a generated A.
//
// FP64 arithmetic bounds it: two operations a clock and SM, a warp's
// instruction takes 16 cycles of one.  So what counts is the number of
// operations - one quadrant of A generated and transformed instead of the whole
// grid, half of the energy transforms - and the kernels are plain: transforms
// of radix 4, 3 and 2 in shared memory.  Columns of a pass go four to a CTA,
// energy lines one to a warp, so that small grids still fill the chip.
// Us a call, general form -> this: 32^2 x 40 109 -> 50, 64^2 x 128 382 -> 123,
// 128^2 x 200 2692 -> 650.
#include "even64.cuh"

namespace lh {

constexpr int E64_C = 4, E64_T = 64, E64_WARPS = 4;

__device__ __forceinline__ double2 add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 sub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 conj_mul(double2 a, double2 b)   // conj(a) b
{
    return make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
template <bool CONJ> __device__ __forceinline__ double2 mul(double2 a, double2 w)   // a w or a conj(w)
{
    return CONJ ? make_double2(a.x * w.x + a.y * w.y, a.y * w.x - a.x * w.y)
                : make_double2(a.x * w.x - a.y * w.y, a.y * w.x + a.x * w.y);
}
// a + i s b, s = +-1
template <bool POS> __device__ __forceinline__ double2 add_i(double2 a, double2 b)
{
    return POS ? make_double2(a.x - b.y, a.y + b.x) : make_double2(a.x + b.y, a.y - b.x);
}

// Transforms of N values (Stockham, natural order), `cols` columns ld apart, by
// nt threads (WARP: the lanes of a warp); a and b change places with every
// stage, the result's buffer is returned.  INV: positive exponent.  tab: e64_table.
template <int N, bool INV, bool WARP, int Ns = 1>
__device__ __forceinline__ double2 *fft64(double2 *a, double2 *b, int ld, int cols, int tid, int nt,
                                          const double2 *__restrict__ tab)
{
    if constexpr (Ns == N) {
        return a;
    } else {
        constexpr int L = N / Ns, R = L % 4 == 0 ? 4 : L % 3 == 0 ? 3 : 2, NB = N / R;
        for (int i = tid; i < cols * NB; i += nt) {
            const int c = i / NB, j = i % NB, k = j % Ns;
            const double2 *s = a + c * ld + j;
            double2 v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = s[r * NB];
            if constexpr (Ns > 1) {
#pragma unroll
                for (int r = 1; r < R; ++r) v[r] = mul<INV>(v[r], __ldg(tab + 4 * (k * r * (N / (Ns * R)))));
            }
            if constexpr (R == 4) {
                const double2 p = add(v[0], v[2]), m = sub(v[0], v[2]), q = add(v[1], v[3]), d = sub(v[1], v[3]);
                v[0] = add(p, q);
                v[2] = sub(p, q);
                v[1] = add_i<INV>(m, d);
                v[3] = add_i<!INV>(m, d);
            } else if constexpr (R == 3) {
                const double2 t = add(v[1], v[2]), d = sub(v[1], v[2]);
                const double2 m = make_double2(v[0].x - 0.5 * t.x, v[0].y - 0.5 * t.y);
                const double2 q = make_double2(0.86602540378443864676 * d.x, 0.86602540378443864676 * d.y);
                v[0] = add(v[0], t);
                v[1] = add_i<INV>(m, q);
                v[2] = add_i<!INV>(m, q);
            } else {
                const double2 t = v[1];
                v[1] = sub(v[0], t);
                v[0] = add(v[0], t);
            }
            double2 *o = b + c * ld + (j / Ns) * (Ns * R) + k;
#pragma unroll
            for (int r = 0; r < R; ++r) o[r * Ns] = v[r];
        }
        if constexpr (WARP) __syncwarp();
        else __syncthreads();
        return fft64<N, INV, WARP, Ns * R>(b, a, ld, cols, tid, nt, tab);
    }
}

__global__ void k_e64_tables(double2 *out)
{
    const int n = 4 * e64_len(blockIdx.x);
    int o = 0;
    for (int i = 0; i < (int)blockIdx.x; ++i) o += 4 * e64_len(i);
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        double s, c;
        sincospi(-2.0 * (double)k / (double)n, &s, &c);
        out[o + k] = make_double2(c, s);
    }
}

// xi_p = e0(p) - mu and |M(p)|^2 gamma / pi (Eqs. 4-5)
__device__ __forceinline__ double2 e64_point(const Band &band, const AxisTab &ax, const AxisTab &ay, const InstState *st)
{
    const double e0 = band.band_kind == 1 ? 0.5 * (ax.p2 + ay.p2)
                                          : -2.0 * band.t * (ax.c1 + ay.c1) - 4.0 * band.tp * ax.c1 * ay.c1
                                                - 2.0 * band.tpp * (ax.c2 + ay.c2);
    return make_double2(e0 - st->mu, ax.g * ay.g * band.gamma / 3.14159265358979323846);
}
// The columns' cosine transform (DCT-III order of even.cuh) of z in za; zb is
// the other buffer.  Returns the result's.
template <int M>
__device__ __forceinline__ double2 *e64_dct3(double2 *za, double2 *zb, const double2 *__restrict__ tab)
{
    constexpr int LD = M + 1;
    for (int i = threadIdx.x; i < E64_C * M; i += E64_T) {
        const int c = i / M, n = i % M;
        const double2 a = za[c * LD + n];
        // V_n = w_n (z_n - i z_{M-n}), w_n = e^{i pi n / 2M}
        zb[c * LD + n] = n == 0 ? a : mul<true>(add_i<false>(a, za[c * LD + M - n]), __ldg(tab + n));
    }
    __syncthreads();
    return fft64<M, true, false>(zb, za, LD, E64_C, threadIdx.x, E64_T, tab);
}
// 2 z_n of the DCT-II from the transform V (column of LD values): conj(w_n) V_n +
// w_n V_{M-n}; the even part reads its real half at n, the odd its imaginary at M - n.
template <int M>
__device__ __forceinline__ double2 e64_even_odd(const double2 *V, int n, const double2 *__restrict__ tab)
{
    if (n == 0) return make_double2(2.0 * V[0].x, 0.0);
    const double2 a = V[n], b = V[M - n], w = __ldg(tab + n), x = __ldg(tab + M - n);   // conj(w_n), conj(w_{M-n})
    return make_double2((a.x * w.x - a.y * w.y) + (b.x * w.x + b.y * w.y),
                        (b.x * x.y + b.y * x.x) + (a.y * x.x - a.x * x.y));
}

// B1 [Nh][M][ES]: A over p_y >= 0 for each p_x >= 0, transformed along p_y.
template <int M>
__global__ void __launch_bounds__(E64_T)
k_e64_gen_y(Geom g, E64Geom v, Band band, const AxisTab *axis, const double *eps,
            const InstState *st, double *__restrict__ B1, const double2 *__restrict__ tab, int ntile)
{
    constexpr int LD = M + 1;
    __shared__ double2 za[E64_C * LD], zb[E64_C * LD];
    after_previous();
    const int jx = blockIdx.x / ntile, e = 2 * E64_C * (blockIdx.x % ntile), half = g.N / 2;
    // the edge (index 0 of the axis): half its weight on either side
    for (int i = threadIdx.x; i < v.Nh; i += E64_T) {
        double2 q = e64_point(band, axis[jx == half ? 0 : half + jx], axis[i == half ? 0 : half + i], st);
        if (jx == half) q.y *= 0.5;
        if (i == half) q.y *= 0.5;
        zb[i] = q;
    }
    __syncthreads();
    const double g2 = band.gamma * band.gamma;
    for (int i = threadIdx.x; i < E64_C * M; i += E64_T) {
        const int c = i / M, n = i % M, k = e + 2 * c;
        double2 a = make_double2(0.0, 0.0);
        if (n < v.Nh) {
            const double2 q = zb[n];
            if (k < v.ne) { const double d = eps[v.e0 + k] - q.x; a.x = q.y / (d * d + g2); }
            if (k + 1 < v.ne) { const double d = eps[v.e0 + k + 1] - q.x; a.y = q.y / (d * d + g2); }
        }
        za[c * LD + n] = a;
    }
    __syncthreads();
    const double2 *y = e64_dct3<M>(za, zb, tab);
    for (int i = threadIdx.x; i < E64_C * M; i += E64_T) {
        const int c = i % E64_C, n = i / E64_C, k = e + 2 * c;
        if (k < v.ES) *reinterpret_cast<double2 *>(B1 + ((size_t)jx * M + n) * v.ES + k) = y[c * LD + n];
    }
}

// B2 [M][M][ES] (k_x <= k_y): B1 transformed along p_x for each k_y.
template <int M>
__global__ void __launch_bounds__(E64_T)
k_e64_x(E64Geom v, const double *B1, double *__restrict__ B2, const double2 *__restrict__ tab, int ntile)
{
    constexpr int LD = M + 1;
    __shared__ double2 za[E64_C * LD], zb[E64_C * LD];
    after_previous();
    const int ky = blockIdx.x / ntile, e = 2 * E64_C * (blockIdx.x % ntile);
    for (int i = threadIdx.x; i < E64_C * M; i += E64_T) {
        const int c = i % E64_C, n = i / E64_C, k = e + 2 * c;
        za[c * LD + n] = n < v.Nh && k < v.ES
                             ? *reinterpret_cast<const double2 *>(B1 + ((size_t)n * M + ky) * v.ES + k)
                             : make_double2(0.0, 0.0);
    }
    __syncthreads();
    const double2 *y = e64_dct3<M>(za, zb, tab);
    for (int i = threadIdx.x; i < E64_C * M; i += E64_T) {
        const int c = i % E64_C, n = i / E64_C, k = e + 2 * c;
        if (k < v.ES && n <= ky) *reinterpret_cast<double2 *>(B2 + ((size_t)n * M + ky) * v.ES + k) = y[c * LD + n];
    }
}

// Occupied (re) and empty (im) parts of A at energy n of the window, with the
// 1/2 of the separation: the split at e = 0, or the Fermi weights of Eq. A1.
__device__ __forceinline__ double2 e64_split(const Geom &g, const E64Geom &v, const Band &band, double A, int n)
{
    if (g.quantity == LINDHARD_IMCHI) return n < v.J0 ? make_double2(0.5 * A, 0.0) : make_double2(0.0, 0.5 * A);
    const double x = (double)(2 * n + 1 - g.n_eps) * band.x_step64;
    const double u = exp(-fabs(x)), big = 1.0 / (1.0 + u), small = u * big;
    return x < 0 ? make_double2(0.5 * A * big, 0.5 * A * small) : make_double2(0.5 * A * small, 0.5 * A * big);
}
struct E64Line { double2 occ, emp; };
__device__ __forceinline__ E64Line e64_separate(double2 k, double2 m)
{
    return {make_double2(k.x + m.x, k.y - m.y), make_double2(k.y + m.y, m.x - k.x)};
}

// Spectra of the edge lines a(k_t, e), t < M, and c(e), t = M (k_even_edge.cu):
// [line][PE/2 + 1][occupied, empty], then sin(N theta_k / 2) of every row.
template <int L>
__global__ void __launch_bounds__(32 * E64_WARPS)
k_e64_edge(Geom g, E64Geom v, Band band, const AxisTab *axis, const double *eps,
           const InstState *st, const double *B1, double2 *__restrict__ lines,
           const double2 *__restrict__ tab)
{
    __shared__ double2 buf[E64_WARPS][2][L];
    after_previous();
    double *sines = reinterpret_cast<double *>(lines) + e64_lines(v);
    for (int n = blockIdx.x * 32 * E64_WARPS + threadIdx.x; n < v.M; n += gridDim.x * 32 * E64_WARPS) {
        const int k = n < v.M / 2 ? 2 * n : 2 * (v.M - 1 - n) + 1;
        sines[n] = sinpi((double)((long long)g.N * (2 * k + 1) % (8LL * v.M)) / (4.0 * v.M));
    }
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, t = blockIdx.x * E64_WARPS + warp;
    if (t > v.M) return;
    double2 q = make_double2(0.0, 0.0);
    if (t == v.M) q = e64_point(band, axis[0], axis[0], st);
    for (int n = lane; n < L; n += 32) {
        double A = 0.0;
        if (n < v.ne) {
            if (t < v.M) {
                A = 2.0 * B1[((size_t)(v.Nh - 1) * v.M + t) * v.ES + n];
            } else {
                const double d = eps[v.e0 + n] - q.x;
                A = q.y / (d * d + band.gamma * band.gamma);
            }
        }
        buf[warp][0][n] = e64_split(g, v, band, A, n);
    }
    __syncwarp();
    const double2 *Z = fft64<L, false, true>(buf[warp][0], buf[warp][1], L, 1, lane, 32, tab);
    double2 *o = lines + (size_t)t * (L / 2 + 1) * 2;
    for (int k = lane; k <= L / 2; k += 32) {
        const E64Line s = e64_separate(Z[k], Z[(L - k) % L]);
        o[2 * k] = s.occ;
        o[2 * k + 1] = s.emp;
    }
}

// B3 [M][M][WS] of (EE, OY, OX, OO), k_x <= k_y: the energy correlation's parity
// parts, a line a warp.
template <int L>
__global__ void __launch_bounds__(32 * E64_WARPS)
k_e64_corr(Geom g, E64Geom v, Band band, const double *B2, const double2 *lines,
           double2 *__restrict__ B3, const double2 *__restrict__ tab)
{
    __shared__ double2 buf[E64_WARPS][3][L];
    after_previous();
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, t = blockIdx.x * E64_WARPS + warp;
    const int M = v.M;
    if (t >= M * (M + 1) / 2) return;
    // rows k_x and M - 1 - k_x folded to M + 1 lines
    const int f = t / (M + 1), c = t - f * (M + 1);
    const int kx = c < M - f ? f : M - 1 - f, ky = c < M - f ? f + c : c - 1;
    const bool odd = g.quantity == LINDHARD_IMCHI_T;
    const double *in = B2 + ((size_t)kx * M + ky) * v.ES;
    for (int n = lane; n < L; n += 32) buf[warp][0][n] = e64_split(g, v, band, n < v.ne ? in[n] : 0.0, n);
    __syncwarp();
    double2 *Z = fft64<L, false, true>(buf[warp][0], buf[warp][1], L, 1, lane, 32, tab);
    double2 *spare = Z == buf[warp][0] ? buf[warp][1] : buf[warp][0], *W = buf[warp][2];
    const double *sines = reinterpret_cast<const double *>(lines) + e64_lines(v);
    const double sx = sines[kx], sy = sines[ky], sxy = sx * sy;
    const double2 *ly = lines + (size_t)ky * (L / 2 + 1) * 2, *lx = lines + (size_t)kx * (L / 2 + 1) * 2,
                  *lc = lines + (size_t)M * (L / 2 + 1) * 2;
    auto scaled = [](double2 a, double s) { return make_double2(a.x * s, a.y * s); };
    for (int k = lane; k <= L / 2; k += 32) {
        const int km = (L - k) % L;
        const E64Line e = e64_separate(Z[k], Z[km]);
        const double2 co = scaled(lc[2 * k], sxy), cu = scaled(lc[2 * k + 1], sxy);
        const double2 xo = scaled(ly[2 * k], sx), xu = scaled(ly[2 * k + 1], sx);
        const double2 yo = scaled(lx[2 * k], sy), yu = scaled(lx[2 * k + 1], sy);
        const double2 r1o = sub(e.occ, co), r1u = sub(e.emp, cu), r2o = add(e.occ, co), r2u = add(e.emp, cu);
        const double2 i1o = add(yo, xo), i1u = add(yu, xu), i2o = sub(yo, xo), i2u = sub(yu, xu);
        const double2 re1 = add(conj_mul(r1o, r1u), conj_mul(i1o, i1u)), re2 = add(conj_mul(r2o, r2u), conj_mul(i2o, i2u));
        const double2 im1 = sub(conj_mul(i1o, r1u), conj_mul(r1o, i1u)), im2 = sub(conj_mul(i2o, r2u), conj_mul(r2o, i2u));
        double2 ee = add(re1, re2), oo = sub(re2, re1), ox = sub(im1, im2), oy = add(im1, im2);
        if (odd) {   // C(s, w) - C(-s, -w)
            ee = make_double2(0.0, 2.0 * ee.y);
            oo = make_double2(0.0, 2.0 * oo.y);
            ox = make_double2(2.0 * ox.x, 0.0);
            oy = make_double2(2.0 * oy.x, 0.0);
        }
        // EE + i OY and OX + i OO at k, the conjugates' at -k
        Z[km] = make_double2(ee.x + oy.y, oy.x - ee.y);
        W[km] = make_double2(ox.x + oo.y, oo.x - ox.y);
        Z[k] = make_double2(ee.x - oy.y, ee.y + oy.x);
        W[k] = make_double2(ox.x - oo.y, ox.y + oo.x);
    }
    __syncwarp();
    const double2 *p = fft64<L, true, true>(Z, spare, L, 1, lane, 32, tab);
    double2 *o = B3 + ((size_t)kx * M + ky) * v.WS * 2;
    for (int m = lane; m < v.WS; m += 32) o[2 * m] = p[m];
    __syncwarp();
    p = fft64<L, true, true>(W, spare, L, 1, lane, 32, tab);
    for (int m = lane; m < v.WS; m += 32) o[2 * m + 1] = p[m];
}

// B4 [Q][M][WS] of (even, odd in y): B3 back along k_x, to every lag s_x of the
// window.  Two columns a transfer: EE + i OX and OY + i OO.
template <int M>
__global__ void __launch_bounds__(E64_T)
k_e64_inv_x(E64Geom v, int Q, const double2 *B3, double2 *__restrict__ B4,
            const double2 *__restrict__ tab, int ntile)
{
    constexpr int LD = M + 1, MT = E64_C / 2;
    __shared__ double2 za[E64_C * LD], zb[E64_C * LD];
    after_previous();
    const int ky = blockIdx.x / ntile, m0 = MT * (blockIdx.x % ntile);
    for (int i = threadIdx.x; i < MT * M; i += E64_T) {
        const int c = i % MT, kx = i / MT, m = m0 + c;
        double2 p = make_double2(0.0, 0.0), q = p;
        if (m < v.WS) {
            const int lo = min(kx, ky), hi = max(kx, ky);
            const double2 *s = B3 + (((size_t)lo * M + hi) * v.WS + m) * 2;
            p = s[0];
            q = s[1];
        }
        const double oy = kx <= ky ? p.y : q.x, ox = kx <= ky ? q.x : p.y, sg = kx < M / 2 ? 1.0 : -1.0;
        za[2 * c * LD + kx] = make_double2(p.x, sg * ox);
        za[(2 * c + 1) * LD + kx] = make_double2(oy, sg * q.y);
    }
    __syncthreads();
    const double2 *V = fft64<M, false, false>(za, zb, LD, E64_C, threadIdx.x, E64_T, tab);
    for (int i = threadIdx.x; i < MT * M; i += E64_T) {
        const int c = i % MT, l = i / MT, m = m0 + c;
        if (m >= v.WS || l > Q / 2) continue;
        const double2 a = e64_even_odd<M>(V + 2 * c * LD, l, tab), b = e64_even_odd<M>(V + (2 * c + 1) * LD, l, tab);
        if (l < Q / 2) B4[((size_t)(Q / 2 + l) * M + ky) * v.WS + m] = make_double2(a.x + a.y, b.x + b.y);
        if (l > 0) B4[((size_t)(Q / 2 - l) * M + ky) * v.WS + m] = make_double2(a.x - a.y, b.x - b.y);
    }
    // lag -M of grids that keep it (Q = 2N = 2M): no pair of points is that far apart
    if (Q / 2 == M && threadIdx.x < MT && m0 + (int)threadIdx.x < v.WS)
        B4[(size_t)ky * v.WS + m0 + threadIdx.x] = make_double2(0.0, 0.0);
}

// B4 -> Im chi at (s_x, +-s_y), times the Eq. 9 prefactor.
template <int M>
__global__ void __launch_bounds__(E64_T)
k_e64_inv_y(E64Geom v, int Q, int n_omega, const double2 *B4, double *__restrict__ out,
            const double2 *__restrict__ tab, int ntile)
{
    constexpr int LD = M + 1;
    __shared__ double2 za[E64_C * LD], zb[E64_C * LD];
    after_previous();
    const int row = blockIdx.x / ntile, m0 = E64_C * (blockIdx.x % ntile);
    for (int i = threadIdx.x; i < E64_C * M; i += E64_T) {
        const int c = i % E64_C, ky = i / E64_C, m = m0 + c;
        const double2 p = m < v.WS ? B4[((size_t)row * M + ky) * v.WS + m] : make_double2(0.0, 0.0);
        za[c * LD + ky] = make_double2(p.x, ky < M / 2 ? p.y : -p.y);
    }
    __syncthreads();
    const double2 *V = fft64<M, false, false>(za, zb, LD, E64_C, threadIdx.x, E64_T, tab);
    double *o = out + ((size_t)row * Q + Q / 2) * n_omega;
    for (int i = threadIdx.x; i < E64_C * M; i += E64_T) {
        const int c = i % E64_C, l = i / E64_C, m = m0 + c;
        if (m >= n_omega || l > Q / 2) continue;
        const double2 a = e64_even_odd<M>(V + c * LD, l, tab);
        if (l < Q / 2) o[(long long)l * n_omega + m] = v.scale * (a.x + a.y);
        if (l > 0) o[-(long long)l * n_omega + m] = v.scale * (a.x - a.y);
    }
    if (Q / 2 == M && threadIdx.x < E64_C && m0 + (int)threadIdx.x < n_omega)
        o[-(long long)M * n_omega + m0 + threadIdx.x] = 0.0;
}

size_t e64_table_bytes() { return e64_table_entries() * sizeof(double2); }
cudaError_t launch_e64_tables(double2 *out, cudaStream_t s)
{
    int n = 0;
    while (e64_len(n) != 0) ++n;
    k_e64_tables<<<n, 256, 0, s>>>(out);
    return cudaGetLastError();
}
template <int M>
cudaError_t launch_e64_momentum(int pass, const Geom &g, const E64Geom &v, const Band &band, const Work<double> &w,
                                double *out, cudaStream_t s)
{
    const double2 *tab = (const double2 *)w.evt + e64_table(M);
    double *X = (double *)w.X, *Y = (double *)w.Y;
    const int te = (v.ES / 2 + E64_C - 1) / E64_C, tx = (v.WS + E64_C / 2 - 1) / (E64_C / 2), ty = (v.WS + E64_C - 1) / E64_C;
    switch (pass) {
    case 0: return launch_after(k_e64_gen_y<M>, v.Nh * te, E64_T, 0, s, g, v, band, w.axis, (const double *)w.eps, w.state,
                                X, tab, te);
    case 1: return launch_after(k_e64_x<M>, M * te, E64_T, 0, s, v, (const double *)X, Y, tab, te);
    case 2: return launch_after(k_e64_inv_x<M>, M * tx, E64_T, 0, s, v, g.Q, (const double2 *)X, (double2 *)Y, tab, tx);
    default: return launch_after(k_e64_inv_y<M>, g.Q * ty, E64_T, 0, s, v, g.Q, g.n_omega, (const double2 *)Y, out, tab, ty);
    }
}
template <int L>
cudaError_t launch_e64_energy(const Geom &g, const E64Geom &v, const Band &band, const Work<double> &w, cudaStream_t s)
{
    const double2 *tab = (const double2 *)w.evt + e64_table(L);
    double *X = (double *)w.X, *Y = (double *)w.Y;
    double2 *lines = (double2 *)(Y + (size_t)v.M * v.M * v.ES);
    const int n = v.M * (v.M + 1) / 2;
    const cudaError_t e = launch_after(k_e64_edge<L>, (v.M + E64_WARPS) / E64_WARPS, 32 * E64_WARPS, 0, s, g, v, band,
                                       w.axis, (const double *)w.eps, w.state, (const double *)X, lines, tab);
    if (e != cudaSuccess) return e;
    return launch_after(k_e64_corr<L>, (n + E64_WARPS - 1) / E64_WARPS, 32 * E64_WARPS, 0, s, g, v, band,
                        (const double *)Y, (const double2 *)lines, (double2 *)X, tab);
}
// Passes 0 p_y, 1 p_x, 2 inverse k_x, 3 inverse k_y.
cudaError_t launch_e64_pass(int pass, const Geom &g, const E64Geom &v, const Band &band, const Work<double> &w, double *out,
                            cudaStream_t s)
{
    switch (v.M) {
    case 16: return launch_e64_momentum<16>(pass, g, v, band, w, out, s);
    case 24: return launch_e64_momentum<24>(pass, g, v, band, w, out, s);
    case 32: return launch_e64_momentum<32>(pass, g, v, band, w, out, s);
    case 48: return launch_e64_momentum<48>(pass, g, v, band, w, out, s);
    case 64: return launch_e64_momentum<64>(pass, g, v, band, w, out, s);
    case 96: return launch_e64_momentum<96>(pass, g, v, band, w, out, s);
    case 128: return launch_e64_momentum<128>(pass, g, v, band, w, out, s);
    default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_e64_corr(const Geom &g, const E64Geom &v, const Band &band, const Work<double> &w, cudaStream_t s)
{
    switch (v.PE) {
    case 16: return launch_e64_energy<16>(g, v, band, w, s);
    case 24: return launch_e64_energy<24>(g, v, band, w, s);
    case 32: return launch_e64_energy<32>(g, v, band, w, s);
    case 48: return launch_e64_energy<48>(g, v, band, w, s);
    case 64: return launch_e64_energy<64>(g, v, band, w, s);
    case 96: return launch_e64_energy<96>(g, v, band, w, s);
    case 128: return launch_e64_energy<128>(g, v, band, w, s);
    case 192: return launch_e64_energy<192>(g, v, band, w, s);
    case 256: return launch_e64_energy<256>(g, v, band, w, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lh
