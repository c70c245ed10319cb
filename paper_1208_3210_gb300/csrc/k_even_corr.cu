// Energy correlation of the even form (even.cuh): for every momentum frequency
// pair k_x <= k_y, C(k, w_m) = sum_j a(k, e_j) b(k, e_{j+m}) of Eq. 9, where a
// and b are the occupied and empty parts of the real spectrum A(k, e) (Sec. 3 /
// Appendix A: the split at e = 0, or at temperature kT the Fermi weights of
// Eq. A1), by FFT along the energy axis.
//
// A pair of lines per TPL lanes: each line's z = a + i b is transformed, a^ and
// b^ are separated and conj(a^) b^ formed in registers, then the two lines'
// products share one inverse transform (W = P1 + i P2).  The forward's last
// stage and the inverse's first own the same frequencies in the same threads,
// so nothing between the transforms leaves the registers.  1.5 transforms a
// line, of two stages and one exchange each (even_line.cuh).
#include "even.cuh"
#include "even_line.cuh"
#include "et_tiles.cuh"

namespace lh {

// FULL: ne == L with the split at L/2.  THERMAL: Fermi weights (odd: the odd
// part, Im chi_T).  HALF: WS <= L/2, the upper half of the lags is not formed.
template <int L, bool FULL, bool THERMAL, bool HALF>
__global__ void __launch_bounds__(32 * EVC_WARPS, EvLine<L>::MINB)
k_ev_corr(Geom g, EvGeom v, Band band, const float *B2, float *__restrict__ B3,
          const float2 *__restrict__ tab, int iters, int odd)
{
    using E = EvLine<L>;
    constexpr int VPT = E::VPT, TPL = E::TPL, R0 = E::R0, R1 = E::R1;
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
    const int npairs = v.M / 2 * (v.M + 1) / 2;
    const bool u0 = u == 0;

    for (int it = 0; it < iters; ++it) {
        const int f = ((blockIdx.x * EVC_WARPS + warp) * iters + it) * E::LPI + sl;
        const bool live = f < npairs;
        float2 pa[2][R1 / 2], pb[2][R1 / 2], ph[2], x[VPT];
#pragma unroll
        for (int r = 0; r < R1 / 2; ++r) pa[1][r] = pb[1][r] = make_float2(0.f, 0.f);
        ph[1] = make_float2(0.f, 0.f);
        float raw[VPT];
        int kx, ky;
        ev_tri(live ? 2 * f : 0, v.M, kx, ky);
        auto load = [&] {
            const float *p = B2 + (kx * v.s2 + (long long)ky * v.ES + u);
#pragma unroll
            for (int i = 0; i < VPT; ++i)
                raw[i] = live && (FULL || u + E::first(i) < v.ne) ? __ldcs(p + E::first(i)) : 0.f;
        };
        load();
        // one copy of the forward code for both lines (the body unrolled twice
        // spent a tenth of its time waiting for instructions)
#pragma unroll 1
        for (int q = 0; q < 2; ++q) {
#pragma unroll
            for (int r = 0; r < R1 / 2; ++r) {
                pa[0][r] = pa[1][r];
                pb[0][r] = pb[1][r];
            }
            ph[0] = ph[1];
            E::template first_stage<FULL, THERMAL>(x, raw, u, v.J0, wf);
            if (q == 0) {   // the second line's values travel during the first one's transform
                ev_tri(live ? 2 * f + 1 : 0, v.M, kx, ky);
                load();
            }
            E::forward_rest(x, sm, u, tab);
            // conj(a^) b^ with a^ = Z(k) + conj Z(-k), b^ = (Z(k) - conj Z(-k)) / i
            // (halved in the input), k <= L/2
            auto prod = [&](float2 zk, float2 zm) {
                const float2 p = cmulc(make_float2(zk.y + zm.y, zm.x - zk.x), make_float2(zk.x + zm.x, zk.y - zm.y));
                return THERMAL ? odd_part(p, odd != 0) : p;
            };
#pragma unroll
            for (int r = 0; r < R1 / 2; ++r) {
                pa[1][r] = prod(x[r], u0 ? x[(R1 - r) % R1] : x[R1 + R1 - 1 - r]);
                pb[1][r] = prod(x[R1 + r], u0 ? x[R1 + R1 - 1 - r] : x[R1 - 1 - r]);
            }
            ph[1] = prod(x[R1 / 2], x[R1 / 2]);   // k = L/2, used where u = 0
        }
        // W(k) = P1 + i P2 and W(L - k) = conj P1 + i conj P2 in the inverse's
        // first-stage order (rows j2[b] + r R0)
        auto w_of = [](float2 x1, float2 x2) { return make_float2(x1.x - x2.y, x1.y + x2.x); };
        auto w_conj = [](float2 x1, float2 x2) { return make_float2(x1.x + x2.y, x2.x - x1.y); };
#pragma unroll
        for (int r = 0; r < R1 / 2; ++r) {
            x[r] = w_of(pa[0][r], pa[1][r]);
            x[R1 + r] = w_of(pb[0][r], pb[1][r]);
            x[R1 + R1 - 1 - r] = u0 ? w_conj(pb[0][r], pb[1][r]) : w_conj(pa[0][r], pa[1][r]);
        }
        // u > 0: row R1 - 1 - r mirrors pb[r]; u = 0: row R1 - r mirrors pa[r], row R1/2 is k = L/2
#pragma unroll
        for (int r = R1 / 2; r < R1; ++r) {
            const float2 hi = w_conj(pb[0][R1 - 1 - r], pb[1][R1 - 1 - r]);
            const float2 lo = r == R1 / 2 ? w_of(ph[0], ph[1]) : w_conj(pa[0][(R1 - r) % (R1 / 2)], pa[1][(R1 - r) % (R1 / 2)]);
            x[r] = u0 ? lo : hi;
        }
        E::inverse(x, sm, u, tab);
        if (live) {
            long long ob[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                ev_tri(2 * f + q, v.M, kx, ky);
                ob[q] = kx * v.s3 + (long long)ky * v.WS + u;
            }
#pragma unroll
            for (int i = 0; i < VPT; ++i) {
                const int m = E::last(i);
                if ((!HALF || i % R0 < R0 / 2) && u + m < v.WS) {   // the row's padding too: finite values (WS <= L)
                    B3[ob[0] + m] = x[i].x;
                    B3[ob[1] + m] = x[i].y;
                }
            }
        }
    }
}

// The same at 768 energies, which has no two-stage schedule at these register
// counts: three stages on the schedules and tables of et_tiles.cuh.
// THERMAL: Fermi weights; odd: the odd part (Im chi_T).
template <int L, bool THERMAL>
__global__ void __launch_bounds__(32 * EVC_WARPS)
k_ev_corr3(Geom g, EvGeom v, Band band, const float *B2, float *__restrict__ B3,
          const float2 *__restrict__ etw, int iters, int odd)
{
    using G = EtGeo<L>;
    constexpr int VPT = G::VPT, TPL = G::TPL, LPI = G::LPI, LP = G::LP;
    constexpr int R0 = G::R0, R1 = G::R1, R2 = G::R2, N1 = G::N1, N2 = G::N2, NB2 = L / R2;
    constexpr int S0 = et_radix(L, 0, true), S1 = et_radix(L, 1, true), S2 = et_radix(L, 2, true);
    constexpr int M1 = et_ns(L, 1, true), M2 = et_ns(L, 2, true);
    static_assert(S0 == R2 && VPT == 2 * S0, "the product stays in registers");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(EVC_WARPS * LPI * LP + (THERMAL ? L : 0), float2)
    after_previous();
    const int lane = (int)threadIdx.x % 32, warp = (int)threadIdx.x / 32;
    const int sl = lane / TPL, u = lane % TPL;
    float2 *sm = reinterpret_cast<float2 *>(smem_raw) + (warp * LPI + sl) * LP;
    float2 *wf = reinterpret_cast<float2 *>(smem_raw) + EVC_WARPS * LPI * LP;
    if constexpr (THERMAL) {
        et_fermi_weights<L>(g, band, wf, (int)threadIdx.x, 32 * EVC_WARPS);
        __syncthreads();
    }
    const float2 *tw1 = etw + et_table_offset(L, 1), *tw2 = etw + et_table_offset(L, 2);
    const float2 *iw1 = etw + et_table_offset(L, 1, true), *iw2 = etw + et_table_offset(L, 2, true);
    const int npairs = v.M / 2 * (v.M + 1) / 2;
    const int j2[2] = {u, u == 0 ? TPL : NB2 - u};
    const bool u0 = u == 0;

    for (int it = 0; it < iters; ++it) {
        const int f = ((blockIdx.x * EVC_WARPS + warp) * iters + it) * LPI + sl;
        const bool live = f < npairs;
        long long in[2], ob[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            int kx, ky;
            ev_tri(live ? 2 * f + q : 0, v.M, kx, ky);
            in[q] = kx * v.s2 + (long long)ky * v.ES;
            ob[q] = kx * v.s3 + (long long)ky * v.WS;
        }
        float raw[2][VPT];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int b = 0; b < VPT / R0; ++b)
#pragma unroll
                for (int r = 0; r < R0; ++r) {
                    const int n = u + b * TPL + r * (L / R0);
                    raw[q][b * R0 + r] = live && n < v.ne ? __ldcs(B2 + in[q] + n) : 0.f;
                }
        float2 pa[2][R2 / 2], pb[2][R2 / 2], ph[2], x[VPT];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            // forward transform of z = a + i b
#pragma unroll
            for (int b = 0; b < VPT / R0; ++b) {
#pragma unroll
                for (int r = 0; r < R0; ++r) {
                    const int n = u + b * TPL + r * (L / R0);
                    const float A = 0.5f * raw[q][b * R0 + r];   // the 1/2 of the separation below
                    if constexpr (THERMAL) {
                        const float2 w = wf[n];
                        x[b * R0 + r] = make_float2(A * w.x, A * w.y);
                    } else {
                        x[b * R0 + r] = n < v.J0 ? make_float2(A, 0.f) : make_float2(0.f, A);
                    }
                }
                Dft<R0, false, float2>::run(x + b * R0);
            }
            __syncwarp();
#pragma unroll
            for (int b = 0; b < VPT / R0; ++b) {
                float2 *p = sm + et_pad((u + b * TPL) * R0);
#pragma unroll
                for (int r = 0; r < R0; ++r) p[r] = x[b * R0 + r];
            }
            __syncwarp();
#pragma unroll
            for (int b = 0; b < VPT / R1; ++b) {
                const int j = u + b * TPL, pj = et_pad(j);
#pragma unroll
                for (int r = 0; r < R1; ++r) x[b * R1 + r] = sm[pj + et_pad(r * (L / R1))];
                et_twiddle<R1, false>(x + b * R1, reinterpret_cast<const float4 *>(tw1 + (j % N1) * R1));
                Dft<R1, false, float2>::run(x + b * R1);
            }
            __syncwarp();
#pragma unroll
            for (int b = 0; b < VPT / R1; ++b) {
                const int j = u + b * TPL, pb_ = et_pad((j / N1) * N2 + j % N1);
#pragma unroll
                for (int r = 0; r < R1; ++r) sm[pb_ + r * N1 + (r * N1) / 16] = x[b * R1 + r];
            }
            __syncwarp();
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int pj = et_pad(j2[b]);
#pragma unroll
                for (int r = 0; r < R2; ++r) x[b * R2 + r] = sm[pj + et_pad(r * NB2)];
                et_twiddle<R2, false>(x + b * R2, reinterpret_cast<const float4 *>(tw2 + j2[b] * R2));
                Dft<R2, false, float2>::run(x + b * R2);
            }
            // conj(a^) b^, a^ = Z(k) + conj Z(-k), b^ = (Z(k) - conj Z(-k)) / i
            // (halved in the input), k <= L/2; partners as in et_tiles.cuh
            auto prod = [&](float2 zk, float2 zm) {
                const float2 p = cmulc(make_float2(zk.y + zm.y, zm.x - zk.x), make_float2(zk.x + zm.x, zk.y - zm.y));
                return THERMAL ? odd_part(p, odd != 0) : p;
            };
#pragma unroll
            for (int r = 0; r < R2 / 2; ++r) {
                pa[q][r] = prod(x[r], u0 ? x[(R2 - r) % R2] : x[R2 + R2 - 1 - r]);
                pb[q][r] = prod(x[R2 + r], u0 ? x[R2 + R2 - 1 - r] : x[R2 - 1 - r]);
            }
            ph[q] = prod(x[R2 / 2], x[R2 / 2]);   // k = L/2, used where u = 0
        }
        // W(k) = P1 + i P2 and W(L - k) = conj P1 + i conj P2 in the inverse's
        // first-stage order (rows j2[b] + r NB2)
        auto w_of = [](float2 x1, float2 x2) { return make_float2(x1.x - x2.y, x1.y + x2.x); };
        auto w_conj = [](float2 x1, float2 x2) { return make_float2(x1.x + x2.y, x2.x - x1.y); };
#pragma unroll
        for (int r = 0; r < S0 / 2; ++r) {
            x[r] = w_of(pa[0][r], pa[1][r]);
            x[S0 + r] = w_of(pb[0][r], pb[1][r]);
            x[S0 + S0 - 1 - r] = u0 ? w_conj(pb[0][r], pb[1][r]) : w_conj(pa[0][r], pa[1][r]);
        }
        // u > 0: row S0 - 1 - r mirrors pb[r]; u = 0: row S0 - r mirrors pa[r], row S0/2 is k = L/2
#pragma unroll
        for (int r = S0 / 2; r < S0; ++r) {
            const float2 hi = w_conj(pb[0][S0 - 1 - r], pb[1][S0 - 1 - r]);
            const float2 lo = r == S0 / 2 ? w_of(ph[0], ph[1]) : w_conj(pa[0][(S0 - r) % (S0 / 2)], pa[1][(S0 - r) % (S0 / 2)]);
            x[r] = u0 ? lo : hi;
        }
        Dft<S0, true, float2>::run(x);
        Dft<S0, true, float2>::run(x + S0);
        __syncwarp();
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int base = j2[b] * S0;
#pragma unroll
            for (int r = 0; r < S0; ++r) sm[et_pad(base + r)] = x[b * S0 + r];
        }
        __syncwarp();
#pragma unroll
        for (int b = 0; b < VPT / S1; ++b) {
            const int j = u + b * TPL, pj = et_pad(j);
#pragma unroll
            for (int r = 0; r < S1; ++r) x[b * S1 + r] = sm[pj + et_pad(r * (L / S1))];
            et_twiddle<S1, true>(x + b * S1, reinterpret_cast<const float4 *>(iw1 + (j % M1) * S1));
            Dft<S1, true, float2>::run(x + b * S1);
        }
        __syncwarp();
#pragma unroll
        for (int b = 0; b < VPT / S1; ++b) {
            const int j = u + b * TPL, base = (j / M1) * M2 + j % M1;
#pragma unroll
            for (int r = 0; r < S1; ++r) sm[et_pad(base + r * M1)] = x[b * S1 + r];
        }
        __syncwarp();
#pragma unroll
        for (int b = 0; b < VPT / S2; ++b) {
            const int j = u + b * TPL, pj = et_pad(j);
#pragma unroll
            for (int r = 0; r < S2; ++r) x[b * S2 + r] = sm[pj + et_pad(r * (L / S2))];
            et_twiddle<S2, true>(x + b * S2, reinterpret_cast<const float4 *>(iw2 + j * S2));
            Dft<S2, true, float2>::run(x + b * S2);
        }
        if (live) {
#pragma unroll
            for (int b = 0; b < VPT / S2; ++b)
#pragma unroll
                for (int r = 0; r < S2; ++r) {
                    const int m = u + b * TPL + r * (L / S2);
                    if (m < v.WS) {   // the row's padding too: finite values (WS <= L)
                        B3[ob[0] + m] = x[b * S2 + r].x;
                        B3[ob[1] + m] = x[b * S2 + r].y;
                    }
                }
        }
        __syncwarp();
    }
}

template <int L, bool FULL, bool THERMAL, bool HALF>
cudaError_t launch_ev_corr_t(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, int sms,
                             cudaStream_t s)
{
    using E = EvLine<L>;
    const size_t smem = sizeof(float2) * (EVC_WARPS * E::WARP_ELEMS + (THERMAL ? L : 0));
    static const cudaError_t e = smem_attrs(k_ev_corr<L, FULL, THERMAL, HALF>, smem);
    if (e != cudaSuccess) return e;
    const int npairs = v.M / 2 * (v.M + 1) / 2, iters = ev_corr_iters(npairs, E::LPI, sms);
    const int per = EVC_WARPS * iters * E::LPI;
    return launch_after(k_ev_corr<L, FULL, THERMAL, HALF>, (npairs + per - 1) / per, 32 * EVC_WARPS, smem, s, g, v, band,
                        (const float *)w.Y, (float *)w.X, (const float2 *)w.evt + ev_line_table<L>(), iters,
                        g.quantity == LINDHARD_IMCHI_T);
}
template <int L>
cudaError_t launch_ev_corr_l(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, int sms,
                             cudaStream_t s)
{
    const bool half = v.WS <= L / 2;
    if (g.quantity != LINDHARD_IMCHI)
        return half ? launch_ev_corr_t<L, false, true, true>(g, v, band, w, sms, s)
                    : launch_ev_corr_t<L, false, true, false>(g, v, band, w, sms, s);
    if (v.ne == L && v.J0 == L / 2 && half) return launch_ev_corr_t<L, true, false, true>(g, v, band, w, sms, s);
    return half ? launch_ev_corr_t<L, false, false, true>(g, v, band, w, sms, s)
                : launch_ev_corr_t<L, false, false, false>(g, v, band, w, sms, s);
}
template <bool THERMAL>
cudaError_t launch_ev_corr3(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, int sms,
                            cudaStream_t s)
{
    constexpr int L = 768, LPI = EtGeo<L>::LPI;
    const size_t smem = sizeof(float2) * (EVC_WARPS * LPI * EtGeo<L>::LP + (THERMAL ? L : 0));
    static const cudaError_t e = smem_attrs(k_ev_corr3<L, THERMAL>, smem);
    if (e != cudaSuccess) return e;
    const int npairs = v.M / 2 * (v.M + 1) / 2, iters = ev_corr_iters(npairs, LPI, sms);
    const int per = EVC_WARPS * iters * LPI;
    return launch_after(k_ev_corr3<L, THERMAL>, (npairs + per - 1) / per, 32 * EVC_WARPS, smem, s, g, v, band,
                        (const float *)w.Y, (float *)w.X, (const float2 *)w.etw, iters,
                        g.quantity == LINDHARD_IMCHI_T);
}
cudaError_t launch_ev_corr(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, int sms,
                           cudaStream_t s)
{
    switch (v.PE) {
    case 128: return launch_ev_corr_l<128>(g, v, band, w, sms, s);
    case 256: return launch_ev_corr_l<256>(g, v, band, w, sms, s);
    case 384: return launch_ev_corr_l<384>(g, v, band, w, sms, s);
    case 512: return launch_ev_corr_l<512>(g, v, band, w, sms, s);
    case 768:
        return g.quantity != LINDHARD_IMCHI ? launch_ev_corr3<true>(g, v, band, w, sms, s)
                                            : launch_ev_corr3<false>(g, v, band, w, sms, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lh
