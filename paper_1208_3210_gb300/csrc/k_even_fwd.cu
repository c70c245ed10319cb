// Forward momentum passes of the even form (even.cuh): A(p, e) generated
// (Eqs. 4-5) for p >= 0 and its cosine transforms along p_y and p_x
// (Sec. 3's transforms of the spectral function).
//
//   k_ev_gen_y : B1 [Nh][M][ES]: for each p_x >= 0, A over all p_y >= 0 for a
//                tile of energies, transformed along p_y
//   k_ev_x     : B2 [M][M][ES]: B1 transformed along p_x for each k_y; only
//                k_x <= k_y is written (A is symmetric under p_x <-> p_y and
//                both axes list their frequencies in the same order)
#include "even.cuh"

namespace lh {

// One block per table and slice: the tables' places and periods come as an
// argument (evaluating ev_table_offset per entry on the device took 0.5 ms).
struct EvTabs {
    struct { int off, count, period; } t[64];   // period 0: the w_j of length `count`
};
__global__ void k_ev_tables(float2 *out, EvTabs tabs)
{
    const int off = tabs.t[blockIdx.x].off, count = tabs.t[blockIdx.x].count, period = tabs.t[blockIdx.x].period;
    for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < count; i += gridDim.y * blockDim.x) {
        double s, c;
        if (period == 0) sincospi(0.5 * (double)i / (double)count, &s, &c);
        else sincospi(-2.0 * (double)((i / 2) * (i % 2 + 1)) / (double)period, &s, &c);
        out[off + i] = make_float2((float)c, (float)s);
    }
}
cudaError_t launch_ev_tables(float2 *out, cudaStream_t s)
{
    EvTabs tabs;
    int n = 0, o = 0;
    for (int i = 0; ev_len(i) != 0; ++i) {   // the order of ev_table_offset
        const int M = ev_len(i);
        tabs.t[n++] = {o, M, 0};
        o += M;
        for (int d = 0; d < 2; ++d)
            for (int st = 1; st < ev_nstages(M); ++st) {
                const int Ns = ev_ns(M, st, d != 0);
                tabs.t[n++] = {o, 2 * Ns, Ns * ev_radix(M, st, d != 0)};
                o += 2 * Ns;
            }
    }
    k_ev_tables<<<dim3(n, 4), 128, 0, s>>>(out, tabs);
    return cudaGetLastError();
}
size_t ev_table_bytes() { return (size_t)ev_table_entries() * sizeof(float2); }

// Grid: Nh x (column tiles), the tiles of one p_x neighbours.
template <int M>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_ev_gen_y(Geom g, EvGeom v, Band band, const AxisTab *__restrict__ axis, const float2 *__restrict__ eps,
           const InstState *__restrict__ st, float *__restrict__ B1, const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, false>;
    constexpr int C = F::C, T = F::T, VPT = F::VPT, TPC = F::TPC, RP = F::RP, NBP = F::NBP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float2)
    float2 *sm = reinterpret_cast<float2 *>(smem_raw);
    const int jx = blockIdx.x / ntile, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;

    // band energy and amplitude of every row, once per tile (3 Nh floats in
    // the exchange buffer: Nh <= M and at least 4 columns of 8 bytes)
    float *bx = reinterpret_cast<float *>(smem_raw), *bl = bx + v.Nh, *ba = bl + v.Nh;
    const AxisTab ax = axis[g.N / 2 + jx];
    for (int i = threadIdx.x; i < v.Nh; i += T)
        band_point_f32(band, ax, axis[g.N / 2 + i], st, bx[i], bl[i], ba[i]);
    __syncthreads();

    // energies 2c, 2c + 1 of the window; columns past its end hold zeros
    const int e = 2 * (ct * C + col);
    const float2 e0 = e < v.ne ? __ldg(&eps[v.e0 + e]) : make_float2(0.f, 0.f);
    const float2 e1 = e + 1 < v.ne ? __ldg(&eps[v.e0 + e + 1]) : make_float2(0.f, 0.f);
    const float on0 = e < v.ne ? 1.f : 0.f, on1 = e + 1 < v.ne ? 1.f : 0.f;
    const float g2 = band.gam2;
    float2 z[VPT];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const int j = F::template butterfly<0>(b, u);
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            const int n = j + r * NBP;
            float2 a = make_float2(0.f, 0.f);
            if (n < v.Nh) {
                const float xhi = bx[n], xlo = bl[n], amp = ba[n];
                const float d0 = (e0.x - xhi) + (e0.y - xlo), d1 = (e1.x - xhi) + (e1.y - xlo);
                a = make_float2(on0 * amp * __fdividef(1.0f, fmaf(d0, d0, g2)),
                                on1 * amp * __fdividef(1.0f, fmaf(d1, d1, g2)));
            }
            z[b * RP + r] = a;
        }
    }
    ev_pre<M>(z, u, tab);
    __syncthreads();   // the rows' values have been read
    F::run(z, sm + col, u, tab);
    if (e < v.ES) {
        float *o = B1 + (long long)jx * v.s1 + e;
        constexpr int RL = ev_radix(M, F::NS - 1, false);
#pragma unroll
        for (int b = 0; b < VPT / RL; ++b)
#pragma unroll
            for (int r = 0; r < RL; ++r)
                *reinterpret_cast<float2 *>(o + (long long)(u + b * TPC + r * (M / RL)) * v.ES) = z[b * RL + r];
    }
}

// Grid: M x (column tiles), the tiles of one k_y neighbours.
template <int M>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_ev_x(EvGeom v, const float *__restrict__ B1, float *__restrict__ B2, const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, false>;
    constexpr int C = F::C, VPT = F::VPT, TPC = F::TPC, RP = F::RP, NBP = F::NBP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float2)
    float2 *sm = reinterpret_cast<float2 *>(smem_raw);
    const int ky = blockIdx.x / ntile, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;
    const int e = 2 * (ct * C + col);
    const bool on = e < v.ES;
    const float *in = B1 + (long long)ky * v.ES + e;
    float2 z[VPT];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const int j = F::template butterfly<0>(b, u);
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            const int n = j + r * NBP;
            z[b * RP + r] = on && n < v.Nh ? __ldcs(reinterpret_cast<const float2 *>(in + n * v.s1))
                                           : make_float2(0.f, 0.f);
        }
    }
    ev_pre<M>(z, u, tab);
    F::run(z, sm + col, u, tab);
    if (on) {
        float *o = B2 + (long long)ky * v.ES + e;
        constexpr int RL = ev_radix(M, F::NS - 1, false);
#pragma unroll
        for (int b = 0; b < VPT / RL; ++b)
#pragma unroll
            for (int r = 0; r < RL; ++r) {
                const int kx = u + b * TPC + r * (M / RL);
                if (kx <= ky) *reinterpret_cast<float2 *>(o + kx * v.s2) = z[b * RL + r];
            }
    }
}

template <int M>
cudaError_t launch_ev_gen_y_t(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, cudaStream_t s)
{
    const size_t smem = sizeof(float2) * EvFft<M, false>::SMEM_ELEMS;
    static const cudaError_t e = smem_attrs(k_ev_gen_y<M>, smem);
    if (e != cudaSuccess) return e;
    const int ntile = (v.ES + 2 * EvCfg<M>::C - 1) / (2 * EvCfg<M>::C);
    k_ev_gen_y<M><<<v.Nh * ntile, EvCfg<M>::T, smem, s>>>(g, v, band, w.axis, (const float2 *)w.eps, w.state,
                                                          (float *)w.X, (const float2 *)w.evt, ntile);
    return cudaGetLastError();
}
template <int M>
cudaError_t launch_ev_x_t(const EvGeom &v, const Work<float> &w, cudaStream_t s)
{
    const size_t smem = sizeof(float2) * EvFft<M, false>::SMEM_ELEMS;
    static const cudaError_t e = smem_attrs(k_ev_x<M>, smem);
    if (e != cudaSuccess) return e;
    const int ntile = (v.ES + 2 * EvCfg<M>::C - 1) / (2 * EvCfg<M>::C);
    k_ev_x<M><<<M * ntile, EvCfg<M>::T, smem, s>>>(v, (const float *)w.X, (float *)w.Y, (const float2 *)w.evt, ntile);
    return cudaGetLastError();
}
cudaError_t launch_ev_gen_y(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, cudaStream_t s)
{
#define CALL(M_) launch_ev_gen_y_t<M_>(g, v, band, w, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}
cudaError_t launch_ev_x(const EvGeom &v, const Work<float> &w, cudaStream_t s)
{
#define CALL(M_) launch_ev_x_t<M_>(v, w, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}

}  // namespace lh
