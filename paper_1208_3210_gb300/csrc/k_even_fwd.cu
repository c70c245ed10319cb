// Forward momentum passes of the even form (even.cuh): A(p, e) generated
// (Eqs. 4-5) for p >= 0 and its cosine transforms along p_y and p_x
// (Sec. 3's transforms of the spectral function).
//
//   k_ev_gen_y : B1 [Nh][M][ES]: for each p_x >= 0, A over all p_y >= 0 for a
//                tile of energies, transformed along p_y
//   k_ev_x     : B2 [M][M][ES]: B1 transformed along p_x for each k_y; only
//                k_x <= k_y is written (A is symmetric under p_x <-> p_y and
//                both axes list their frequencies in the same order).  The
//                adjoint's weights take it too (k_even_bw.cu), with every k_x.
#include "even.cuh"
#include "even_line.cuh"

namespace lh {

// One block per table and slice: the tables' places and periods come as an
// argument (evaluating ev_table_offset per entry on the device took 0.5 ms).
struct EvTabs {
    struct { int off, count, row, period; } t[112];   // row 0: the w_j, j < period; row -1: even_line.cuh
};
__global__ void k_ev_tables(float2 *out, EvTabs tabs)
{
    const int off = tabs.t[blockIdx.x].off, count = tabs.t[blockIdx.x].count, row = tabs.t[blockIdx.x].row,
              period = tabs.t[blockIdx.x].period;
    for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < count; i += gridDim.y * blockDim.x) {
        double s, c;
        if (row == 0) sincospi(0.5 * (double)i / (double)period, &s, &c);
        else if (row > 0) sincospi(-2.0 * (double)((i / row) * (i % row + 1)) / (double)period, &s, &c);
        else sincospi(-2.0 * (double)((i % 64 / 2) * (i < 128 ? i / 64 * 2 + i % 2 + 1 : i % 2 ? 16 : 8)) / (double)period, &s, &c);
        out[off + i] = make_float2((float)c, (float)s);
    }
}
cudaError_t launch_ev_tables(float2 *out, cudaStream_t s)
{
    EvTabs tabs;
    int n = 0, o = 0;
    for (int i = 0; ev_len(i) != 0; ++i) {   // the order of ev_table_offset
        const int M = ev_len(i);
        tabs.t[n++] = {o, M, 0, M};
        o += M;
        for (int d = 0; d < 2; ++d)
            for (int st = 1; st < ev_nstages(M); ++st) {
                const int Ns = ev_ns(M, st, d != 0), R = ev_radix(M, st, d != 0);
                tabs.t[n++] = {o, Ns * ev_row(R), ev_row(R), Ns * R};
                o += Ns * ev_row(R);
            }
    }
    for (int i = 0; ev_line_len(i) != 0; ++i) tabs.t[n++] = {(o + 1) / 2 * 2 + EV_LINE_TABLE * i, EV_LINE_TABLE, -1, ev_line_len(i)};
    k_ev_tables<<<dim3(n, 4), 128, 0, s>>>(out, tabs);
    return cudaGetLastError();
}
size_t ev_table_bytes() { return (size_t)ev_all_tables() * sizeof(float2); }

// Grid: Nh x (column tiles), the tiles of one p_x neighbours.
template <int M>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB_GEN)
k_ev_gen_y(Geom g, EvGeom v, Band band, const AxisTab *axis, const float2 *eps,
           const InstState *st, float *__restrict__ B1, const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, false>;
    constexpr int C = F::C, T = F::T, VPT = F::VPT, TPC = F::TPC, RP = F::RP, NBP = F::NBP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float4)
    after_previous();
    float4 *sm = reinterpret_cast<float4 *>(smem_raw);
    const int jx = blockIdx.x / ntile, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;

    // band energy and amplitude of every row, once per tile (16 Nh bytes in the
    // exchange buffer, which has M > Nh rows of at least two packs)
    float4 *rows = sm;
    const int half = g.N / 2;   // the edge, where it is kept: index 0 of the axis, half its weight on either side
    const AxisTab ax = axis[jx == half ? 0 : half + jx];
    for (int i = threadIdx.x; i < v.Nh; i += T) {
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        band_point_f32(band, ax, axis[i == half ? 0 : half + i], st, q.x, q.y, q.z);
        if (jx == half) q.z *= 0.5f;
        if (i == half) q.z *= 0.5f;
        rows[i] = q;
    }
    __syncthreads();

    // energies e..e+3 of the window, as (hi, lo); past its end amplitude 0
    const int e = 4 * (ct * C + col);
    float2 eh[2], el[2], on[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int k = e + 2 * h;
        const float2 a = eps[v.e0 + min(k, v.ne - 1)], b = eps[v.e0 + min(k + 1, v.ne - 1)];
        eh[h] = make_float2(a.x, b.x);
        el[h] = make_float2(a.y, b.y);
        on[h] = make_float2(k < v.ne ? 1.f : 0.f, k + 1 < v.ne ? 1.f : 0.f);
    }
    const float2 g2 = dup2(band.gam2);
    Cx2 z[VPT];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const int j = F::template butterfly<0>(b, u);
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            const int n = j + r * NBP;
            float2 a[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
            if (n < v.Nh) {
                const float4 q = rows[n];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 d = add2(sub2(eh[h], dup2(q.x)), sub2(el[h], dup2(q.y)));
                    const float2 x = fma2(d, d, g2);
                    a[h] = mul2(mul2(on[h], dup2(q.z)), make_float2(rcp_approx(x.x), rcp_approx(x.y)));
                }
            }
            z[b * RP + r] = {a[0], a[1]};
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
                F::st(reinterpret_cast<float4 *>(o + (u + b * TPC + r * (M / RL)) * v.ES), z[b * RL + r]);
    }
}

// Grid: M x (column tiles), the tiles of one k_y neighbours.  Rows [0, rows) of
// planes of RS-float rows, sp floats apart in B1 and dp in B2.  TRI: k_x <= k_y.
template <int M, bool TRI>
__global__ void __launch_bounds__(EvCfg<M>::T, EvCfg<M>::MINB)
k_ev_x(int rows, int RS, long long sp, long long dp, const float *B1, float *__restrict__ B2,
       const float2 *__restrict__ tab, int ntile)
{
    using F = EvFft<M, false>;
    constexpr int C = F::C, VPT = F::VPT, TPC = F::TPC, RP = F::RP, NBP = F::NBP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LH_REQUIRE_SMEM(F::SMEM_ELEMS, float4)
    after_previous();
    float4 *sm = reinterpret_cast<float4 *>(smem_raw);
    const int ky = blockIdx.x / ntile, ct = blockIdx.x % ntile;
    const int col = threadIdx.x % C, u = threadIdx.x / C;
    const int e = 4 * (ct * C + col);
    const bool on = e < RS;
    const float *in = B1 + (long long)ky * RS + e;
    Cx2 z[VPT];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const int j = F::template butterfly<0>(b, u);
#pragma unroll
        for (int r = 0; r < RP; ++r) {
            const int n = j + r * NBP;
            z[b * RP + r] = on && n < rows ? ev_load(in + n * sp) : Cx2{dup2(0.f), dup2(0.f)};
        }
    }
    ev_pre<M>(z, u, tab);
    F::run(z, sm + col, u, tab);
    if (on) {
        float *o = B2 + (long long)ky * RS + e;
        constexpr int RL = ev_radix(M, F::NS - 1, false);
#pragma unroll
        for (int b = 0; b < VPT / RL; ++b)
#pragma unroll
            for (int r = 0; r < RL; ++r) {
                const int kx = u + b * TPC + r * (M / RL);
                if (!TRI || kx <= ky) F::st(reinterpret_cast<float4 *>(o + kx * dp), z[b * RL + r]);
            }
    }
}

template <int M>
cudaError_t launch_ev_gen_y_t(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, cudaStream_t s)
{
    const size_t smem = sizeof(float4) * EvFft<M, false>::SMEM_ELEMS;
    static const cudaError_t e = smem_attrs(k_ev_gen_y<M>, smem);
    if (e != cudaSuccess) return e;
    const int ntile = (v.ES + 4 * EvCfg<M>::C - 1) / (4 * EvCfg<M>::C);
    return launch_after(k_ev_gen_y<M>, v.Nh * ntile, EvCfg<M>::T, smem, s, g, v, band, w.axis, (const float2 *)w.eps,
                        w.state, (float *)w.X, (const float2 *)w.evt, ntile);
}
template <int M, bool TRI>
cudaError_t launch_ev_x_t(int rows, int RS, long long sp, long long dp, const float *src, float *dst,
                          const Work<float> &w, cudaStream_t s)
{
    const size_t smem = sizeof(float4) * EvFft<M, false>::SMEM_ELEMS;
    static const cudaError_t e = smem_attrs(k_ev_x<M, TRI>, smem);
    if (e != cudaSuccess) return e;
    const int ntile = (RS + 4 * EvCfg<M>::C - 1) / (4 * EvCfg<M>::C);
    return launch_after(k_ev_x<M, TRI>, M * ntile, EvCfg<M>::T, smem, s, rows, RS, sp, dp, src, dst,
                        (const float2 *)w.evt, ntile);
}
cudaError_t launch_ev_gen_y(const Geom &g, const EvGeom &v, const Band &band, const Work<float> &w, cudaStream_t s)
{
#define CALL(M_) launch_ev_gen_y_t<M_>(g, v, band, w, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}
cudaError_t launch_ev_x(const EvGeom &v, const Work<float> &w, cudaStream_t s)
{
#define CALL(M_) launch_ev_x_t<M_, true>(v.Nh, v.ES, v.s1, v.s2, (const float *)w.X, (float *)w.Y, w, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}
cudaError_t launch_ev_x_all(const EvGeom &v, const Work<float> &w, const float *src, float *dst, cudaStream_t s)
{
#define CALL(M_) launch_ev_x_t<M_, false>(v.nl < v.M ? v.nl : v.M, v.WS, v.s4, v.s3, src, dst, w, s)
    LH_EV_SWITCH(v.M, CALL)
#undef CALL
}

}  // namespace lh
