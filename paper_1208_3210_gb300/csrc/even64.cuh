// Geometry of the FP64 even form (k_even64.cu).
#pragma once

#include "kernels.cuh"

namespace lh {

// Transform lengths, both axes: the general FP64 form ends at 256 too, where the
// momentum axis is of 2 M.
__host__ __device__ constexpr int e64_len(int i)
{
    constexpr int n[] = {16, 24, 32, 48, 64, 96, 128, 192, 256};
    return i < 9 ? n[i] : 0;
}
// Tables (double2), one after another: e^{-2 pi i k / 4n}, k < 4n, per length n.
__host__ __device__ constexpr int e64_table(int n)
{
    int o = 0;
    for (int i = 0; e64_len(i) != 0 && e64_len(i) != n; ++i) o += 4 * e64_len(i);
    return o;
}
__host__ __device__ constexpr int e64_table_entries() { return e64_table(0); }

struct E64Geom {
    int M, Nh;         // frequencies per momentum axis; rows p = 0, ..., N/2
    int e0, ne, J0;    // energy window, occupied: j < J0
    int PE, ES, WS;    // energy transform; energies and transfers of a row (even)
    double scale;
};
inline bool e64_geom(const Geom &g, E64Geom &v)
{
    if (g.periodic) return false;
    v.e0 = 0;
    v.ne = g.n_eps;
    if (g.quantity == LINDHARD_IMCHI) {   // as in ev_geom
        const int lo = g.J0 - g.n_omega > 0 ? g.J0 - g.n_omega : 0;
        const int hi = g.J0 + g.n_omega < g.n_eps ? g.J0 + g.n_omega : g.n_eps;
        v.e0 = lo;
        v.ne = hi - lo;
    }
    v.J0 = g.J0 - v.e0;
    v.Nh = g.N / 2 + 1;
    const int need_m = (g.N + g.Q / 2 + 1) / 2, need_e = g.quantity == LINDHARD_IMCHI ? v.ne : g.n_eps + g.n_omega - 1;
    v.M = v.PE = 0;
    for (int i = 0; e64_len(i) != 0; ++i) {
        if (v.M == 0 && e64_len(i) >= need_m) v.M = e64_len(i);
        if (v.PE == 0 && e64_len(i) >= need_e) v.PE = e64_len(i);
    }
    if (v.M == 0 || v.M > 128 || v.PE == 0) return false;
    v.ES = (v.ne + 1) / 2 * 2;
    v.WS = (g.n_omega + 1) / 2 * 2;
    if (v.WS > v.PE) return false;
    v.scale = g.scale * ((double)g.P * g.P * g.PE) / (8.0 * (double)v.M * v.M * v.PE);
    return true;
}
// Doubles of the edge lines (and the M sines after them), behind B2 in Y.
__host__ __device__ inline size_t e64_lines(const E64Geom &v) { return 4 * (size_t)(v.M + 1) * (v.PE / 2 + 1); }
inline size_t e64_x_doubles(const E64Geom &v)
{
    const size_t a = (size_t)v.Nh * v.M * v.ES, b = 4 * (size_t)v.M * v.M * v.WS;
    return a > b ? a : b;
}
inline size_t e64_y_doubles(const Geom &g, const E64Geom &v)
{
    const size_t a = (size_t)v.M * v.M * v.ES + e64_lines(v) + v.M, b = 2 * (size_t)g.Q * v.M * v.WS;
    return a > b ? a : b;
}

}  // namespace lh
