// Set-up kernels: twiddle tables, per-axis momentum tables, the energy grid,
// and the rigid-band chemical potential (Sec. 3: the Fermi level is shifted to
// hold the requested electron count).
#include <math.h>
#include <stddef.h>

#include "kernels.cuh"

namespace lh {

// Every twiddle table (see twiddle_offset), FP64 sincospi.
__global__ void k_twiddles(int max_len, float2 *tw32, double2 *tw64)
{
    (void)max_len;
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= twiddle_entries()) return;
    int L, n;
    if (idx < 8176) {                       // powers of two
        L = 16;
        while (2 * L - 16 <= idx) L *= 2;   // the table that holds idx
        n = idx - (L - 16);
    } else {                                // 3 * 2^k
        int r = idx - 8176;
        L = 48;
        while (2 * L - 48 <= r) L *= 2;
        n = r - (L - 48);
    }
    double s, c;
    sincospi(-2.0 * (double)n / (double)L, &s, &c);
    tw32[idx] = make_float2((float)c, (float)s);
    tw64[idx] = make_double2(c, s);
}

// ---------------------------------------------------------------------------
// Set-up and chemical potential.
//
// Tables: per-axis values at p_i = (i - N/2) 2 pi / npz and the energy grid
// e_j = -e_max + (j + 1/2) de, all in FP64.  The FP32 path stores e_j as an
// unevaluated pair hi + lo so that e_j - xi_p keeps full precision near the
// Lorentzian peak.
//
// Chemical potential (Sec. 3: the Fermi level is placed to hold the requested
// electron count).  n(mu) = (2/npz^2) sum_k occ(e0_k - mu) with the Lorentzian
// occupation occ(xi) = 1/2 - atan(xi/gamma)/pi of Eq. 5 below the Fermi level,
// summed over the first-zone grid p = 2 pi r / npz, r in [-npz/2, npz/2).
// n is strictly increasing in mu.  Both band kinds depend on p_x and p_y only
// through even functions (cos p, cos 2p, p^2) and are symmetric under
// p_x <-> p_y, so the sum runs over the classes m = |r| in [0, npz/2] with
// weights w(0) = w(npz/2) = 1, w(m) = 2 otherwise, and over pairs
// m_x <= m_y (twice for m_x < m_y): (npz/2 + 1)(npz/2 + 2)/2 terms instead of
// npz^2 (561 instead of 4096 at npz = 64).
//
// Launches (no CTA ever waits for another; zones of at most 160 points per
// axis instead solve in one CTA of k_setup, see mu_solve_one_cta):
//   k_setup     multisection pass 0 over [-B-3, B+3] eV on G CTAs, and the
//               tables on further CTAs of the same launch (their FP64 cospi and
//               exp chains run beside the multisection, not before it)
//   k_mu_sect   further multisection passes (one, or two when gamma < 0.02 eV)
//   k_mu_halley one FP64 Halley step from the midpoint of the last bracket
// A multisection pass samples NC = 8 G candidates (G CTAs, eight candidates
// each) in FP32.  Every CTA sums the whole zone for its own candidates (the
// pairs' band energies and weights staged in shared memory, lane % 8 picks
// the candidate), so no cross-CTA reduction is needed; it records the first
// of its candidates whose total reaches the target, and the next launch's CTAs
// each take the minimum over the G records.  Two passes shrink the bracket by
// (NC - 1)^2 (to about 1e-5 eV), three to below FP32 resolution; FP32
// rounding moves the sampled n(mu) by the equivalent of some 1e-7 eV at most.
// The Halley step (cubic convergence; its error is of order (d/gamma)^2 d for
// a distance d to the root) then lands at FP64 precision.  Its per-CTA sums of
// n (FP64), gamma n' and gamma^2 n'' (FP32 terms: they only scale the step)
// are stored, and the last CTA to finish (an atomic counter) adds them in a
// fixed tree order and forms the step.
//
// On this GPU a dependent FP64 operation takes about 60 cycles, an FP64
// division about 450 and an FP64 atan about 1900, so the few FP64 steps on
// the critical path use constants computed on the host.
constexpr int MU_THREADS = 512;      // multisection CTAs
constexpr int MU_NT_THREADS = 128;   // Halley CTAs (at most; one warp when the pairs fit)
constexpr int MU_TAB_THREADS = 32;   // table entries per table CTA
constexpr int MU_NCPT = 8;           // candidates per CTA
constexpr int MU_MAX_PASSES = 3;
constexpr int MU_RES = 16;           // doubles of results at the start of acc
constexpr int MU_MAXC = 2049;        // classes for npz <= 4096
constexpr int MU_CHUNK = 2048;       // pairs staged per round
constexpr float MU_SECT_SCALE = 4294967296.0f;   // 2^32

// Layout of acc: res[3 p + 0, 1, 2] = (lo, hi, not-bracketed flag) of the
// interval pass p sampled (p = passes: that of the Halley step); then
// [G][4] doubles of per-CTA Halley sums; then [MU_MAX_PASSES][G] int first
// crossings (index in the CTA's candidates, MU_NCPT = none).
size_t mu_acc_doubles(int G) { return MU_RES + 4 * (size_t)G + ((size_t)MU_MAX_PASSES * G + 1) / 2; }
size_t mu_barrier_words() { return 32; }   // the arrival counter (one 128-byte line)

// CTAs of each chemical-potential launch: one per SM.
int mu_grid_size(int num_sms, int npts)
{
    (void)npts;
    return num_sms < 1 ? 1 : num_sms;
}

// Host-computed constants of one solve.
struct MuConst {
    double inv_nc1;      // 1 / (NC - 1)
    double inv_gam;      // 1 / gamma
    double target;       // filling npz^2 / 2 (sum of occupations)
    long long target32;  // the same in 2^-32 fixed point
    double B;            // bracket half-width - 3 eV
    int NC, passes;
    int single;          // the whole solve in one CTA of the set-up launch
    // of the one-CTA solve: the filling, and as FP32 pairs 1/gamma and
    // e^{i pi (npz^2 / 2 - target)}
    float target_f, Bf, igh, igl, cth, ctl, sth, stl;
    float step_tol;      // the last step is not repeated at this length
    int narrow;          // it sums arctangents in FP64
};

// Zones small enough for the one-CTA solve: the whole search and the final step
// in one CTA of the set-up launch, beside the table CTAs, and no further launch
// (npz <= 160).  The multi-CTA passes cost two more launches and their
// grid-wide exchanges (36 us in all at npz = 128, the one-CTA solve 25 us).
constexpr int MU_SINGLE_MAX_H = 80;
constexpr int MU_SINGLE_MAX_PAIRS = (MU_SINGLE_MAX_H + 1) * (MU_SINGLE_MAX_H + 2) / 2;   // 3321
__host__ __device__ inline bool mu_single(const Geom &g)
{
    const int h = g.npz / 2;
    return (h + 1) * (h + 2) / 2 <= MU_SINGLE_MAX_PAIRS;
}

__device__ __forceinline__ int *mu_cross(double *acc, int G, int pass)
{
    return (int *)(acc + MU_RES + 4 * (size_t)G) + (size_t)pass * G;
}

__device__ __forceinline__ double band_e0(const Band &b, const AxisTab &ax, const AxisTab &ay)
{
    if (b.band_kind == 1) return 0.5 * (ax.p2 + ay.p2);
    return -2.0 * b.t * (ax.c1 + ay.c1) - 4.0 * b.tp * ax.c1 * ay.c1 - 2.0 * b.tpp * (ax.c2 + ay.c2);
}

__device__ __forceinline__ ClsTab class_values(int m, int npz)
{
    auto pair = [](double v, float &hi, float &lo) {
        hi = (float)v;
        lo = (float)(v - (double)hi);
    };
    const double u = 2.0 * (double)m / (double)npz, p = u * 3.14159265358979323846;
    ClsTab t;
    t.c1 = cospi(u);
    t.c2 = cospi(2.0 * u);
    pair(t.c1, t.c1h, t.c1l);
    pair(t.c2, t.c2h, t.c2l);
    pair(p * p, t.p2h, t.p2l);
    return t;
}
__global__ void k_classes(int npz, ClsTab *cls)
{
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m <= npz / 2) cls[m] = class_values(m, npz);
}
cudaError_t launch_classes(int npz, ClsTab *cls, cudaStream_t s)
{
    k_classes<<<npz / 2 / 64 + 1, 64, 0, s>>>(npz, cls);
    return cudaGetLastError();
}

// Pair index k in [0, (h+1)(h+2)/2) -> classes (a, b), 0 <= a <= b <= h, row
// a holding b = a..h; row a starts at a (2h + 3 - a) / 2.
__device__ __forceinline__ void tri_pair(int k, int h, int &a, int &b)
{
    const float c = 2.0f * (float)h + 3.0f;
    int x = (int)((c - sqrtf(c * c - 8.0f * (float)k)) * 0.5f);
    x = max(0, min(x, h));
    while (x < h && (x + 1) * (2 * h + 2 - x) / 2 <= k) ++x;
    while (x > 0 && x * (2 * h + 3 - x) / 2 > k) --x;
    a = x;
    b = x + (k - x * (2 * h + 3 - x) / 2);
}
// Multiplicity of pair (a, b): w(a) w(b), twice when a != b.
__device__ __forceinline__ int pair_weight(int a, int b, int h)
{
    int wa = (a == 0 || a == h) ? 1 : 2, wb = (b == 0 || b == h) ? 1 : 2;
    return wa * wb * (a == b ? 1 : 2);
}

struct MuBracket {
    int wmin[MU_THREADS / 32];
    double lo, hi, step;
    int flag;
};
struct MuShared {
    float c1[MU_MAXC], c2[MU_MAXC], p2[MU_MAXC];   // class values in FP32
    float2 ew[MU_CHUNK];                           // (band energy, weight) of staged pairs
    long long red[MU_THREADS / 32][MU_NCPT];
    float mu_c[MU_NCPT];
    MuBracket br;
};

// Class values at p = 2 pi m / npz, FP32 (the multisection only needs them to
// about 1e-7).
__device__ __forceinline__ void stage_classes(const Geom &g, MuShared &sh)
{
    const int h = g.npz / 2;
    const float inv = 2.0f / (float)g.npz;
    for (int m = threadIdx.x; m <= h; m += blockDim.x) {
        float u = (float)m * inv;                  // p / pi
        float p = u * 3.14159265358979f;
        sh.c1[m] = cospif(u);
        sh.c2[m] = cospif(2.0f * u);
        sh.p2[m] = p * p;
    }
}

// Bracket from the first-crossing records of pass p: sh.lo, sh.hi, sh.flag
// (read after the next __syncthreads).  Every thread takes part.
__device__ __forceinline__ void bracket_from(const double *res, const int *cross_p, const MuConst &mc, int p,
                                             MuBracket &sh)
{
    const int G = mc.NC / MU_NCPT;
    double plo = 0.0, phi = 0.0, pflag = 0.0;
    if (threadIdx.x == 0) {   // issued together with the records' loads
        plo = __ldcg(res + 3 * p);
        phi = __ldcg(res + 3 * p + 1);
        pflag = __ldcg(res + 3 * p + 2);
    }
    int first = mc.NC;
    for (int j = threadIdx.x; j < G; j += blockDim.x) {
        int q = __ldcg(cross_p + j);
        if (q < MU_NCPT) first = min(first, MU_NCPT * j + q);
    }
    first = (int)__reduce_min_sync(0xffffffffu, (unsigned)first);
    if ((threadIdx.x & 31) == 0) sh.wmin[threadIdx.x >> 5] = first;
    __syncthreads();
    if (threadIdx.x == 0) {
        int c = mc.NC;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) c = min(c, sh.wmin[w]);
        sh.flag = pflag != 0.0 || (p == 0 && (c == 0 || c == mc.NC));
        c = max(1, min(c, mc.NC - 1));
        const double step = (phi - plo) * mc.inv_nc1;
        sh.lo = plo + (double)(c - 1) * step;
        sh.hi = sh.lo + step;
    }
}

// One multisection pass over [sh.br.lo, sh.br.hi] (set by thread 0 before the
// call): this CTA's candidates; records the first one whose total reaches
// the target in cross[blockIdx.x].
// Band energies and weights of pairs [base, base + n) into sh.ew (FP32).
__device__ __forceinline__ void stage_pairs(const Geom &g, const Band &band, MuShared &sh, int base, int n)
{
    const int h = g.npz / 2;
    const float t = (float)band.t, tp = (float)band.tp, tpp = (float)band.tpp;
    const bool free_e = band.band_kind == 1;
    for (int k = threadIdx.x; k < n; k += MU_THREADS) {
        int a, b;
        tri_pair(base + k, h, a, b);
        const float e = free_e ? 0.5f * (sh.p2[a] + sh.p2[b])
                               : -2.0f * t * (sh.c1[a] + sh.c1[b]) - 4.0f * tp * sh.c1[a] * sh.c1[b]
                                     - 2.0f * tpp * (sh.c2[a] + sh.c2[b]);
        sh.ew[k] = make_float2(e, (float)pair_weight(a, b, h));
    }
}

// prestaged: the first chunk of pairs is already in sh.ew (staged before the
// bracket was known; the classes must then have been staged and synchronised)
__device__ __forceinline__ void sect_pass(const Geom &g, const Band &band, const MuConst &mc, MuShared &sh,
                                          int *cross, bool prestaged = false)
{
    const int h = g.npz / 2;
    const int npairs = (h + 1) * (h + 2) / 2;
    const int c0 = MU_NCPT * blockIdx.x;
    if (threadIdx.x == 0) sh.br.step = (sh.br.hi - sh.br.lo) * mc.inv_nc1;
    __syncthreads();
    if (threadIdx.x < MU_NCPT) sh.mu_c[threadIdx.x] = (float)(sh.br.lo + (double)(c0 + (int)threadIdx.x) * sh.br.step);
    const float inv_gam = (float)mc.inv_gam, inv_pi = 0.318309886183790672f;
    const int q = threadIdx.x % MU_NCPT;        // this thread's candidate
    constexpr int LANES = MU_THREADS / MU_NCPT;  // threads per candidate
    long long acc = 0;
    for (int base = 0; base < npairs; base += MU_CHUNK) {
        const int n = min(MU_CHUNK, npairs - base);
        __syncthreads();   // previous chunk consumed; mu_c written
        if (!(prestaged && base == 0)) stage_pairs(g, band, sh, base, n);
        __syncthreads();
        const float mu = sh.mu_c[q];
        float s[4] = {0.f, 0.f, 0.f, 0.f};   // four chains; at most MU_CHUNK / LANES terms of at most 8
        int k = threadIdx.x / MU_NCPT;
        for (; k + 3 * LANES < n; k += 4 * LANES) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float2 ew = sh.ew[k + u * LANES];
                s[u] += ew.y * (0.5f - atanf((ew.x - mu) * inv_gam) * inv_pi);
            }
        }
        for (; k < n; k += LANES) {
            const float2 ew = sh.ew[k];
            s[0] += ew.y * (0.5f - atanf((ew.x - mu) * inv_gam) * inv_pi);
        }
        acc += __float2ll_rn(((s[0] + s[1]) + (s[2] + s[3])) * MU_SECT_SCALE);
    }
    // lanes l, l ^ 8, l ^ 16, l ^ 24 share a candidate
    acc += __shfl_xor_sync(0xffffffffu, acc, 8);
    acc += __shfl_xor_sync(0xffffffffu, acc, 16);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane < MU_NCPT) sh.red[warp][lane] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        long long tsum = 0;
        if (lane < MU_NCPT)
            for (int w = 0; w < MU_THREADS / 32; ++w) tsum += sh.red[w][lane];
        unsigned hit = __ballot_sync(0xffffffffu, lane < MU_NCPT && tsum >= mc.target32);
        if (lane == 0) cross[blockIdx.x] = hit ? __ffs(hit) - 1 : MU_NCPT;
    }
    (void)c0;
}

// One-CTA solve (mu_single).
//
// 1. One multisection pass in FP32 over [-B - 3, B + 3], a warp a candidate
//    (its lanes sum the pairs; no exchange but the candidates' totals), to a
//    bracket of about 0.7 eV.
// 2. A bracketed Halley iteration in FP32 over all threads, to 1e-6 eV (a step
//    that leaves the bracket, or a flat n, falls back to bisection).
// 3. A Halley step in twice FP32 precision.  The occupations' sum needs
//    Theta = sum w atan(x_k), and that is the argument of prod (1 + i x_k)^w:
//    the product is formed in unevaluated FP32 pairs (each factor scaled to
//    modulus 1 by an FP32 factor, which leaves its argument), multiplied by
//    e^{-i Theta_target} from the host, and the remaining angle, some 1e-2 at
//    most after step 2, comes from three terms of its series: no arctangent,
//    and no multiple of 2 pi to find.  The product's rounding is some 1e-12 of
//    an electron state, 1e-15 eV; the step itself, below 1e-6 eV, is FP32.
//    Below MU_PAIR_GAMMA the angle left is no longer small (a level of weight 8
//    turns it by 8 d / gamma), and the step sums the arctangents in FP64.
// 4. Where n(mu) is flat (nearly empty or full bands) the FP32 search ends
//    farther off, its sums being rounded at 1e-3 of a state, and for narrow
//    Lorentzians the remainder (d / gamma)^2 d of a step d counts: step 3 is
//    repeated until d^3 <= 1e-13 gamma^2, d = 6e-6 eV at gamma = 0.05.  So it runs
//    once at ordinary fillings.  Replayed on the CPU for gamma from 1e-6 to 1 eV
//    and fillings from 0.001 to 1.999: mu within 4e-12 eV and no filling refused
//    that has a root (with one step 8e-9 at gamma = 1e-5, and some refused).
//
// What bounds it is one SM's latency.  FP64 units are what it avoids: they
// retire two operations a cycle and SM, so a warp's FP64 instruction takes 16
// cycles whatever its lanes hold; the FP64 arctangents of the last step and the
// cosines of the classes (now laid out once per plan) were most of the time.
// Set-up and solve at npz = 64: 22.9 -> 14.4 us, mu within 2e-15 eV on average
// (9e-15 before; the product in FP64 by two warps: 17 us, its errors no smaller).
// The test whether to repeat the step costs some 0.7 us of it.
constexpr int MU_NEWTON_MAX = 64;    // bisection alone reaches 1e-6 eV in 24 steps
constexpr int MU_STEP_MAX = 8;
constexpr double MU_PAIR_GAMMA = 0.002;   // eV
struct C2 { F2 r, i; };
__device__ __forceinline__ F2 f2_div(F2 a, F2 b)
{
    const float q = a.h / b.h;
    return f2_fast(q, (fmaf(-q, b.h, a.h) + a.l - q * b.l) / b.h);
}
__device__ __forceinline__ F2 f2_neg(F2 a) { return {-a.h, -a.l}; }
__device__ __forceinline__ C2 c2_mul(C2 a, C2 b)
{
    return {f2_add(f2_mul(a.r, b.r), f2_neg(f2_mul(a.i, b.i))), f2_add(f2_mul(a.r, b.i), f2_mul(a.i, b.r))};
}
__device__ __forceinline__ F2 f2_shfl(F2 a, int o)
{
    return {__shfl_down_sync(0xffffffffu, a.h, o), __shfl_down_sync(0xffffffffu, a.l, o)};
}
__device__ __forceinline__ C2 c2_shfl(C2 a, int o) { return {f2_shfl(a.r, o), f2_shfl(a.i, o)}; }
struct MuSingle {
    float2 ew[MU_SINGLE_MAX_PAIRS];            // (band energy, weight) of the pairs
    F2 c1[MU_SINGLE_MAX_H + 1], c2[MU_SINGLE_MAX_H + 1], p2[MU_SINGLE_MAX_H + 1];   // cos p, cos 2p, p^2
    float cnt[MU_THREADS / 32];                // totals of the first pass's candidates
    float red[2][MU_THREADS / 32][3];          // warp sums of a Halley step
    C2 z[MU_THREADS / 32];                     // warp products and sums of the last step
    F2 n1[MU_THREADS / 32];
    float d2[MU_THREADS / 32];
    double f64[MU_THREADS / 32];
    F2 mu, step;                               // the last step's result and the step
    int done;
};
// The Halley step from mu, added to mu, in FP64 (thread 0 returns it; every
// thread takes part).  Not inlined: its FP64 constants would be formed by every
// solve (256 cycles an operation over the CTA's warps).
__device__ __noinline__ F2 mu_step_fp64(MuSingle &sh, F2 mu2, int h, bool free_e, double t, double tp, double tpp,
                                        double inv_gam, double target)
{
    constexpr int NW = MU_THREADS / 32;
    const int npairs = (h + 1) * (h + 2) / 2, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto wide = [](F2 a) { return (double)a.h + (double)a.l; };
    const double ipi = 0.31830988618379067154, mu = wide(mu2);
    double f = 0.0;
    float d1 = 0.f, d2 = 0.f;
    for (int k = threadIdx.x; k < npairs; k += MU_THREADS) {
        int a, b;
        tri_pair(k, h, a, b);
        const double c1a = wide(sh.c1[a]), c1b = wide(sh.c1[b]), w = pair_weight(a, b, h);
        const double e0 = free_e ? 0.5 * (wide(sh.p2[a]) + wide(sh.p2[b]))
                                 : -2.0 * t * (c1a + c1b) - 4.0 * tp * c1a * c1b
                                       - 2.0 * tpp * (wide(sh.c2[a]) + wide(sh.c2[b]));
        const double x = (e0 - mu) * inv_gam;
        f += w * (0.5 - atan(x) * ipi);
        const float xf = (float)x, r = 1.0f / (1.0f + xf * xf);
        d1 += (float)w * r;
        d2 += (float)w * 2.0f * xf * r * r;
    }
    F2 n1{d1, 0.f};
    for (int o = 16; o > 0; o >>= 1) {
        f += __shfl_down_sync(0xffffffffu, f, o);
        n1 = f2_add(n1, F2{__shfl_down_sync(0xffffffffu, n1.h, o), __shfl_down_sync(0xffffffffu, n1.l, o)});
        d2 += __shfl_down_sync(0xffffffffu, d2, o);
    }
    if (lane == 0) { sh.f64[warp] = f; sh.n1[warp] = n1; sh.d2[warp] = d2; }
    __syncthreads();
    if (threadIdx.x != 0) return F2{0.f, 0.f};
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int w = 0; w < NW; ++w) { s0 += sh.f64[w]; s1 += wide(sh.n1[w]); s2 += (double)sh.d2[w]; }
    const double d = s0 - target, dd1 = s1 * ipi * inv_gam, dd2 = s2 * ipi * inv_gam * inv_gam;
    const double step = -2.0 * d * dd1 / (2.0 * dd1 * dd1 - d * dd2);
    const float hi = (float)step;
    return F2{hi, (float)(step - (double)hi)};
}
// The same in twice FP32 precision.
__device__ __forceinline__ F2 mu_step_pairs(const Geom &g, const Band &band, const MuConst &mc, MuSingle &sh, F2 mu)
{
    constexpr int NW = MU_THREADS / 32;
    const int h = g.npz / 2, npairs = (h + 1) * (h + 2) / 2, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool free_e = band.band_kind == 1;
    const F2 igp{mc.igh, mc.igl}, mm = f2_neg(mu);
    const F2 k1{band.k1[0], band.k1[1]}, k2{band.k2[0], band.k2[1]}, k3{band.k3[0], band.k3[1]};
    const F2 one{1.f, 0.f}, nil{0.f, 0.f};
    C2 z8{one, nil}, z4{one, nil}, z1{one, nil};   // products of the factors of weight 8, 4, and 1 or 2
    float d1 = 0.f, d2 = 0.f;
    for (int k = threadIdx.x; k < npairs; k += MU_THREADS) {
        int a, b;
        tri_pair(k, h, a, b);
        const int w = pair_weight(a, b, h);
        F2 e0;
        if (free_e) {
            e0 = f2_add(sh.p2[a], sh.p2[b]);
            e0.h *= 0.5f;
            e0.l *= 0.5f;
        } else {
            e0 = f2_add(f2_add(f2_mul(k1, f2_add(sh.c1[a], sh.c1[b])), f2_mul(k2, f2_mul(sh.c1[a], sh.c1[b]))),
                        f2_mul(k3, f2_add(sh.c2[a], sh.c2[b])));
        }
        const F2 x = f2_mul(f2_add(e0, mm), igp);
        const float q = 1.0f + x.h * x.h, s = rsqrtf(q), r = 1.0f / q;
        const C2 f{{s, 0.f}, f2_mul(x, F2{s, 0.f})};
        if (w == 8) z8 = c2_mul(z8, f);
        else if (w == 4) z4 = c2_mul(z4, f);
        else z1 = c2_mul(z1, w == 2 ? c2_mul(f, f) : f);
        d1 += (float)w * r;                       // pi gamma n'
        d2 += (float)w * 2.0f * x.h * r * r;      // pi gamma^2 n''
    }
    C2 z = c2_mul(z4, c2_mul(z8, z8));   // (z4 z8^2)^4 z1
    z = c2_mul(z, z);
    z = c2_mul(c2_mul(z, z), z1);
    F2 n1{d1, 0.f};   // the slope divides the step: its tree is summed as a pair
    for (int o = 16; o > 0; o >>= 1) {
        z = c2_mul(z, c2_shfl(z, o));
        n1 = f2_add(n1, f2_shfl(n1, o));
        d2 += __shfl_down_sync(0xffffffffu, d2, o);
    }
    if (lane == 0) { sh.z[warp] = z; sh.n1[warp] = n1; sh.d2[warp] = d2; }
    __syncthreads();
    if (warp != 0) return nil;
    z = lane < NW ? sh.z[lane] : C2{one, nil};
    n1 = lane < NW ? sh.n1[lane] : nil;
    d2 = lane < NW ? sh.d2[lane] : 0.f;
    for (int o = 8; o > 0; o >>= 1) {
        z = c2_mul(z, c2_shfl(z, o));
        n1 = f2_add(n1, f2_shfl(n1, o));
        d2 += __shfl_down_sync(0xffffffffu, d2, o);
    }
    z = c2_mul(z, C2{{mc.cth, mc.ctl}, {-mc.sth, -mc.stl}});
    // the angle left, Theta - Theta_target = -pi (n - target), and the step, as
    // pairs where they scale the result
    const F2 tn = f2_div(z.i, z.r);
    const float t2 = tn.h * tn.h;
    F2 ang = f2_fast(tn.h, tn.l - tn.h * t2 * (1.0f / 3.0f - t2 * (0.2f - t2 * (1.0f / 7.0f))));
    if (!(fabsf(tn.h) <= 0.1f) || !(z.r.h > 0.f)) ang = {atan2f(z.i.h, z.r.h), 0.f};   // not after a search that converged
    const F2 a1 = f2_mul(n1, igp);                                       // pi n'
    const float eps = ang.h * d2 / (2.0f * n1.h * n1.h);                     // -(n - target) n'' / (2 n'^2)
    return f2_mul(f2_div(ang, a1), F2{1.0f, -eps / (1.0f + eps)});           // Halley's 1 / (1 + eps)
}
__device__ void mu_solve_one_cta(const Geom &g, const Band &band, const MuConst &mc, MuSingle &sh, InstState *st,
                                 unsigned *status, double *mu_out, const ClsTab *__restrict__ cls)
{
    constexpr int NW = MU_THREADS / 32;
    static_assert(NW == 16, "the first pass's totals fit one half warp");
    const int h = g.npz / 2, npairs = (h + 1) * (h + 2) / 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool free_e = band.band_kind == 1;
    for (int m = threadIdx.x; m <= h; m += MU_THREADS) {
        const ClsTab c = cls ? cls[m] : class_values(m, g.npz);
        sh.c1[m] = {c.c1h, c.c1l};
        sh.c2[m] = {c.c2h, c.c2l};
        sh.p2[m] = {c.p2h, c.p2l};
    }
    __syncthreads();
    const float t = band.k1[0], tp = band.k2[0], tpp = band.k3[0];   // -2t, -4t', -2t''
    for (int k = threadIdx.x; k < npairs; k += MU_THREADS) {
        int a, b;
        tri_pair(k, h, a, b);
        const float e = free_e ? 0.5f * (sh.p2[a].h + sh.p2[b].h)
                               : t * (sh.c1[a].h + sh.c1[b].h) + tp * sh.c1[a].h * sh.c1[b].h
                                     + tpp * (sh.c2[a].h + sh.c2[b].h);
        sh.ew[k] = make_float2(e, (float)pair_weight(a, b, h));
    }
    __syncthreads();

    const float ig = mc.igh, inv_pi = 0.318309886183790672f, target = mc.target_f;
    float lo = -mc.Bf - 3.0f, hi = mc.Bf + 3.0f;
    {
        const float dc = (hi - lo) / (float)(NW - 1), c = lo + (float)warp * dc;
        float s0 = 0.f, s1 = 0.f;
        int k = lane;
        for (; k + 32 < npairs; k += 64) {
            const float2 x = sh.ew[k], y = sh.ew[k + 32];
            s0 += x.y * (0.5f - atanf((x.x - c) * ig) * inv_pi);
            s1 += y.y * (0.5f - atanf((y.x - c) * ig) * inv_pi);
        }
        if (k < npairs) s0 += sh.ew[k].y * (0.5f - atanf((sh.ew[k].x - c) * ig) * inv_pi);
        s0 += s1;
        for (int o = 16; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        if (lane == 0) sh.cnt[warp] = s0;
        __syncthreads();
        const unsigned hit = __ballot_sync(0xffffffffu, lane < NW && sh.cnt[lane % NW] >= target);
        const int first = hit ? __ffs((int)hit) - 1 : NW;   // the first candidate that reaches the filling
        if (first == 0 || first == NW) {                     // the filling is not bracketed
            if (threadIdx.x == 0) {
                const double mu = 0.5 * ((double)lo + (double)hi);
                atomicCAS(status, (unsigned)DEV_OK, (unsigned)DEV_ENOCONV);
                set_mu(st, mu);
                st->last_step = INFINITY;
                if (mu_out) *mu_out = mu;
            }
            return;
        }
        hi = lo + (float)first * dc;
        lo += (float)(first - 1) * dc;
    }
    float mu = 0.5f * (lo + hi), mu_l = 0.f;   // the estimate; mu_l: what its last rounding dropped
    for (int it = 0; it < MU_NEWTON_MAX; ++it) {
        float n0 = 0.f, n1 = 0.f, n2 = 0.f;   // n(mu), gamma n', gamma^2 n''
        for (int k = threadIdx.x; k < npairs; k += MU_THREADS) {
            const float2 ew = sh.ew[k];
            const float x = (ew.x - mu) * ig, r = __fdividef(1.0f, 1.0f + x * x);
            n0 += ew.y * (0.5f - atanf(x) * inv_pi);
            n1 += ew.y * r;
            n2 += ew.y * 2.0f * x * r * r;
        }
        for (int o = 16; o > 0; o >>= 1) {
            n0 += __shfl_xor_sync(0xffffffffu, n0, o);
            n1 += __shfl_xor_sync(0xffffffffu, n1, o);
            n2 += __shfl_xor_sync(0xffffffffu, n2, o);
        }
        if (lane == 0) {
            sh.red[it & 1][warp][0] = n0;
            sh.red[it & 1][warp][1] = n1;
            sh.red[it & 1][warp][2] = n2;
        }
        __syncthreads();
        n0 = sh.red[it & 1][lane % NW][0];   // every warp adds the 16 sums in the same order
        n1 = sh.red[it & 1][lane % NW][1];
        n2 = sh.red[it & 1][lane % NW][2];
        for (int o = 8; o > 0; o >>= 1) {
            n0 += __shfl_xor_sync(0xffffffffu, n0, o);
            n1 += __shfl_xor_sync(0xffffffffu, n1, o);
            n2 += __shfl_xor_sync(0xffffffffu, n2, o);
        }
        const float F = n0 - target, a1 = n1 * inv_pi * ig, a2 = n2 * inv_pi * ig * ig;   // n - target, n', n''
        if (F < 0.f) lo = mu; else hi = mu;
        const float den = 2.0f * a1 * a1 - F * a2;
        // Halley, or Newton far from the root
        const float dx = a1 > 0.f ? (den > a1 * a1 ? 2.0f * F * a1 / den : F / a1) : INFINITY;
        float nxt = mu - dx;
        mu_l = (mu - nxt) - dx;   // exact near the root (|dx| < |mu|), and below 1e-7 eV else
        if (!(nxt > lo && nxt < hi)) {
            nxt = 0.5f * (lo + hi);
            mu_l = 0.f;
        }
        const bool done = fabsf(nxt - mu) < 1e-6f || hi - lo < 1e-6f;
        mu = nxt;
        if (done) break;
    }

    // the last step, from mu + mu_l
    if (!(fabsf(mu_l) < 1e-6f)) mu_l = 0.f;
    F2 cur = f2_fast(mu, mu_l);
    for (int it = 1;; ++it) {
        const F2 step = mc.narrow ? mu_step_fp64(sh, cur, h, free_e, band.t, band.tp, band.tpp, mc.inv_gam, mc.target)
                                  : mu_step_pairs(g, band, mc, sh, cur);
        if (threadIdx.x == 0) {
            // a step that grows has left the root's neighbourhood: the one before counts
            const bool grows = it > 1 && !(fabsf(step.h) < 2.f * fabsf(sh.step.h));
            const float len = fabsf(grows ? sh.step.h : step.h);
            const F2 m = grows ? cur : f2_add(cur, step);
            const int done = grows || it == MU_STEP_MAX || !(len > mc.step_tol);
            if (done) {
                const double mu_new = (double)m.h + (double)m.l;
                set_mu(st, mu_new);
                st->last_step = (double)len;
                if (mu_out) *mu_out = mu_new;
                // the search ends within 1e-4 eV of the root: a larger last step means it went wrong
                if (!(len <= 1e-4f)) atomicCAS(status, (unsigned)DEV_OK, (unsigned)DEV_ENOCONV);
            }
            sh.mu = m;
            sh.step = step;
            sh.done = done;
        }
        __syncthreads();
        if (sh.done) return;
        cur = sh.mu;
    }
}

// Set-up launch.  CTAs [0, G): multisection pass 0 (mu from the filling);
// CTAs [G, G + GT): the per-axis tables and the energy grid, one entry per
// thread of their first warp; without a filling solve only the table CTAs run
// and the first of them records the given mu.
__global__ void __launch_bounds__(MU_THREADS, 2)
k_setup(Geom g, Band band, AxisTab *axis, float2 *eps32, double *eps64, InstState *st, double *acc,
        unsigned *counter, unsigned *status, double *mu_out, MuConst mc, int G, Band *band_out,
        const ClsTab *__restrict__ cls)
{
    if (band_out && blockIdx.x == 0 && threadIdx.x == 0) *band_out = band;   // the call's band, for later launches
    if ((int)blockIdx.x >= G) {
        const int tb = blockIdx.x - G;
        if (!band.solve_mu && tb == 0 && threadIdx.x == 0) {
            set_mu(st, band.mu);
            st->last_step = 0.0;
            if (mu_out) *mu_out = band.mu;
        }
        const int i = tb * MU_TAB_THREADS + threadIdx.x;
        if (threadIdx.x >= MU_TAB_THREADS) return;
        if (i < g.N) {
            const int k = i - g.N / 2, r = (k < 0 ? -k : k) % g.npz, m = 2 * r > g.npz ? g.npz - r : r;   // its class
            const ClsTab c = cls ? cls[m] : class_values(m, g.npz);
            const double p = (double)k * g.dp;
            AxisTab a;
            a.c1 = c.c1;
            a.c2 = c.c2;
            const double pa = p * band.ff_a;   // ff_a^2 by itself may overflow, and 0 inf is NaN at p = 0
            a.g = exp(-0.125 * (pa * pa));
            a.p2 = p * p;
            a.c1h = c.c1h;
            a.c1l = c.c1l;
            a.c2h = c.c2h;
            a.c2l = c.c2l;
            a.p2h = (float)a.p2;
            a.p2l = (float)(a.p2 - (double)a.p2h);
            a.gf = (float)a.g;
            a.pad = 0.f;
            axis[i] = a;
        }
        if (i < g.n_eps) {
            double e = -g.e_max + ((double)i + 0.5) * g.de;
            if (eps32) {
                float hi = (float)e;
                eps32[i] = make_float2(hi, (float)(e - (double)hi));
            }
            if (eps64) eps64[i] = e;
        }
        return;
    }
    __shared__ union Scratch {
        MuShared sect;
        MuSingle single;
        __device__ Scratch() {}
    } u;
    if (mc.single) {
        mu_solve_one_cta(g, band, mc, u.single, st, status, mu_out, cls);
        return;
    }
    MuShared &sh = u.sect;
    stage_classes(g, sh);
    if (threadIdx.x == 0) {
        sh.br.lo = -mc.B - 3.0;
        sh.br.hi = mc.B + 3.0;
        if (blockIdx.x == 0) {
            acc[0] = sh.br.lo;
            acc[1] = sh.br.hi;
            acc[2] = 0.0;
            *counter = 0;
        }
    }
    sect_pass(g, band, mc, sh, mu_cross(acc, G, 0));
}

// Multisection pass `pass` >= 1.
__global__ void __launch_bounds__(MU_THREADS, 2)
k_mu_sect(Geom g, Band band, double *acc, int pass, MuConst mc)
{
    __shared__ MuShared sh;
    const int G = gridDim.x;
    stage_classes(g, sh);
    __syncthreads();
    // the first chunk of pair energies does not depend on the bracket
    const int h = g.npz / 2, npairs = (h + 1) * (h + 2) / 2;
    stage_pairs(g, band, sh, 0, min(MU_CHUNK, npairs));
    bracket_from(acc, mu_cross(acc, G, pass - 1), mc, pass - 1, sh.br);
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        acc[3 * pass + 0] = sh.br.lo;
        acc[3 * pass + 1] = sh.br.hi;
        acc[3 * pass + 2] = sh.br.flag;
    }
    __syncthreads();
    if (sh.br.flag) return;   // the filling was not bracketed
    sect_pass(g, band, mc, sh, mu_cross(acc, G, pass), true);
}

// Halley step in FP64 from the midpoint of the last bracket; publishes mu.
__global__ void __launch_bounds__(MU_NT_THREADS)
k_mu_halley(Geom g, Band band, const AxisTab *__restrict__ axis, InstState *st, double *acc, unsigned *counter,
            unsigned *status, double *mu_out, MuConst mc)
{
    const int P = mc.passes, G = gridDim.x;
    __shared__ struct { MuBracket br; } sh;
    __shared__ double s_red[MU_NT_THREADS / 32][3];
    double *part = acc + MU_RES;   // [G][4]
    const int h = g.npz / 2, npairs = (h + 1) * (h + 2) / 2, c = g.N / 2;
    // the band energy of this thread's first pair does not depend on mu: its
    // loads and FP64 chain overlap the bracket search
    const int k0 = blockIdx.x + G * threadIdx.x;
    double e0_first = 0.0;
    int w_first = 0;
    if (k0 < npairs) {
        int a, b;
        tri_pair(k0, h, a, b);
        w_first = pair_weight(a, b, h);
        e0_first = band_e0(band, axis[c - a], axis[c - b]);
    }
    bracket_from(acc, mu_cross(acc, G, P - 1), mc, P - 1, sh.br);
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        acc[3 * P + 0] = sh.br.lo;
        acc[3 * P + 1] = sh.br.hi;
        acc[3 * P + 2] = sh.br.flag;
    }
    __syncthreads();
    const double mu = 0.5 * (sh.br.lo + sh.br.hi);
    if (sh.br.flag) {   // the filling was not bracketed
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            atomicCAS(status, (unsigned)DEV_OK, (unsigned)DEV_ENOCONV);
            set_mu(st, mu);
            st->last_step = INFINITY;
            if (mu_out) *mu_out = mu;
        }
        return;
    }
    const double igam = mc.inv_gam, ipi = 0.31830988618379067154;
    double f = 0.0;
    float f1 = 0.f, f2 = 0.f;
    // pairs interleaved over the CTAs first, so every SM's FP64 units share the work
    for (int k = k0; k < npairs; k += G * (int)blockDim.x) {
        double e0 = e0_first;
        int w = w_first;
        if (k != k0) {
            int a, b;
            tri_pair(k, h, a, b);
            w = pair_weight(a, b, h);
            e0 = band_e0(band, axis[c - a], axis[c - b]);
        }
        const double x = (e0 - mu) * igam;                                       // xi / gamma
        f += (double)w * (0.5 - atan(x) * ipi);                                   // occupation
        const float xf = (float)x, r = 1.0f / (1.0f + xf * xf);                    // gamma^2 / (xi^2 + gamma^2)
        f1 += (float)w * r * (float)ipi;                                           // gamma d occ / d mu
        f2 += (float)w * 2.0f * xf * r * r * (float)ipi;                           // gamma^2 d^2 occ / d mu^2
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        f += __shfl_down_sync(0xffffffffu, f, o);
        f1 += __shfl_down_sync(0xffffffffu, f1, o);
        f2 += __shfl_down_sync(0xffffffffu, f2, o);
    }
    if (lane == 0) { s_red[warp][0] = f; s_red[warp][1] = f1; s_red[warp][2] = f2; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double F = 0, F1 = 0, F2 = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { F += s_red[w][0]; F1 += s_red[w][1]; F2 += s_red[w][2]; }
        part[4 * (size_t)blockIdx.x + 0] = F;
        part[4 * (size_t)blockIdx.x + 1] = F1;
        part[4 * (size_t)blockIdx.x + 2] = F2;
    }
    // the last CTA to finish adds the partial sums in a fixed order
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
        if (s_last) *counter = 0;   // no other CTA touches it again in this launch
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double F = 0.0, F1 = 0.0, F2 = 0.0;
    for (int q = threadIdx.x; q < G; q += (int)blockDim.x) {
        F += __ldcg(part + 4 * (size_t)q + 0);
        F1 += __ldcg(part + 4 * (size_t)q + 1);
        F2 += __ldcg(part + 4 * (size_t)q + 2);
    }
    for (int o = 16; o > 0; o >>= 1) {
        F += __shfl_down_sync(0xffffffffu, F, o);
        F1 += __shfl_down_sync(0xffffffffu, F1, o);
        F2 += __shfl_down_sync(0xffffffffu, F2, o);
    }
    __syncthreads();
    if (lane == 0) { s_red[warp][0] = F; s_red[warp][1] = F1; s_red[warp][2] = F2; }
    __syncthreads();
    if (threadIdx.x == 0) {
        F = F1 = F2 = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { F += s_red[w][0]; F1 += s_red[w][1]; F2 += s_red[w][2]; }
        const double d = F - mc.target;                   // n - target
        const double d1 = F1 * igam, d2 = F2 * igam * igam;  // dn/dmu, d2n/dmu2
        const double step = 2.0 * d * d1 / (2.0 * d1 * d1 - d * d2);
        const double mu_new = mu - step;
        set_mu(st, mu_new);
        st->last_step = fabs(step);
        if (mu_out) *mu_out = mu_new;
        // the root lies within the last bracket up to FP32 noise (below
        // 1e-6 eV); a larger step means the multisection went wrong
        if (!(fabs(step) <= 2.0 * (sh.br.hi - sh.br.lo) + 1e-5))
            atomicCAS(status, (unsigned)DEV_OK, (unsigned)DEV_ENOCONV);
    }
}

static MuConst mu_const(const Geom &g, const Band &band, int G)
{
    MuConst mc;
    mc.NC = MU_NCPT * G;
    mc.passes = band.gamma < 0.02 ? 3 : 2;
    mc.single = mu_single(g) ? 1 : 0;
    mc.inv_nc1 = 1.0 / (double)(mc.NC - 1);
    mc.inv_gam = 1.0 / band.gamma;
    mc.target = band.filling * 0.5 * (double)g.npz * (double)g.npz;
    mc.target32 = llrint(mc.target * (double)MU_SECT_SCALE);
    mc.target_f = (float)mc.target;
    auto pair = [](double v, float &hi, float &lo) {
        hi = (float)v;
        lo = (float)(v - (double)hi);
    };
    pair(mc.inv_gam, mc.igh, mc.igl);
    // e^{i pi u}, u = npz^2 / 2 - target
    const double u = fmod(0.5 * (double)g.npz * (double)g.npz - mc.target, 2.0);
    pair(cos(M_PI * u), mc.cth, mc.ctl);
    pair(sin(M_PI * u), mc.sth, mc.stl);
    mc.B = (band.band_kind == 1) ? 9.869604401089358 : 4.0 * (fabs(band.t) + fabs(band.tp) + fabs(band.tpp));
    mc.Bf = (float)mc.B;
    mc.step_tol = (float)cbrt(1e-13 * band.gamma * band.gamma);
    mc.narrow = band.gamma < MU_PAIR_GAMMA;
    return mc;
}

cudaError_t launch_twiddles(int len, float2 *tw32, double2 *tw64, cudaStream_t s)
{
    k_twiddles<<<(twiddle_entries() + 255) / 256, 256, 0, s>>>(len, tw32, tw64);
    return cudaGetLastError();
}

// Tables plus the first chemical-potential launch (multisection pass 0, or
// the given mu).
// band_out (device, or null): receives the call's band for later launches.
// cls: the zone's class table (k_classes), or null: formed in the launch.
cudaError_t launch_setup_band(const Geom &g, const Band &band, AxisTab *axis, float2 *eps32, double *eps64,
                              InstState *st, double *acc, unsigned *bar, unsigned *status, double *mu_out, int G,
                              Band *band_out, const ClsTab *cls, cudaStream_t s)
{
    const int ntab = g.N > g.n_eps ? g.N : g.n_eps;
    const int GT = (ntab + MU_TAB_THREADS - 1) / MU_TAB_THREADS;
    const int Gs = band.solve_mu ? (mu_single(g) ? 1 : G) : 0;
    k_setup<<<Gs + GT, MU_THREADS, 0, s>>>(g, band, axis, eps32, eps64, st, acc, bar, status, mu_out,
                                           mu_const(g, band, G), Gs, band_out, cls);
    return cudaGetLastError();
}
cudaError_t launch_setup(const Geom &g, const Band &band, AxisTab *axis, float2 *eps32, double *eps64,
                         InstState *st, double *acc, unsigned *bar, unsigned *status, double *mu_out, int G,
                         const ClsTab *cls, cudaStream_t s)
{
    return launch_setup_band(g, band, axis, eps32, eps64, st, acc, bar, status, mu_out, G, nullptr, cls, s);
}

// Whether the chemical potential is solved inside the set-up launch.
bool mu_solve_in_setup(const Geom &g) { return mu_single(g); }

// The remaining chemical-potential launches (none for a given mu).
cudaError_t launch_solve_mu(const Geom &g, const Band &band, const AxisTab *axis, InstState *st, double *acc,
                            unsigned *bar, unsigned *status, double *mu_out, int G, cudaStream_t s)
{
    if (!band.solve_mu || mu_single(g)) return cudaSuccess;   // solved in the set-up launch
    const MuConst mc = mu_const(g, band, G);
    for (int pass = 1; pass < mc.passes; ++pass) k_mu_sect<<<G, MU_THREADS, 0, s>>>(g, band, acc, pass, mc);
    // one warp per CTA when every CTA has at most 32 pairs (the FP64 chains
    // then run side by side and the reductions are short)
    const int h = g.npz / 2, npairs = (h + 1) * (h + 2) / 2;
    const int T = npairs <= 32 * G ? 32 : MU_NT_THREADS;
    k_mu_halley<<<G, T, 0, s>>>(g, band, axis, st, acc, bar, status, mu_out, mc);
    return cudaGetLastError();
}

}  // namespace lh
