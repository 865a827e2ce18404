// Statistical equilibrium: FP64, state reduction, G lanes per point.
//
// Rates i -> j per point (s^-1):
//   radiative, preconditioned by the diagonal approximate Lambda operator
//   (Rybicki & Hummer 1991), J_eff = Jbar - Lambda* S_old:
//       u -> l : max(A_ul (1 - Lambda*) + B_ul J_eff, 0)
//       l -> u : max(B_lu J_eff, 0)
//   collisional: C_ul = n_coll K_ul, C_lu = C_ul (g_u/g_l) exp(-(E_u - E_l)/kT).
// The steady state sum_j n_j R_ji = n_i sum_j R_ij, normalised to n_spec, is
// found by state reduction (Grassmann, Taksar & Heyman 1985): eliminate the
// highest level first, folding the paths through it into the remaining rates,
// R_ij += R_in R_nj / S_n with S_n = sum_{j<n} R_nj; then n_0 = 1,
// n_k = sum_{i<k} n_i R_ik / S_k and normalise.  Only non-negative numbers are
// added, so populations many decades below the ground level keep full
// relative accuracy.  All reductions run in a fixed lane order, so the result
// is bitwise reproducible.
//
// What bounds it: the FP64 pipe, 16 cycles per warp instruction and SM whatever
// the number of active lanes (two lanes per cycle).  The elimination of 41
// levels is 22,140 multiply-adds, 692 full warp instructions; with one warp per
// point another 1,440 went into work that fills few lanes: the sum and the
// reciprocal of every pivot, rates assembled from all L^2 entries, the back
// substitution.  So a warp takes 32 / G points and every such instruction
// serves all of them, and the rates are filled in from the lists of lines and
// collisions.  100k points: 41 levels 11.8 -> 7.5 ms, 21 levels 3.34 -> 1.47,
// 11 levels 1.49 -> 0.44, 5 levels 0.76 -> 0.17.
#include <algorithm>
#include <cstring>

#include "mgt_common.cuh"

namespace mgt {

namespace {

struct SEArgs {
    int64_t N;
    int L, M, Mpad, K;
    const double *pops_old;   // [N][L]
    const double *J, *Lst;    // [N][M]
    const double *T, *ncoll, *nspec;
    const double *line_tab;   // [8][Mpad]: nu, A, Bul, Blu, ...
    const int32_t *line_ul;   // [2][Mpad]
    const double *level_tab;  // [2][L]: E, g
    const double *Kul;        // [K]
    const int32_t *coll_ul;   // [2][K]
    double *pops_out;         // [N][L] (may be pops_old: each point's row is read before it is written)
    double *pops_prev;        // [N][L] copy of pops_old
    int wpb;                  // warps of a CTA that take points (what its shared memory holds)
    int lanes;                // lanes per point
};

constexpr int kMaxWarpsPerBlock = 4;
constexpr size_t kSEMaxSmem = 227 * 1024;
constexpr size_t kSEBatchStatic = (sizeof(SEArgs) + sizeof(int64_t) + 31) / 16 * 16;   // k_se_batch's static arrays

// A point's working memory in doubles: the rates, the reciprocals 1/bz (later
// the unnormalised populations), and the lines' rates (later the pivots'
// reciprocals).
__host__ __device__ inline int se_point_doubles(int L, int M) { return L * L + L + (L > 2 * M ? L : 2 * M); }

constexpr int kLevelsPerLane = 4;                 // G lanes hold up to 4 G levels
static_assert(kMaxLevels <= 16 * kLevelsPerLane, "levels per lane");

// Lanes per point.  Many points: the fewest lanes, so that an FP64 instruction
// serves as many points as possible, with two warps per scheduler in an SM's
// shared memory.  100k points: 11 levels 4 lanes 0.44 ms, 8 lanes 0.60; 21
// levels 8 lanes 1.49, 16 lanes 2.08; 28 levels 2.90, 3.34; 32 levels (8 lanes:
// one warp per scheduler) 5.89, 16 lanes 4.25; 41 levels 16 lanes 7.51, 32 lanes
// 9.34; 48 levels 15.9, 13.2.  Few points: more lanes while they still get a
// scheduler to themselves, or half of one above 16 levels (a point's chain is
// what lasts then): 1,200 points of 11 levels 16 lanes 18.5 us, 4 lanes 36.4; 21
// levels 32 lanes 41, 8 lanes 63; 3,000 points of 21 levels 16 lanes 82, 8 lanes
// 80.  Results do not depend on it.
inline int se_lanes(int L, int M, int64_t points, int sms)
{
    constexpr size_t sm_smem = 228 * 1024, cta_smem = 1024;    // an SM's, and what a CTA takes of it by itself
    auto few_resident = [&](int g) {
        return 2 * (kMaxWarpsPerBlock * sizeof(double) * (32 / g) * (size_t)se_point_doubles(L, M) + cta_smem) > sm_smem;
    };
    int g = 4;
    while (g < 32 && (L > kLevelsPerLane * g || few_resident(g))) g *= 2;
    while (g < 32 && points * 2 * g <= (int64_t)sms * 32 * (L > 16 ? 8 : 4)) g *= 2;
    return g;
}

// The device's SMs (0 where there is none: host checks).
int se_sms()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return sms;
}

// Sum of v[0 .. n-1] (n <= 64) over the point's lanes, in the order of a warp
// that holds v[l] + v[l + 32] in lane l and adds lanes 16, 8, 4, 2 and 1 apart,
// whatever G is: accelerated iterations amplify a changed rounding.  Additions
// of what lies past n are skipped.  Every lane ends with the sum.
template <int G> __device__ __forceinline__ double point_sum(const double *v, int n, int t)
{
    double s[32 / G];
#pragma unroll
    for (int q = 0; q < 32 / G; ++q) {
        const int l = t + q * G;
        s[q] = l < n ? v[l] : 0.0;
        if (n > 32 + q * G) s[q] += l + 32 < n ? v[l + 32] : 0.0;
    }
#pragma unroll
    for (int o = 16; o >= G; o >>= 1)
#pragma unroll
        for (int q = 0; q < o / G; ++q)
            if (n > o + q * G) s[q] += s[q + o / G];
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1)
        if (n > o) s[0] += __shfl_xor_sync(0xffffffffu, s[0], o, G);
    return __shfl_sync(0xffffffffu, s[0], 0, G);
}

// v > 0 for a sum of non-negative numbers (false for NaN), by its bits: a
// comparison on the FP64 pipe costs as much as a multiply-add.
__device__ __forceinline__ bool positive_bits(double v)
{
    const long long b = __double_as_longlong(v);
    return b > 0 && b <= 0x7ff0000000000000ll;
}

// Point p, solved by the G lanes t = 0 .. G - 1 of its group in their
// shared-memory slice sm; `write` false: a group past the last point, which
// repeats that point (same warp) and writes nothing.
template <int G> __device__ __forceinline__ void se_point(const SEArgs &a, int64_t p, double *sm, int t, bool write)
{
    const int L = a.L, LL = L * L;
    double *R = sm;                       // R[i*L + j]: rate i -> j; diagonal: bz_i = g_i exp(-(E_i - E_0)/kT)
    double *xx = R + LL;                  // [L] 1/bz, later the unnormalised populations
    double *Sn = xx + L;                  // [L] reciprocals of the pivots
    double *rdown = Sn, *rup = Sn + a.M;  // [M] each, before the pivots: radiative u -> l, l -> u rate per line

    const double *po = a.pops_old + p * L;
    if (write)
        for (int i = t; i < L; i += G) a.pops_prev[p * L + i] = po[i];
    const double Tp = a.T[p], nc = a.ncoll[p];
    // per-line preconditioned radiative rates
    for (int k = t; k < a.M; k += G) {
        const int u = a.line_ul[k], l = a.line_ul[a.Mpad + k];
        const double A = a.line_tab[a.Mpad + k], Bul = a.line_tab[2 * a.Mpad + k], Blu = a.line_tab[3 * a.Mpad + k];
        const double x_l = po[l] * Blu, x_u = po[u] * Bul;
        double net = x_l - x_u;
        const double fl = 1e-30 * (x_l + x_u);
        if (net < fl) net = fl;
        const double S_old = net > 0.0 ? po[u] * A / net : 0.0;
        const double Js = a.J[p * a.M + k], Ls = a.Lst[p * a.M + k];
        const double Jeff = Js - Ls * S_old;
        rdown[k] = fmax(A * (1.0 - Ls) + Bul * Jeff, 0.0);
        rup[k] = fmax(Blu * Jeff, 0.0);
    }
    for (int e = t; e < LL; e += G) R[e] = 0.0;
    __syncwarp();
    for (int k = t; k < a.M; k += G) R[a.line_ul[a.Mpad + k] * L + a.line_ul[k]] = rup[k];
    const double *E = a.level_tab, *g = a.level_tab + L;
    const double ikT = 1.0 / (kKB * Tp);
    // one exponential per level instead of one per collisional pair: the
    // upward rate C_lu = C_ul (g_u/g_l) exp(-(E_u - E_l)/kT) = C_ul bz_u / bz_l,
    // formed with 1/bz_l from one division per level (FP64 division is a long
    // sequence, and there are L^2/2 upward pairs)
    for (int i = t; i < L; i += G) {
        const double b = g[i] * exp(-(E[i] - E[0]) * ikT);
        R[i * L + i] = b;
        xx[i] = b > 1e-290 ? 1.0 / b : 0.0;
    }
    __syncwarp();
    for (int k = t; k < a.K; k += G) {
        const int u = a.coll_ul[k], l = a.coll_ul[a.K + k];
        const double Cul = __dmul_rn(nc, a.Kul[k]);
        const double bu = R[u * L + u], ru = xx[u], rl = xx[l];
        double &up = R[l * L + u];
        R[u * L + l] = Cul;
        // (1/bz is zero where the factor is near the bottom of the FP64 range:
        // then the pair's own exponential)
        if (__double2hiint(rl) != 0 && __double2hiint(ru) != 0)
            up = __fma_rn(__dmul_rn(Cul, bu), rl, up);
        else
            up = __fma_rn(Cul * g[u] / g[l], exp(-(E[u] - E[l]) * ikT), up);
    }
    __syncwarp();
    for (int k = t; k < a.M; k += G) {
        double &down = R[a.line_ul[k] * L + a.line_ul[a.Mpad + k]];
        down = __dadd_rn(rdown[k], down);
    }
    __syncwarp();
    // state reduction, highest level first
    for (int n = L - 1; n >= 1; --n) {
        double s = point_sum<G>(R + n * L, n, t);
        s = positive_bits(s) ? s : 1e-300;
        const double rs = 1.0 / s;
        if (t == 0) Sn[n] = rs;
        for (int j = t; j < n; j += G) R[n * L + j] *= rs;
        __syncwarp();
        // rows i, columns j < n: entry e = i n + j, the stride advances (i, j)
        // by (di, dj); with few warps per scheduler two entries at a time,
        // loads before stores, so that their latencies overlap
        constexpr int kUpdate = G >= 16 ? 2 : 1;
        const int di = G / n, dj = G - di * n;
        int i = t / n, j = t - i * n;
        for (int e = t; e < n * n; e += kUpdate * G) {
            double *at[kUpdate];
            double r[kUpdate], x[kUpdate], y[kUpdate];
#pragma unroll
            for (int q = 0; q < kUpdate; ++q) {
                const bool in = e + q * G < n * n;
                at[q] = R + (in ? i * L + j : 0);
                r[q] = *at[q];
                x[q] = R[in ? i * L + n : 0];
                y[q] = R[n * L + (in ? j : 0)];
                i += di;
                j += dj;
                if (j >= n) {
                    j -= n;
                    ++i;
                }
            }
#pragma unroll
            for (int q = 0; q < kUpdate; ++q) r[q] += x[q] * y[q];
#pragma unroll
            for (int q = 0; q < kUpdate; ++q)
                if (e + q * G < n * n) *at[q] = r[q];
        }
        __syncwarp();
    }
    // back substitution n_k = sum_{i<k} n_i R_ik / S_k, column by column: lane
    // t keeps the running sums of levels t, t + G, ..., and once n_{k-1} is
    // known every lane adds its term to the levels above it (one FP64
    // multiply-add per lane and level instead of a sum over lanes per level)
    double acc[kLevelsPerLane];
#pragma unroll
    for (int q = 0; q < kLevelsPerLane; ++q) acc[q] = 0.0;
    if (t == 0) xx[0] = 1.0;
    double xprev = 1.0;                   // n_0
    for (int k = 1; k < L; ++k) {
        const int i = k - 1;              // n_i is known: add n_i R_ij to every level j > i
        double ak = 0.0;
#pragma unroll
        for (int q = 0; q < kLevelsPerLane; ++q) {
            const int j = t + q * G;
            if (j > i && j < L) acc[q] += xprev * R[i * L + j];
            if (q == k / G) ak = acc[q];
        }
        // n_k = acc / S_k from the lane that holds level k
        double nk = 0.0;
        if (k % G == t) {
            nk = ak * Sn[k];
            xx[k] = nk;
        }
        xprev = __shfl_sync(0xffffffffu, nk, k % G, G);
    }
    __syncwarp();
    const double f = a.nspec[p] / point_sum<G>(xx, L, t);
    if (write)
        for (int i = t; i < L; i += G) a.pops_out[p * L + i] = xx[i] * f;
}

// The calling warp's points of one model (32 / G of them, from first_warp on).
template <int G> __device__ __forceinline__ void se_warp(const SEArgs &a, int64_t warp, double *sm)
{
    const int lane = threadIdx.x & 31, grp = lane / G;
    const int64_t p = warp * (32 / G) + grp;
    if (p - grp >= a.N) return;           // whole warp
    se_point<G>(a, min(p, a.N - 1), sm + grp * se_point_doubles(a.L, a.M), lane - grp * G, p < a.N);
}

__device__ __forceinline__ void se_block(const SEArgs &a, int64_t block, double *sm)
{
    const int w = threadIdx.x >> 5;
    if (w >= a.wpb) return;               // whole warp
    const int G = a.lanes;
    const int64_t warp = block * a.wpb + w;
    sm += (int64_t)w * (32 / G) * se_point_doubles(a.L, a.M);
    if (G == 32)
        se_warp<32>(a, warp, sm);
    else if (G == 16)
        se_warp<16>(a, warp, sm);
    else if (G == 8)
        se_warp<8>(a, warp, sm);
    else
        se_warp<4>(a, warp, sm);
}

__global__ void __launch_bounds__(32 * kMaxWarpsPerBlock) k_se(SEArgs a)
{
    extern __shared__ __align__(16) double sm[];
    se_block(a, blockIdx.x, sm);
}

// Many models in one launch, one model per CTA: blk_end[i] is one past the last
// CTA of model i.
__global__ void __launch_bounds__(32 * kMaxWarpsPerBlock) k_se_batch(const SEArgs *__restrict__ args,
                                                                     const int64_t *__restrict__ blk_end, int n_models)
{
    extern __shared__ __align__(16) double sm[];
    __shared__ SEArgs sa;
    __shared__ int64_t s_first;
    if (threadIdx.x == 0) {
        const int64_t b = blockIdx.x;
        int lo = 0, hi = n_models - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (blk_end[mid] > b) hi = mid; else lo = mid + 1;
        }
        sa = args[lo];
        s_first = lo > 0 ? blk_end[lo - 1] : 0;
    }
    __syncthreads();
    se_block(sa, (int64_t)blockIdx.x - s_first, sm);
}

// Arguments of model m in a launch over `points` points.
SEArgs fill_se_args(const mgt_model *m, int64_t points)
{
    SEArgs a{};
    a.N = m->N;
    a.L = m->L;
    a.M = m->M;
    a.Mpad = m->Mpad;
    a.K = m->K;
    a.pops_old = m->d_pops;
    a.J = m->d_J;
    a.Lst = m->d_Lst;
    a.T = m->d_temp;
    a.ncoll = m->d_ncoll;
    a.nspec = m->d_nspec;
    a.line_tab = m->d_line_tab;
    a.line_ul = m->d_line_ul;
    a.level_tab = m->d_level_tab;
    a.Kul = m->d_coll_tab;
    a.coll_ul = m->d_coll_ul;
    a.pops_out = m->d_pops;
    a.pops_prev = m->d_pops_prev;
    a.lanes = se_lanes(m->L, m->M, points, se_sms());
    return a;
}

// Warps per CTA, CTAs and a CTA's dynamic shared memory (at most `most`); false
// if no warp's points fit.
bool se_layout(const mgt_model *m, int lanes, size_t most, int *wpb, int64_t *blocks, size_t *smem)
{
    const int points = 32 / lanes;
    const size_t per_warp = sizeof(double) * points * (size_t)se_point_doubles(m->L, m->M);
    *wpb = (int)std::min<size_t>(kMaxWarpsPerBlock, most / per_warp);
    if (*wpb < 1) return false;
    *blocks = ceil_div(m->N, (int64_t)*wpb * points);
    *smem = per_warp * *wpb;
    return true;
}

}  // namespace

mgt_status launch_stat_eq(mgt_model *m, cudaStream_t s)
{
    SEArgs a = fill_se_args(m, m->N);
    int64_t blocks = 0;
    size_t smem = 0;
    if (!se_layout(m, a.lanes, kSEMaxSmem, &a.wpb, &blocks, &smem))
        return set_error(MGT_ERR_ARG, "statistical equilibrium: too many levels/lines for shared memory");
    MGT_TRY_STATUS(raise_smem_limit((const void *)k_se, smem));
    {
        MGT_KTIMER("k_se", s);
        k_se<<<(unsigned)blocks, 32 * a.wpb, smem, s>>>(a);
    }
    MGT_LAUNCH_CHECK("k_se");
    return MGT_OK;
}

size_t se_args_bytes() { return sizeof(SEArgs); }

mgt_status se_batch_args(const mgt_model *m, int64_t points, void *args, int64_t *blocks, size_t *smem)
{
    SEArgs a = fill_se_args(m, points);
    // the batch's documented limit
    if (4 * sizeof(double) * ((size_t)m->L * m->L + 3 * m->L + 2 * m->Mpad) > kSEMaxSmem)
        return set_error(MGT_ERR_ARG, "batched statistical equilibrium: too many levels");
    // (k_se_batch also holds a model's arguments in shared memory)
    if (!se_layout(m, a.lanes, kSEMaxSmem - kSEBatchStatic, &a.wpb, blocks, smem))
        return set_error(MGT_ERR_ARG, "batched statistical equilibrium: too many levels");
    std::memcpy(args, &a, sizeof a);
    return MGT_OK;
}

mgt_status se_batch_prepare(size_t smem)
{
    MGT_TRY_STATUS(raise_smem_limit((const void *)k_se_batch, smem));
    return MGT_OK;
}

mgt_status se_batch_launch(const void *d_args, const int64_t *d_blk_end, int n_models, int64_t n_blocks, size_t smem,
                           cudaStream_t s)
{
    k_se_batch<<<(unsigned)n_blocks, 32 * kMaxWarpsPerBlock, smem, s>>>(static_cast<const SEArgs *>(d_args), d_blk_end,
                                                                       n_models);
    MGT_LAUNCH_CHECK("k_se_batch");
    return MGT_OK;
}

}  // namespace mgt
