// Per-point kernels: line widths, LTE populations, line opacity / source
// function, and the ray walk through the neighbour graph.
#include <cub/cub.cuh>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

#include "mgt_common.cuh"

namespace mgt {

// ---------------------------------------------------------------------------
// Relative line width w = dnu/nu = sqrt(2 k T / m + vturb^2) / c (Sec. 4.3,
// eq. line width); one value per point serves every line of the species.
// ---------------------------------------------------------------------------
__global__ void k_widths(int64_t N, const double *__restrict__ T, const double *__restrict__ vt2,
                         double two_k_over_m, double inv_c, double *__restrict__ w64,
                         float2 *__restrict__ w32)
{
    int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= N) return;
    double w = sqrt(two_k_over_m * T[p] + vt2[p]) * inv_c;
    w64[p] = w;
    w32[p] = make_float2((float)w, (float)(1.0 / w));
}

mgt_status launch_widths(mgt_model *m, cudaStream_t s)
{
    k_widths<<<ceil_div(m->N, 256), 256, 0, s>>>(m->N, m->d_temp, m->d_vturb2, 2.0 * kKB / m->mol_mass,
                                                 1.0 / kC, m->d_w64, m->d_w32);
    MGT_LAUNCH_CHECK("k_widths");
    return MGT_OK;
}

// ---------------------------------------------------------------------------
// Walk tables built on the device at model set-up (from the uploaded
// positions, velocities, neighbour lists and boundary mask):
//  * positions times pos_scale and v/c, each split into float hi + lo;
//  * the FP64 position of every neighbour entry;
//  * the packed neighbour rows (see kWalkRow in mgt_common.cuh);
//  * the Morton (Z-curve) visiting order of the points: 21 bits per axis of
//    the point's place in the bounding box, sorted with ties to the lower
//    index.
// The arithmetic is the host definition's (IEEE operations, no contraction),
// so the tables do not depend on where they are built.
// ---------------------------------------------------------------------------
__global__ void k_split_hl(int64_t N, const double *__restrict__ pos, const double *__restrict__ vel, double scale,
                           double inv_c, float *__restrict__ pos_hl, float *__restrict__ vel_hl)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= 3 * N) return;
    const int64_t i = t / 3;
    const int c = (int)(t - 3 * i);
    const double xs = __dmul_rn(pos[t], scale);
    const float hi = __double2float_rn(xs);
    pos_hl[6 * i + c] = hi;
    pos_hl[6 * i + 3 + c] = __double2float_rn(__dsub_rn(xs, (double)hi));
    const double vb = __dmul_rn(vel[t], inv_c);
    const float vh = __double2float_rn(vb);
    vel_hl[6 * i + c] = vh;
    vel_hl[6 * i + 3 + c] = __double2float_rn(__dsub_rn(vb, (double)vh));
}

__global__ void k_nbr_pos(int64_t nnz, const int32_t *__restrict__ nb, const double *__restrict__ pos,
                          double *__restrict__ nb_pos)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= 3 * nnz) return;
    const int64_t k = t / 3;
    nb_pos[t] = pos[3 * (int64_t)nb[k] + (t - 3 * k)];
}

__device__ __forceinline__ void put_entry(float4 *ent, int64_t e, const float *phl, int64_t mpt, uint32_t word,
                                          int32_t noff)
{
    const float nan = __int_as_float(0x7fffffff);  // empty: no comparison of the walk's filter holds
    float v[6] = {nan, nan, nan, nan, nan, nan};
    if (mpt >= 0)
        for (int c = 0; c < 6; ++c) v[c] = phl[6 * mpt + c];
    ent[2 * e] = make_float4(v[0], v[1], v[2], __uint_as_float(word));
    ent[2 * e + 1] = make_float4(v[3], v[4], v[5], __int_as_float(noff));
}

// One thread per point (rows of ~15 entries).  A row is padded with empty
// entries to whole chunks of kWalkRow entries (one 128-byte line), and every
// entry of a row's last chunk carries the last-of-row flag.
__global__ void k_pack_rows(int64_t N, const int32_t *__restrict__ off, const int32_t *__restrict__ nb,
                            const uint8_t *__restrict__ bnd, const float *__restrict__ phl,
                            const int32_t *__restrict__ row, float4 *__restrict__ ent)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int32_t k0 = off[i], deg = off[i + 1] - k0;
    const int64_t e0 = (int64_t)row[i] * kWalkRow;
    const int32_t n = max(1, (deg + kWalkRow - 1) / kWalkRow) * kWalkRow;
    for (int32_t k = 0; k < n; ++k) {
        const uint32_t last = k >= n - kWalkRow ? kEntLast : 0u;
        if (k >= deg) {
            put_entry(ent, e0 + k, phl, -1, kEntEmpty | last, 0);
            continue;
        }
        const int32_t mpt = nb[k0 + k];
        put_entry(ent, e0 + k, phl, mpt, (uint32_t)mpt | last | (bnd[mpt] ? kEntBnd : 0u), row[mpt]);
    }
}

__device__ __forceinline__ uint64_t morton_spread(uint64_t v)
{
    v &= 0x1fffff;
    v = (v | v << 32) & 0x1f00000000ffffULL;
    v = (v | v << 16) & 0x1f0000ff0000ffULL;
    v = (v | v << 8) & 0x100f00f00f00f00fULL;
    v = (v | v << 4) & 0x10c30c30c30c30c3ULL;
    v = (v | v << 2) & 0x1249249249249249ULL;
    return v;
}

__global__ void k_morton_keys(int64_t N, const double *__restrict__ pos, double lo0, double lo1, double lo2,
                              double sp0, double sp1, double sp2, uint64_t *__restrict__ key,
                              int32_t *__restrict__ idx)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double lo[3] = {lo0, lo1, lo2}, sp[3] = {sp0, sp1, sp2};
    uint64_t k = 0;
    for (int d = 0; d < 3; ++d) {
        const double x = __dmul_rn(__ddiv_rn(__dsub_rn(pos[3 * i + d], lo[d]), sp[d]), 2097151.0);
        const uint64_t q = (uint64_t)fmin(2097151.0, fmax(0.0, x));
        k |= morton_spread(q) << d;
    }
    key[i] = k;
    idx[i] = (int32_t)i;
}

// Longest graph edge at each point, over the edges of its own neighbour list
// and those that name it (so that every step of a walk, from a point to one of
// its neighbours, is no longer than dxmax at either end): FP64 distance in
// length units, rounded up to FP32 with a margin over the walk's own FP32 step
// lengths.  Non-negative floats order like their bit patterns.
__global__ void k_edge_max(int64_t N, const int32_t *__restrict__ off, const int32_t *__restrict__ nbrs,
                           const double *__restrict__ pos, double inv_Lunit, float *__restrict__ dxmax)
{
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= N) return;
    int *dm = reinterpret_cast<int *>(dxmax);
    float best = 0.0f;
    for (int32_t k = off[p]; k < off[p + 1]; ++k) {
        const int64_t q = nbrs[k];
        const double dx = pos[3 * q] - pos[3 * p], dy = pos[3 * q + 1] - pos[3 * p + 1],
                     dz = pos[3 * q + 2] - pos[3 * p + 2];
        const float d = __double2float_ru(sqrt(dx * dx + dy * dy + dz * dz) * inv_Lunit * (1.0 + 1e-5));
        best = fmaxf(best, d);
        atomicMax(dm + q, __float_as_int(d));
    }
    atomicMax(dm + p, __float_as_int(best));
}

mgt_status build_walk_tables(mgt_model *m, const double lo[3], const double hi[3], cudaStream_t s)
{
    const int64_t N = m->N;
    MGT_CUDA(cudaMemsetAsync(m->d_dxmax, 0, sizeof(float) * N, s));
    k_edge_max<<<ceil_div(N, 256), 256, 0, s>>>(N, m->d_nbr_off, m->d_nbrs, m->d_pos, 1.0 / m->L_unit, m->d_dxmax);
    MGT_LAUNCH_CHECK("k_edge_max");
    k_split_hl<<<ceil_div(3 * N, 256), 256, 0, s>>>(N, m->d_pos, m->d_vel, m->pos_scale, 1.0 / kC, m->d_pos_hl,
                                                    m->d_vel_hl);
    MGT_LAUNCH_CHECK("k_split_hl");
    if (m->nnz > 0) {
        k_nbr_pos<<<ceil_div(3 * m->nnz, 256), 256, 0, s>>>(m->nnz, m->d_nbrs, m->d_pos, m->d_nbr_pos);
        MGT_LAUNCH_CHECK("k_nbr_pos");
    }
    k_pack_rows<<<ceil_div(N, 128), 128, 0, s>>>(N, m->d_nbr_off, m->d_nbrs, m->d_bnd, m->d_pos_hl, m->d_ent_row,
                                                 m->d_ent);
    MGT_LAUNCH_CHECK("k_pack_rows");
    // Morton order: keys, then a stable radix sort of (key, index)
    uint64_t *keys = nullptr;
    int32_t *idx = nullptr;
    void *tmp = nullptr;
    size_t tmp_bytes = 0;
    mgt_status st = MGT_OK;
    auto fail = [&](cudaError_t e, const char *what) {
        if (st == MGT_OK) st = cuda_status(e, what);
    };
    cudaError_t e = cudaMallocAsync(&keys, sizeof(uint64_t) * 2 * N, s);
    if (e != cudaSuccess) fail(e, "cudaMallocAsync");
    if (st == MGT_OK && (e = cudaMallocAsync(&idx, sizeof(int32_t) * N, s)) != cudaSuccess) fail(e, "cudaMallocAsync");
    double sp[3];
    for (int d = 0; d < 3; ++d) sp[d] = hi[d] > lo[d] ? hi[d] - lo[d] : 1.0;
    if (st == MGT_OK) {
        k_morton_keys<<<ceil_div(N, 256), 256, 0, s>>>(N, m->d_pos, lo[0], lo[1], lo[2], sp[0], sp[1], sp[2], keys,
                                                      idx);
        e = cudaGetLastError();
        if (e != cudaSuccess) fail(e, "k_morton_keys");
        else note_launch();
    }
    if (st == MGT_OK &&
        (e = cub::DeviceRadixSort::SortPairs(nullptr, tmp_bytes, keys, keys + N, idx, m->d_order, (int)N, 0, 64,
                                             s)) != cudaSuccess)
        fail(e, "cub::DeviceRadixSort::SortPairs");
    if (st == MGT_OK && (e = cudaMallocAsync(&tmp, tmp_bytes, s)) != cudaSuccess) fail(e, "cudaMallocAsync");
    if (st == MGT_OK &&
        (e = cub::DeviceRadixSort::SortPairs(tmp, tmp_bytes, keys, keys + N, idx, m->d_order, (int)N, 0, 64, s)) !=
            cudaSuccess)
        fail(e, "cub::DeviceRadixSort::SortPairs");
    if (tmp) cudaFreeAsync(tmp, s);
    if (idx) cudaFreeAsync(idx, s);
    if (keys) cudaFreeAsync(keys, s);
    return st;
}

// ---------------------------------------------------------------------------
// LTE: n_i = n_spec g_i exp(-(E_i - E_0)/kT) / sum_j g_j exp(-(E_j - E_0)/kT).
// ---------------------------------------------------------------------------
// G lanes per point, lanes over levels, the exponentials in shared memory; the
// partition function is summed in level order by every lane (the same bits for
// any G).  Few points: eight lanes, as one lane's chain of L exponentials is
// what lasts (2,000 points, host time per call included: 41 levels 34 us with
// two lanes, 23 with eight; 11 levels 24 with one, 18.6).  Above eight warps of
// eight lanes per SM the FP64 pipe's instructions count, and fewer lanes serve
// more points with each: 100k points of 3, 11 and 16 levels 34, 69 and 89 us with
// one lane, 48, 82 and 91 with two, 72, 135 and 112 with eight; 41 levels 195 with
// two, 288 with eight.  Each lane computing its levels' exponentials twice,
// one lane per point, took 45, 112, 152 and 364 us there and 75 us for 2,000
// points of 41 levels.
constexpr int kLteThreads = 128;

template <int G>
__global__ void __launch_bounds__(kLteThreads) k_lte(int64_t N, int L, const double *__restrict__ T,
                                                     const double *__restrict__ nspec,
                                                     const double *__restrict__ level_tab, double *__restrict__ pops)
{
    extern __shared__ double lte_ex[];               // [kLteThreads / G][L, made odd]
    const int grp = threadIdx.x / G, t = threadIdx.x - grp * G;
    const int64_t p = blockIdx.x * (int64_t)(kLteThreads / G) + grp;
    const double *E = level_tab, *g = level_tab + L;
    double *ex = lte_ex + grp * (L | 1);
    if (p < N) {
        const double beta = 1.0 / (kKB * T[p]);
        for (int i = t; i < L; i += G) ex[i] = exp(-(E[i] - E[0]) * beta);
    }
    __syncwarp();
    if (p >= N) return;
    double Z = 0.0;
    for (int i = 0; i < L; ++i) Z = __fma_rn(g[i], ex[i], Z);
    const double f = nspec[p] / Z;
    for (int i = t; i < L; i += G) pops[p * L + i] = __dmul_rn(__dmul_rn(f, g[i]), ex[i]);
}

mgt_status launch_lte(mgt_model *m, cudaStream_t s)
{
    int sms = 0;
    MGT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, m->device));
    const auto run = [&](auto kernel, int lanes) {
        const int points = kLteThreads / lanes;
        kernel<<<ceil_div(m->N, (int64_t)points), kLteThreads, sizeof(double) * points * (m->L | 1), s>>>(
            m->N, m->L, m->d_temp, m->d_nspec, m->d_level_tab, m->d_pops);
    };
    if (m->N * 8 <= (int64_t)sms * 8 * 32)
        run(k_lte<8>, 8);
    else if (m->L <= 16)
        run(k_lte<1>, 1);
    else
        run(k_lte<2>, 2);
    MGT_LAUNCH_CHECK("k_lte");
    m->line_dirty = true;
    return MGT_OK;
}

// ---------------------------------------------------------------------------
// Line data per (point, line) from the populations.
//   net = n_l B_lu - n_u B_ul, floored at 1e-30 (n_l B_lu + n_u B_ul) (counted),
//   chi^{ij} = (h nu / 4 pi) net,  S^{ij} = n_u A_ul / net.
// Stored scaled for the solver:
//   chi~' = chi^{ij} / (nu w sqrt(pi)) * L_unit  -- opacity per length unit at
//           line centre, so that chi(nu) = chi~ exp(-u^2);
//   S'    = S^{ij} / U_line, U_line = (2 h nu^3/c^2) max(n_bg(nu), 1e-15)
//         = n_u B_ul / (net * nbgmax).
// Row layout (see row_stride32): chi~' of every line, then S' of every line,
// then w and 1/w of the point, then (FP32 rows only) the range figure
// G = max(chi~max dxmax / 2^8, S'max / 2^80) of the formal solution's two-row
// elimination (chi~max, S'max the largest over the point's lines, dxmax its
// longest graph edge) and a zero.
// A block takes kLDPoints points and deals out their (point, line slot) items
// 256 at a time: bound by the FP64 pipe (16 cycles per warp instruction whatever
// the active lanes), which with one warp per point ran 40 slots in two trips of
// 32 lanes and three divisions per point in one lane.  100k points x 40 lines:
// 0.42 -> 0.14 ms; x 4 lines 0.21 -> 0.04 ms.
// ---------------------------------------------------------------------------
struct LDArgs {
    int64_t N;
    int L, M, Mpad;
    const double *pops, *w64, *line_tab;
    const int32_t *line_ul;
    const float *dxmax;
    double Lunit;
    float *out32;
    double *out64;
    unsigned long long *n_floor;
    int *range_bad;           // set when a point's range figure exceeds 1 (zeroed before the launch)
};

constexpr int kLDThreads = 256, kLDPoints = 32;

// Points p0 .. p0 + kLDPoints - 1 of a model, by the whole block.
__device__ __forceinline__ void line_data_block(const LDArgs &d, int64_t p0)
{
    __shared__ double s_cw[kLDPoints];
    __shared__ int s_chi[kLDPoints], s_src[kLDPoints];   // largest chi~', S' (bits; non-negative, a NaN is largest)
    const int n = (int)min((int64_t)kLDPoints, d.N - p0);
    const int Mpad = d.Mpad, RS = row_stride32(Mpad), RS64 = row_stride64(Mpad);
    const double *__restrict__ line_tab = d.line_tab;
    const int32_t *__restrict__ line_ul = d.line_ul;
    const int tid = threadIdx.x;
    if (tid < n) {
        // h L_unit / (4 pi sqrt(pi) w): one FP64 division per point, not per line
        s_cw[tid] = kH * d.Lunit / (4.0 * kPi * kSqrtPi * d.w64[p0 + tid]);
        s_chi[tid] = s_src[tid] = 0;
    }
    __syncthreads();
    // item e = (point e / Mpad, slot e mod Mpad); 8 neighbouring lanes share a
    // point (Mpad and the block are multiples of 8)
    const int dp = kLDThreads / Mpad, dk = kLDThreads - dp * Mpad;
    int i = tid / Mpad, k = tid - i * Mpad;
    for (int e0 = 0; e0 < n * Mpad; e0 += kLDThreads) {
        float f0 = 0.0f, f1 = 0.0f;
        if (i < n) {
            const int64_t p = p0 + i;
            double a0 = 0.0, a1 = 0.0;
            if (k < d.M) {
                const int u = line_ul[k], l = line_ul[Mpad + k];
                const double Bul = line_tab[2 * Mpad + k], Blu = line_tab[3 * Mpad + k];
                const double nbgmax = line_tab[4 * Mpad + k];
                const double nu_ = d.pops[p * d.L + u], nl_ = d.pops[p * d.L + l];
                const double a = nl_ * Blu, b = nu_ * Bul;
                double net = a - b;
                const double floor_ = 1e-30 * (a + b);
                if (net < floor_) {
                    net = floor_;
                    atomicAdd(d.n_floor, 1ULL);
                }
                if (net > 0.0) {
                    a0 = net * s_cw[i];
                    a1 = b / (net * nbgmax);
                }
            }
            f0 = (float)a0;
            f1 = (float)a1;
            float *r32 = d.out32 + p * RS;
            r32[k] = f0;
            r32[Mpad + k] = f1;
            if (d.out64) {
                double *r64 = d.out64 + p * RS64;
                r64[k] = a0;
                r64[Mpad + k] = a1;
            }
        }
        int c = f0 == f0 ? __float_as_int(f0) : 0x7fffffff, t = f1 == f1 ? __float_as_int(f1) : 0x7fffffff;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            c = max(c, __shfl_xor_sync(0xffffffffu, c, o));
            t = max(t, __shfl_xor_sync(0xffffffffu, t, o));
        }
        if ((tid & 7) == 0 && i < n) {
            atomicMax(&s_chi[i], c);
            atomicMax(&s_src[i], t);
        }
        i += dp;
        k += dk;
        if (k >= Mpad) {
            k -= Mpad;
            ++i;
        }
    }
    __syncthreads();
    if (tid < n) {
        const int64_t p = p0 + tid;
        const double w = d.w64[p], rw = 1.0 / w;
        float *r32 = d.out32 + p * RS;
        r32[2 * Mpad] = (float)w;
        r32[2 * Mpad + 1] = (float)rw;
        // range figure of the formal solution's two-row elimination: at most 1
        // when every step through the point has half depths <= kTwoRowDepth and
        // sources <= kTwoRowSource; NaN and infinity give a figure above 1
        // (a width above 1% of c, where no real line is, would also let the
        // background of the far bins outgrow the range: it sets the flag too)
        const float chi_max = __int_as_float(s_chi[tid]), S_max = __int_as_float(s_src[tid]);
        const float G = fmaxf(chi_max * d.dxmax[p] / kTwoRowDepth, S_max / kTwoRowSource);
        const bool inside = chi_max == chi_max && S_max == S_max && G <= 1.0f && w < 0.01;
        r32[2 * Mpad + 2] = inside ? G : 2.0f;
        r32[2 * Mpad + 3] = 0.0f;
        if (!inside) atomicOr(d.range_bad, 1);
        if (d.out64) {
            double *r64 = d.out64 + p * RS64;
            r64[2 * Mpad] = w;
            r64[2 * Mpad + 1] = rw;
        }
    }
}

__global__ void __launch_bounds__(kLDThreads) k_line_data(LDArgs d)
{
    line_data_block(d, (int64_t)blockIdx.x * kLDPoints);
}

// Many models in one launch: blk_end[i] is one past the last CTA of model i.
__global__ void __launch_bounds__(kLDThreads) k_line_data_batch(const LDArgs *__restrict__ args,
                                                                const int64_t *__restrict__ blk_end, int n_models)
{
    __shared__ LDArgs sd;
    __shared__ int64_t s_first;
    if (threadIdx.x == 0) {
        const int64_t b = blockIdx.x;
        int lo = 0, hi = n_models - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (blk_end[mid] > b) hi = mid; else lo = mid + 1;
        }
        sd = args[lo];
        s_first = lo > 0 ? blk_end[lo - 1] : 0;
    }
    __syncthreads();
    line_data_block(sd, ((int64_t)blockIdx.x - s_first) * kLDPoints);
}

static LDArgs fill_ld_args(const mgt_model *m)
{
    return LDArgs{m->N, m->L, m->M, m->Mpad, m->d_pops, m->d_w64, m->d_line_tab, m->d_line_ul, m->d_dxmax,
                  m->L_unit, m->d_line32, m->d_line64, m->d_count + 0, m->d_range_bad};
}

mgt_status launch_line_data(mgt_model *m, cudaStream_t s)
{
    MGT_CUDA(cudaMemsetAsync(m->d_range_bad, 0, sizeof(int), s));
    {
        // populations and w in; the FP32 row (and the FP64 row if kept) out
        const double ld_bytes = (double)m->N * (8.0 * m->L + 8.0 + 4.0 * row_stride32(m->Mpad) +
                                                 (m->d_line64 ? 8.0 * row_stride64(m->Mpad) : 0.0));
        MGT_KTIMER_BYTES("k_line_data", s, ld_bytes);
        k_line_data<<<ceil_div(m->N, (int64_t)kLDPoints), kLDThreads, 0, s>>>(fill_ld_args(m));
    }
    MGT_LAUNCH_CHECK("k_line_data");
    m->line_dirty = false;
    return MGT_OK;
}

size_t ld_args_bytes() { return sizeof(LDArgs); }

mgt_status ld_batch_args(const mgt_model *m, void *args, int64_t *blocks)
{
    const LDArgs a = fill_ld_args(m);
    std::memcpy(args, &a, sizeof a);
    *blocks = ceil_div(m->N, (int64_t)kLDPoints);
    return MGT_OK;
}

// Zero every model's range flag before the batched line data set them.
__global__ void k_reset_range(const LDArgs *__restrict__ args, int n_models)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n_models) *args[i].range_bad = 0;
}

mgt_status ld_batch_launch(const void *d_args, const int64_t *d_blk_end, int n_models, int64_t n_blocks,
                           cudaStream_t s)
{
    k_reset_range<<<ceil_div(n_models, 256), 256, 0, s>>>(static_cast<const LDArgs *>(d_args), n_models);
    MGT_LAUNCH_CHECK("k_reset_range");
    k_line_data_batch<<<(unsigned)n_blocks, kLDThreads, 0, s>>>(static_cast<const LDArgs *>(d_args), d_blk_end, n_models);
    MGT_LAUNCH_CHECK("k_line_data_batch");
    return MGT_OK;
}

// ---------------------------------------------------------------------------
// Ray walk (bit-exact FP64 predicates; no multiply-add fusion).
//
// From the current point c (start c = o) the candidates are the neighbours m
// of c with Z_m = (x_m - x_o).n > Z_c; the winner minimises the squared
// distance to the ray line |(x_m - x_o) - Z_m n|^2, ties to the smaller index.
// The walk ends on a boundary point (kept) or stalls without a candidate (a
// boundary origin without candidates just has an empty half-ray).
// ---------------------------------------------------------------------------
struct WalkArgs {
    int64_t N;
    int32_t R;
    const double *pos;
    const int32_t *off;
    const int32_t *nb;
    const double *nb_pos;     // [nnz][3] position of each neighbour entry (contiguous per point)
    double pos_scale;         // power of two near 1 / (largest coordinate): exact scaling
    const uint8_t *bnd;
    const double *dirs;
    const float4 *ent;        // packed neighbour entries, two float4 each (see kWalkRow)
    const int32_t *ent_row;   // [N] first chunk of each point's row of packed entries
    const float *pos_hl;      // [N][6] positions times pos_scale, split into float hi + lo
    const float4 *dirs32;     // [R] directions in FP32
    const int32_t *order;     // walks of one direction are visited in this point order
    float pos_slack;          // bound on |x - (hi + lo)| over all coordinates
    unsigned long long *n_exact;   // steps decided by the FP64 predicates
    int32_t n_chunks;         // chunks of packed entries (index bound)
    const int32_t *dir_map;   // walk direction r -> model direction (NULL: the same); R counts walk directions
};

__device__ __forceinline__ uint64_t walk_clock_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// First device error wins; err[1..3] say where (site) and which walk / step.
__device__ __forceinline__ void walk_give_up(int *err, int site, int64_t wg, int64_t n)
{
    if (atomicCAS(err, 0, (int)kDevTimeout) == 0) {
        err[1] = site;
        err[2] = (int)wg;
        err[3] = (int)n;
    }
}

__device__ __forceinline__ double dot3_exact(double ax, double ay, double az, double bx, double by, double bz)
{
    return __dadd_rn(__dadd_rn(__dmul_rn(ax, bx), __dmul_rn(ay, by)), __dmul_rn(az, bz));
}

// Next point of the walk from c in FP64, the defining arithmetic, or -1, found
// by the whole warp (every argument the same in every lane): one candidate per
// lane, the least (squared distance, index) over the lanes.  Returned with the
// winner's Z in every lane.  One lane alone took ~15 times the FP64 warp
// instructions, and an instruction costs this GPU's FP64 pipe the same 16
// cycles for one lane as for 32.
__device__ __noinline__ int walk_next_exact(const int32_t *__restrict__ off, const int32_t *__restrict__ nb,
                                            const double *__restrict__ nb_pos, int c, double xo, double yo, double zo,
                                            double n0, double n1, double n2, double Zc, double *Znext)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int32_t k0 = off[c], k1 = off[c + 1];
    int best = 0x7fffffff;
    double bestd = 0.0, bestZ = 0.0;
    bool have = false;
    for (int32_t kb = k0; kb < k1; kb += 32) {
        const int32_t k = kb + lane;
        if (k >= k1) continue;
        const int mm = nb[k];
        const double dx = __dsub_rn(nb_pos[3 * (int64_t)k], xo);
        const double dy = __dsub_rn(nb_pos[3 * (int64_t)k + 1], yo);
        const double dz = __dsub_rn(nb_pos[3 * (int64_t)k + 2], zo);
        const double Z = dot3_exact(dx, dy, dz, n0, n1, n2);
        if (!(Z > Zc)) continue;
        const double px = __dsub_rn(dx, __dmul_rn(Z, n0));
        const double py = __dsub_rn(dy, __dmul_rn(Z, n1));
        const double pz = __dsub_rn(dz, __dmul_rn(Z, n2));
        const double d2 = dot3_exact(px, py, pz, px, py, pz);
        if (!have || d2 < bestd || (d2 == bestd && mm < best)) {
            have = true;
            best = mm;
            bestd = d2;
            bestZ = Z;
        }
    }
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) {
        const bool oh = __shfl_xor_sync(full, have, o);
        const int ob = __shfl_xor_sync(full, best, o);
        const double od = __shfl_xor_sync(full, bestd, o), oz = __shfl_xor_sync(full, bestZ, o);
        if (oh && (!have || od < bestd || (od == bestd && ob < best))) {
            have = true;
            best = ob;
            bestd = od;
            bestZ = oz;
        }
    }
    *Znext = bestZ;
    return have ? best : -1;
}

// Per-walk constants, all FP32 (GB300's FP64 pipe is far too narrow for
// per-walk or per-step FP64 work; the FP64 values are loaded only on the rare
// steps the FP32 filter cannot settle).
struct WalkFrame {
    float ohx, ohy, ohz, olx, oly, olz; // origin (scaled) split into hi + lo floats
    float f0, f1, f2;                  // direction in FP32
};

__device__ __forceinline__ WalkFrame make_frame(const WalkArgs &a, int64_t o, int r)
{
    WalkFrame f;
    const float *p = a.pos_hl + 6 * o;
    f.ohx = p[0];
    f.ohy = p[1];
    f.ohz = p[2];
    f.olx = p[3];
    f.oly = p[4];
    f.olz = p[5];
    const float4 n = a.dirs32[r];
    f.f0 = n.x;
    f.f1 = n.y;
    f.f2 = n.z;
    return f;
}


// 32 bytes at a 32-byte aligned address of read-only memory, in one load.
struct Vec8 {
    float4 a, b;
};

__device__ __forceinline__ Vec8 load32(const void *p)
{
    Vec8 v;
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(v.a.x), "=f"(v.a.y), "=f"(v.a.z), "=f"(v.a.w), "=f"(v.b.x), "=f"(v.b.y), "=f"(v.b.z), "=f"(v.b.w)
        : "l"(p));
    return v;
}

// Minimum over the calling lane's walk (a group of G lanes).
template <int G> __device__ __forceinline__ float group_min(float v)
{
#pragma unroll
    for (int o = 1; o < G; o <<= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// ---------------------------------------------------------------------------
// One walk per group of G lanes: eight walks per warp (G = kWalkRow = 4), or two
// (G = 16) in launches of few walks, see walk_wide.  Each step reads
// the current point's row of packed neighbour entries (the neighbour's scaled
// position as float hi + lo, its index with its boundary flag and a last-chunk
// flag, and its own row), G / 4 chunks (128-byte lines) per load and group, so
// the next step's row, the winner's index and its boundary flag arrive with
// the candidates: one dependent L2 round trip per load.
//
// The lanes evaluate the candidates with FP32 arithmetic and error bounds that
// cover both the FP32 and the FP64 rounding.  With u = 2^-24 = 6e-8, S the sum
// of the offset's three magnitudes, and s = pos_slack = 2^-46 for what hi + lo
// leave out and the low parts' rounding:
//   offsets    d = (h - h_o) + (l - l_o): |d32 - d64| <= 2u |d| + 2s per component
//   projection |Z32 - Z64| <= 2u S + 2s sqrt(3)  (offsets) + u S (direction in FP32)
//              + 3u S (three operations) + u S (adding the bound)
//              <= eZ = 5e-7 S + 4s
//   p = d - Z n: the error's length <= 2u S + 2s sqrt(3) + eZ + 2u S
//              <= ep = 8e-7 S + 8s
//   squared distance |d2_32 - d2_64| <= 2 |p32| ep + ep^2 + 3u d2, and u d2 for
//              each of Lo, U = 2 d2 - Lo and their rounding
//              <= e2 = ep (2.5 |p32| + ep) + 4e-7 d2
// (2.5 for 2 covers the approximate square root).  Coarser bounds from the
// largest components, ten times these, took a quarter more instructions per
// candidate and sent ten times as many steps to FP64.
// The current point's projection Z_c is carried as the winner's FP32 value
// with its bound eZ_c.  A neighbour is a candidate when Z32 - eZ clears
// Z_c + eZ_c, not one when Z32 + eZ stays at or below Z_c - eZ_c; anything in
// between leaves the step undecided.  The FP32 winner (smallest d2, lowest
// lane) is accepted only if its upper d2 bound is below every other
// candidate's lower bound, so near-ties never decide.  Undecided steps run
// walk_next_exact, the FP64 predicates themselves (exact Z_c recomputed by
// the same expression), one walk of the warp after the other.  The point lists
// are therefore those of the FP64 rule.
//
// Four modes share the walk:
//  * kWalkFused: every walk of the grid.  Writes the half-ray length, counts
//    stalls, and writes the point indices into a fixed-stride scratch area
//    (K per walk); those of steps >= K are not kept (such walks are redone by
//    the list mode).  k_walk_compact makes the step records from them.
//  * kWalkList: the walks named in `list` only, point indices written into
//    the records at their final place (ray offsets known).
//  * kWalkImg / kWalkImgFill: the two half-rays of every image pixel (walk
//    2q + h: h = 0 along -n, h = 1 along +n, n toward the observer), from the
//    pixel's anchor point, distances to the pixel line, Z measured from the
//    pixel's reference point; the first mode writes the lengths and the point
//    indices into scratch slots, the fill mode, used when a half-ray is longer
//    than its slot, the point indices of the full ray (far half reversed,
//    anchor, near half).
// ---------------------------------------------------------------------------
constexpr int kWalkFused = 0, kWalkList = 1, kWalkImg = 2, kWalkImgFill = 3;

struct ImgWalkArgs {
    const double *ref;        // [npix][3] pixel reference points
    const int32_t *anchor;    // [npix] start point of both half-rays
    const int64_t *off;       // [npix+1] full-ray offsets (fill mode)
    int32_t *pts;             // full rays (fill mode)
    int64_t npix;
    double n[3];              // unit direction toward the observer
};

// What bounds it: instruction issue (73 warp instructions per step, 75 % of the
// slots, 20k shell points) and the L2 round trips of the rows.  Four lanes per walk
// read a row (15.5 entries on average) in its own 128-byte lines with few lanes
// past its end; the decision's shuffles and the loop serve eight walks at once;
// and walks of neighbouring origins step together, so their rows coincide in
// L1.  Walk kernel, 100k shell points x 48 directions (1.9e8 steps): 36.9 ms
// with 16 lanes per walk, records made inside, 64 registers; 16.0 ms with 4
// lanes and the records left to k_walk_compact; 14.9 ms at 48 registers (ten
// blocks of 128 threads per SM, and 32 to 44 bytes of spills; 16.0 at eight, 18.8
// at six, 17.5 at fourteen);
// 14.4 ms with 256-bit loads; 13.2 ms with the bounds above.  Before those, 8
// lanes per walk took 18.7 ms, 2 lanes 16.2 ms.
// Not kept: loading the next chunk ahead (16.8 ms, a quarter of the loads
// wasted), and giving a finished group the warp's next walk (16.7 ms: the
// walks of a warp no longer pass the same rows together).
// Every launch goes through launch_walk.
constexpr int kWalkThreads = 128, kWalkBlocks = 10;

template <int MODE, int G>
__global__ void __launch_bounds__(kWalkThreads, kWalkBlocks) k_walk(WalkArgs a, int64_t *__restrict__ lens,
                                                          const int64_t *__restrict__ ray_off,
                                                          const int64_t *__restrict__ list, int64_t n_list, int32_t K,
                                                          unsigned long long *__restrict__ n_stall,
                                                          int32_t *__restrict__ scratch, Step32 *__restrict__ steps,
                                                          int *__restrict__ err, ImgWalkArgs im)
{
    constexpr bool IMG = MODE == kWalkImg || MODE == kWalkImgFill;
    static_assert(G % kWalkRow == 0 && 32 % G == 0, "whole chunks per group, whole groups per warp");
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, sl = lane & (G - 1), first = lane & ~(G - 1);
    const unsigned gmask = ((1u << G) - 1u) << first;
    const int64_t wg = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / G;   // walk slot
    const int64_t W = MODE == kWalkFused ? (int64_t)a.R * a.N : IMG ? 2 * im.npix : n_list;
    if (wg - first / G >= W) return;                           // every walk of the warp absent
    bool live = wg < W;
    int r = 0;
    int64_t o64 = 0;
    if (live) {
        if (MODE == kWalkFused) {
            r = (int)(wg / a.N);
            o64 = a.order[wg - (int64_t)r * a.N];
        } else if (IMG) {
            r = (int)(wg & 1);
            o64 = im.anchor[wg >> 1];
        } else {
            const int64_t t = list[wg];
            r = (int)(t / a.N);
            o64 = t - (int64_t)r * a.N;
        }
    }
    if (o64 < 0 || o64 >= a.N || r < 0 || r >= (IMG ? 2 : a.R)) {   // index check: record and skip
        walk_give_up(err, 13, wg, o64);
        o64 = 0;
        r = 0;
        live = false;
    }
    const int o = (int)o64;
    const int64_t wi = (int64_t)r * a.N + o;
    const int rg = (!IMG && a.dir_map) ? a.dir_map[r] : r;   // the model's direction index
    // the walk's frame: origin o and direction r, or for image walks the pixel's
    // reference point and -n / +n (FP64 values are loaded again where needed)
    WalkFrame f;
    double img_Z0 = 0.0;                        // image walks: Z of the anchor
    if (IMG) {
        const double sg = r == 0 ? -1.0 : 1.0;
        const double *pr = im.ref + 3 * (live ? wg >> 1 : 0);
        const double sx = pr[0] * a.pos_scale, sy = pr[1] * a.pos_scale, sz = pr[2] * a.pos_scale;
        f.ohx = (float)sx;
        f.ohy = (float)sy;
        f.ohz = (float)sz;
        f.olx = (float)(sx - (double)f.ohx);
        f.oly = (float)(sy - (double)f.ohy);
        f.olz = (float)(sz - (double)f.ohz);
        f.f0 = (float)(sg * im.n[0]);
        f.f1 = (float)(sg * im.n[1]);
        f.f2 = (float)(sg * im.n[2]);
        const double *q = a.pos + 3 * (int64_t)o;
        img_Z0 = dot3_exact(__dsub_rn(q[0], pr[0]), __dsub_rn(q[1], pr[1]), __dsub_rn(q[2], pr[2]), sg * im.n[0],
                            sg * im.n[1], sg * im.n[2]);
    } else {
        f = make_frame(a, o, rg);
    }
    int c = o, n = 0;                           // current point, steps taken
    int c_row = live ? a.ent_row[o] : 0;        // the current point's row of packed entries
    float Zc = 0.0f, eZc = 0.0f;                // Z of o is exactly 0 (image walks: the anchor's Z)
    if (IMG) {
        Zc = (float)(img_Z0 * a.pos_scale);     // the filter works in scaled units (exact factor)
        eZc = 2e-7f * fabsf(Zc) + 1e-30f;
    }
    // where point index k goes (lane sl keeps the index of step k = sl mod G
    // until the group's G indices are written together)
    auto put = [&](int k, int32_t pt) {
        if (MODE == kWalkFused || MODE == kWalkImg) {
            if (k < K) scratch[(IMG ? wg : wi) * (int64_t)K + k] = pt;
        } else if (MODE == kWalkList) {
            const int64_t at = ray_off[wi] + k;
            if (at < ray_off[wi + 1])
                steps[at].x = pt;
            else
                atomicCAS(err, 0, (int)kDevBounds);    // cannot happen: deterministic walk
        } else if (MODE == kWalkImgFill) {
            const int nfar = (int)lens[wg & ~(int64_t)1];
            if (k < (int)lens[wg])
                im.pts[im.off[wg >> 1] + (r == 0 ? nfar - 1 - k : nfar + 1 + k)] = pt;
            else
                atomicCAS(err, 0, (int)kDevBounds);
        }
    };
    int32_t my_pt = 0;
    bool done = !live, gave_up = false;
    // every loop below is bounded: the walk by the point count and a 2 s
    // clock, a row scan by the number of chunks; running out records the site
    // and returns.  All live walks of the warp have taken `it` steps.
    const uint64_t t_start = walk_clock_ns();
    const float slack4 = 4.0f * a.pos_slack, slack8 = 8.0f * a.pos_slack;
    int it = 0;
    for (; __any_sync(full, !done); ++it) {
        if ((it & 15) == 15 && __any_sync(full, walk_clock_ns() - t_start > 2000000000ull)) {
            if (sl == 0 && !done) walk_give_up(err, 1, wg, n);
            gave_up = true;
            break;
        }
        // each lane keeps the best of its own entries over the row's chunks
        // (smallest d2, the earlier chunk on ties) and the least lower bound
        // of its other candidates; the group decides once per step
        float bd2 = 3.0e38f, bLo = 3.0e38f, bZ = 0.0f, beZ = 0.0f, lo2 = 3.0e38f;
        uint32_t bword = 0u;
        int brow = 0;
        bool und = false;
        const float Zhi = Zc + eZc, Zlo = Zc - eZc;
        auto candidate = [&](const float4 &e0, const float4 &e1) {
            const float2 dxy = __fadd2_rn(__fadd2_rn(make_float2(e0.x, e0.y), make_float2(-f.ohx, -f.ohy)),
                                          __fadd2_rn(make_float2(e1.x, e1.y), make_float2(-f.olx, -f.oly)));
            const float dx = dxy.x, dy = dxy.y, dz = (e0.z - f.ohz) + (e1.z - f.olz);
            const float S = fabsf(dx) + fabsf(dy) + fabsf(dz);
            const float Z = fmaf(dz, f.f2, fmaf(dy, f.f1, dx * f.f0));
            const float eZ = fmaf(5e-7f, S, slack4);
            if (Z - eZ > Zhi) {
                const float px = fmaf(-Z, f.f0, dx), py = fmaf(-Z, f.f1, dy), pz = fmaf(-Z, f.f2, dz);
                const float d2 = fmaf(pz, pz, fmaf(py, py, px * px));
                const float ep = fmaf(8e-7f, S, slack8);
                float rp;
                asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(rp) : "f"(d2));
                const float e2 = fmaf(ep, fmaf(2.5f, rp, ep), 4e-7f * d2);
                const float Lo = d2 - e2;
                const bool best = d2 < bd2;
                lo2 = fminf(lo2, best ? bLo : Lo);
                if (best) {
                    bd2 = d2;
                    bLo = Lo;
                    bZ = Z;
                    beZ = eZ;
                    bword = __float_as_uint(e0.w);
                    brow = __float_as_int(e1.w);
                }
            } else if (Z + eZ > Zlo) {
                und = true;
            }
        };
        if constexpr (G == kWalkRow) {
            for (int kb = done ? -1 : c_row; kb != -1;) {
                if ((unsigned)kb >= (unsigned)a.n_chunks) {    // index check: record and end the row
                    walk_give_up(err, 10, wg, kb);
                    break;
                }
                const Vec8 e = load32(a.ent + 2 * ((int64_t)kb * kWalkRow + sl));
                // (the same in every lane of the group)
                kb = (__float_as_uint(e.a.w) & kEntLast) ? -1 : kb + 1;
                candidate(e.a, e.b);
            }
        } else {
            bool open = !done;
            for (int kb = c_row; __any_sync(full, open); kb += G / kWalkRow) {
                if (open && (unsigned)kb >= (unsigned)a.n_chunks) {
                    walk_give_up(err, 10, wg, kb);
                    open = false;
                }
                const int chunk = kb + sl / kWalkRow;
                const bool in = open && chunk < a.n_chunks;
                Vec8 e{};
                if (in) e = load32(a.ent + 2 * ((int64_t)chunk * kWalkRow + sl % kWalkRow));
                // chunks up to the group's first one with the last-chunk flag belong to the row
                const unsigned last = __ballot_sync(full, in && (__float_as_uint(e.a.w) & kEntLast)) & gmask;
                if (in && (last & ((1u << (lane & ~(kWalkRow - 1))) - 1u)) == 0u) candidate(e.a, e.b);
                open = open && last == 0u;
            }
        }
        __syncwarp();
        // The FP32 winner is the group's smallest d2 (lowest lane on ties); it
        // is accepted only if every other candidate's lower bound lies above
        // its upper bound (a negative lower bound always fails, since upper
        // bounds are >= 0), so a tie never decides.
        const float dmin = group_min<G>(bd2);
        const bool have = dmin < 3.0e38f;
        const unsigned wins = __ballot_sync(full, have && bd2 == dmin) & gmask;
        const int src = wins ? __ffs(wins) - 1 : lane;
        const float bU = 2.0f * dmin - __shfl_sync(full, bLo, src);
        bZ = __shfl_sync(full, bZ, src);
        beZ = __shfl_sync(full, beZ, src);
        bword = __shfl_sync(full, bword, src);
        brow = __shfl_sync(full, brow, src);
        const float lo_other = lane == src ? lo2 : fminf(bLo, lo2);
        // (every warp intrinsic runs in all lanes: none behind a short circuit)
        const bool close = (__ballot_sync(full, und || (have && lo_other <= bU)) & gmask) != 0u;
        const bool exact = !done && close;
        int v = -1;
        double Zn = 0.0;
        // (rare) the FP64 predicates, for one undecided walk after the other
        for (unsigned todo = __ballot_sync(full, exact && sl == 0); todo; todo &= todo - 1u) {
            const int w = __ffs(todo) - 1;
            const int wo = __shfl_sync(full, o, w), wc = __shfl_sync(full, c, w), wr = __shfl_sync(full, rg, w);
            if (!IMG && lane == 0) atomicAdd(a.n_exact, 1ULL);
            double xo, yo, zo, n0, n1, n2;
            if constexpr (IMG) {
                const double *po = im.ref + 3 * (__shfl_sync(full, wg, w) >> 1);
                const double sg = wr == 0 ? -1.0 : 1.0;
                xo = po[0];
                yo = po[1];
                zo = po[2];
                n0 = sg * im.n[0];
                n1 = sg * im.n[1];
                n2 = sg * im.n[2];
            } else {
                const double *po = a.pos + 3 * (int64_t)wo, *pn = a.dirs + 3 * wr;
                xo = po[0];
                yo = po[1];
                zo = po[2];
                n0 = pn[0];
                n1 = pn[1];
                n2 = pn[2];
            }
            double Zc64 = 0.0;
            if (wc != wo || IMG) {
                const double *q = a.pos + 3 * (int64_t)wc;
                Zc64 = dot3_exact(__dsub_rn(q[0], xo), __dsub_rn(q[1], yo), __dsub_rn(q[2], zo), n0, n1, n2);
            }
            double z;
            const int nv = walk_next_exact(a.off, a.nb, a.nb_pos, wc, xo, yo, zo, n0, n1, n2, Zc64, &z);
            if (first == w) {
                v = nv;
                Zn = z;
            }
        }
        if (!done) {
            int nx = -1;
            bool nx_bnd = false;
            if (exact) {
                nx = v;
                if (nx >= a.N) {
                    walk_give_up(err, 11, wg, nx);
                    nx = -1;
                }
                Zc = (float)(Zn * a.pos_scale);      // the filter works in scaled units (exact factor)
                eZc = 2e-7f * fabsf(Zc) + 1e-30f;
                if (nx >= 0) {
                    nx_bnd = a.bnd[nx] != 0;
                    c_row = a.ent_row[nx];
                }
            } else if (have) {
                nx = (int)(bword & kEntIdx);
                if (nx >= a.N) {
                    walk_give_up(err, 12, wg, nx);
                    nx = -1;
                }
                nx_bnd = (bword & kEntBnd) != 0u;
                c_row = brow;
                Zc = bZ;
                eZc = beZ;
            }
            if (nx < 0) {
                if (MODE == kWalkFused && sl == 0 && !(c == o && a.bnd[o])) atomicAdd(n_stall, 1ULL);
                done = true;
            } else {
                if (sl == (it & (G - 1))) my_pt = nx;
                ++n;
                c = nx;
                done = nx_bnd || n >= a.N;
            }
        }
        // a full chunk of indices (a finished walk's last ones are written
        // with its neighbours' next chunk; n bounds what is written)
        if ((it & (G - 1)) == G - 1) {
            const int k = it - (G - 1) + sl;
            if (k < n) put(k, my_pt);
        }
    }
    if ((it & (G - 1)) != 0) {
        const int k = (it & ~(G - 1)) + sl;
        if (k < n) put(k, my_pt);
    }
    if (live && sl == 0) {
        if (MODE == kWalkFused)
            lens[wi] = gave_up ? 0 : n;
        else if (MODE == kWalkImg)
            lens[wg] = gave_up ? 0 : n;
        else if (!gave_up && n != (MODE == kWalkList ? ray_off[wi + 1] - ray_off[wi] : lens[wg]))
            atomicCAS(err, 0, (int)kDevBounds);
    }
}

// Launches of few walks take 16 lanes per walk: a step's latency counts there,
// not its instructions (a row is one or two dependent loads instead of four or
// five).  The line lies where a launch fills three quarters of the GPU at 4
// lanes: 12,000 walks (sphere models, 12 directions) take 32 us with 16 lanes
// and 48 us with 4; 30,000 take 62 and 65; 48,000 take 97 and 85; 240,000 take
// 592 and 386.
inline bool walk_wide(int64_t walks, int sms)
{
    return walks < (int64_t)sms * kWalkBlocks * (kWalkThreads / kWalkRow) * 3 / 4;
}

template <int MODE>
static mgt_status launch_walk(const WalkArgs &a, int64_t walks, int64_t *lens, const int64_t *ray_off,
                              const int64_t *list, int32_t K, unsigned long long *n_stall, int32_t *scratch,
                              Step32 *steps, int *err, const ImgWalkArgs &im, cudaStream_t s)
{
    int dev = 0, sms = 0;
    MGT_CUDA(cudaGetDevice(&dev));
    MGT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const auto run = [&](auto kernel, int lanes) {
        kernel<<<(unsigned)ceil_div(walks * lanes, kWalkThreads), kWalkThreads, 0, s>>>(
            a, lens, ray_off, list, walks, K, n_stall, scratch, steps, err, im);
    };
    if (walk_wide(walks, sms))
        run(k_walk<MODE, 16>, 16);
    else
        run(k_walk<MODE, kWalkRow>, kWalkRow);
    MGT_LAUNCH_CHECK("k_walk");
    return MGT_OK;
}

// Walks whose indices did not fit their scratch slot (length > K).
__global__ void k_walk_overflow(int64_t W, const int64_t *__restrict__ lens, int32_t K, int64_t *__restrict__ list,
                                unsigned long long *__restrict__ count)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= W || lens[t] <= K) return;
    list[atomicAdd(count, 1ULL)] = t;
}

// What a step record takes from a point, one 64-byte row: positions times
// pos_scale and v/c as float hi + lo, and the line width.
struct __align__(64) WalkPoint {
    float4 q[4];              // {hx, hy, hz, lx}, {ly, lz, vhx, vhy}, {vhz, vlx, vly, vlz}, {w, 0, 0, 0}
};

__global__ void k_walk_points(int64_t N, const float *__restrict__ pos_hl, const float *__restrict__ vel_hl,
                              const float2 *__restrict__ w32, WalkPoint *__restrict__ out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const float *p = pos_hl + 6 * i, *v = vel_hl + 6 * i;
    out[i].q[0] = make_float4(p[0], p[1], p[2], p[3]);
    out[i].q[1] = make_float4(p[4], p[5], v[0], v[1]);
    out[i].q[2] = make_float4(v[2], v[3], v[4], v[5]);
    out[i].q[3] = make_float4(w32[i].x, 0.0f, 0.0f, 0.0f);
}

// Step records from the walks' point indices, one walk per 16 lanes: walk t's
// indices in its scratch slot (at most K; a longer walk is left to the list
// form), or (LIST) already in the records of the walks named in `list`.  The
// lanes hold 16 consecutive points of the ray, the first of them from the trip
// before (the origin at first), and lanes 1-15 write the records of the steps
// ending at their points.  All in FP32: dx from the hi + lo scaled positions,
// beta = n.(v_c - v_o)/c and dbeta = n.(v_c - v_prev)/c from hi + lo values of
// v/c (relative error about 1e-7 of |v_c - v_o|/c), the averaged width of the
// segment.  Bound by the gathers of the points' rows (one L1 wavefront per lane
// and 32 bytes): 2.6 ms for 1.9e8 records.  A record moves 20 bytes of DRAM
// traffic here instead of 48 through a slot of finished records, and the walk,
// whose lanes gathered one record at a time, keeps only point indices.
template <bool LIST>
__global__ void __launch_bounds__(256, 5) k_walk_compact(WalkArgs a, int64_t W, const int64_t *__restrict__ ray_off,
                                                      const int64_t *__restrict__ list, int32_t K,
                                                      const int32_t *__restrict__ scratch,
                                                      const WalkPoint *__restrict__ pt, float inv_Lunit, int width_mode,
                                                      Step32 *__restrict__ steps, int *__restrict__ err)
{
    const unsigned full = 0xffffffffu;
    const int64_t slot = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 4;
    const int sl = threadIdx.x & 15;
    int64_t t = 0, base = 0, n = 0;
    if (slot < W) {
        t = LIST ? list[slot] : slot;
        base = ray_off[t];
        n = ray_off[t + 1] - base;
        if (!LIST && n > K) n = 0;
    }
    const int r = (int)(t / a.N);
    const int o = (int)(t - (int64_t)r * a.N);
    const float4 dir = a.dirs32[a.dir_map ? a.dir_map[r] : r];
    const float4 o1 = pt[o].q[1], o2 = pt[o].q[2];
    auto point = [&](int64_t j) {                // step j's point, -1 (and past the end) the origin
        return j >= 0 && j < n ? (LIST ? steps[base + j].x : scratch[t * (int64_t)K + j]) : o;
    };
    int nc = point(sl - 1);
    for (int64_t j0 = -1; __any_sync(full, j0 + 1 < n); j0 += 15) {
        const int64_t j = j0 + sl;
        int c = nc;
        nc = point(j + 15);                      // the next trip's, ahead of this one's gathers
        if (c < 0 || c >= a.N) {                 // index check: record, use the origin
            atomicCAS(err, 0, (int)kDevBounds);
            c = o;
        }
        const Vec8 lo = load32(&pt[c].q[0]), hi = load32(&pt[c].q[2]);
        const float4 c0 = lo.a, c1 = lo.b, c2 = hi.a;
        const float wc = hi.b.x;
        const float pc[6] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y};
        const float vc[6] = {c1.z, c1.w, c2.x, c2.y, c2.z, c2.w};
        const float vo[6] = {o1.z, o1.w, o2.x, o2.y, o2.z, o2.w};
        float pp[6], vp[6];
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            pp[d] = __shfl_up_sync(full, pc[d], 1, 16);
            vp[d] = __shfl_up_sync(full, vc[d], 1, 16);
        }
        const float wp = __shfl_up_sync(full, wc, 1, 16);
        if (sl == 0 || j >= n) continue;
        float e[3], db[3], dp[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            e[d] = (pc[d] - pp[d]) + (pc[3 + d] - pp[3 + d]);
            db[d] = (vc[d] - vo[d]) + (vc[3 + d] - vo[3 + d]);
            dp[d] = (vc[d] - vp[d]) + (vc[3 + d] - vp[3 + d]);
        }
        const float dxs = sqrtf(fmaf(e[2], e[2], fmaf(e[1], e[1], e[0] * e[0]))) * inv_Lunit;
        const float beta = fmaf(dir.z, db[2], fmaf(dir.y, db[1], dir.x * db[0]));
        const float dbeta = fmaf(dir.z, dp[2], fmaf(dir.y, dp[1], dir.x * dp[0]));
        const float wbar = width_mode == 0 ? sqrtf(0.5f * (wc * wc + wp * wp)) : 0.5f * (wc + wp);
        steps[base + j] = make_int4(c, __float_as_int(dxs), __float_as_int(beta), __float_as_int(dbeta / wbar));
    }
}

// Double-precision step geometry for the FP64 formal solution, from the
// traced point lists (one thread per half-ray).
__global__ void k_steps64(int64_t N, int32_t R, const int64_t *__restrict__ off, const Step32 *__restrict__ s32,
                          const double *__restrict__ pos, const double *__restrict__ vel,
                          const double *__restrict__ w64, const double *__restrict__ dirs,
                          const int32_t *__restrict__ dir_map, double inv_Lunit, int width_mode,
                          Step64 *__restrict__ s64)
{
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)R * N) return;
    int r = (int)(t / N);
    int64_t o = t - (int64_t)r * N;
    const int rg = dir_map ? dir_map[r] : r;
    double n0 = dirs[3 * rg], n1 = dirs[3 * rg + 1], n2 = dirs[3 * rg + 2];
    const double vox = vel[3 * o], voy = vel[3 * o + 1], voz = vel[3 * o + 2];
    double px = pos[3 * o], py = pos[3 * o + 1], pz = pos[3 * o + 2];
    double pvx = vox, pvy = voy, pvz = voz, pw = w64[o];
    for (int64_t s = off[t]; s < off[t + 1]; ++s) {
        int64_t c = s32[s].x;
        double qx = pos[3 * c], qy = pos[3 * c + 1], qz = pos[3 * c + 2];
        double vx = vel[3 * c], vy = vel[3 * c + 1], vz = vel[3 * c + 2], wq = w64[c];
        double ex = qx - px, ey = qy - py, ez = qz - pz;
        Step64 st;
        st.dx = sqrt(ex * ex + ey * ey + ez * ez) * inv_Lunit;
        st.beta = (n0 * (vx - vox) + n1 * (vy - voy) + n2 * (vz - voz)) / kC;
        double dbeta = (n0 * (vx - pvx) + n1 * (vy - pvy) + n2 * (vz - pvz)) / kC;
        double wbar = width_mode == 0 ? sqrt(0.5 * (wq * wq + pw * pw)) : 0.5 * (wq + pw);
        st.dbw = dbeta / wbar;
        st.iw = 1.0 / wbar;
        s64[s] = st;
        px = qx; py = qy; pz = qz;
        pvx = vx; pvy = vy; pvz = vz; pw = wq;
    }
}

mgt_status trace_all(mgt_model *m, cudaStream_t s) { return trace_range(m, s, 0, m->P); }

// Trace the rays of pairs [p0, p0 + np).  All pairs: walk direction = model
// direction, ray offsets direction-major over all R directions.  A batch:
// walk directions 2i and 2i+1 are the two directions of pair p0 + i (see
// d_dir_map, d_batch_pairs), ray offsets over the batch's 2 np directions.
mgt_status trace_range(mgt_model *m, cudaStream_t s, int32_t p0, int32_t np)
{
    const bool all = p0 == 0 && np == m->P;
    const int32_t Rw = all ? m->R : 2 * np;
    if (!all) {
        std::vector<int32_t> map(2 * np);
        std::vector<int2> bp(np);
        for (int32_t i = 0; i < np; ++i) {
            map[2 * i] = m->pairs[2 * (p0 + i)];
            map[2 * i + 1] = m->pairs[2 * (p0 + i) + 1];
            bp[i] = make_int2(2 * i, 2 * i + 1);
        }
        MGT_CUDA(cudaMemcpyAsync(m->d_dir_map, map.data(), sizeof(int32_t) * map.size(), cudaMemcpyHostToDevice, s));
        MGT_CUDA(cudaMemcpyAsync(m->d_batch_pairs, bp.data(), sizeof(int2) * bp.size(), cudaMemcpyHostToDevice, s));
        MGT_CUDA(cudaStreamSynchronize(s));
    }
    const int64_t W = (int64_t)Rw * m->N;
    WalkArgs a{m->N,        Rw,            m->d_pos,  m->d_nbr_off, m->d_nbrs,   m->d_nbr_pos,
               m->pos_scale, m->d_bnd,     m->d_dirs, m->d_ent,     m->d_ent_row, m->d_pos_hl,
               m->d_dirs32,  m->d_order,   m->pos_slack, m->d_count + 2, m->n_chunks, all ? nullptr : m->d_dir_map};
    if (!m->d_ray_off) MGT_CUDA(cudaMalloc(&m->d_ray_off, sizeof(int64_t) * ((int64_t)m->R * m->N + 1)));
    // Scratch slot per walk: K point indices, a multiple of 16; the longest
    // half-ray of this model's previous trace when there was one, else four
    // times 4 N^(1/3) + 16 (a few times the mean half-ray of a cloud of N
    // points, so that a first trace rarely redoes a walk: 16 bytes per step of
    // the usual longest), kept within a third of the free device memory
    // (counting what the scratch pool holds unused).  Longer walks are redone.
    int64_t K = m->max_half > 0 ? (m->max_half + 15) / 16 * 16
                                : 4 * (((int64_t)(4.0 * std::cbrt((double)m->N)) + 16 + 15) / 16 * 16);
    cudaMemPool_t pool = nullptr;
    MGT_TRY_STATUS(scratch_pool(&pool));
    {
        size_t freeb = 0, totalb = 0;
        MGT_CUDA(cudaMemGetInfo(&freeb, &totalb));
        uint64_t reserved = 0, used = 0;
        MGT_CUDA(cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved));
        MGT_CUDA(cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used));
        freeb += reserved > used ? (size_t)(reserved - used) : 0;
        while (K > 16 && (size_t)(W * K) * sizeof(int32_t) > freeb / 3) K -= 16;
    }
    int64_t *d_len = nullptr, *d_list = nullptr, *d_max = nullptr;
    int32_t *d_scratch = nullptr;
    WalkPoint *d_pt = nullptr;
    unsigned long long *d_nover = nullptr;
    void *tmp = nullptr, *tmpb = nullptr;
    auto release = [&]() {
        if (tmp) cudaFreeAsync(tmp, s);
        if (tmpb) cudaFreeAsync(tmpb, s);
        if (d_max) cudaFreeAsync(d_max, s);
        if (d_len) cudaFreeAsync(d_len, s);
        if (d_list) cudaFreeAsync(d_list, s);
        if (d_nover) cudaFreeAsync(d_nover, s);
        if (d_scratch) cudaFreeAsync(d_scratch, s);
        if (d_pt) cudaFreeAsync(d_pt, s);
    };
    struct Guard {
        decltype(release) &f;
        ~Guard() { f(); }
    } guard{release};
    MGT_CUDA(cudaMallocFromPoolAsync(&d_len, sizeof(int64_t) * (W + 1), pool, s));
    MGT_CUDA(cudaMallocFromPoolAsync(&d_list, sizeof(int64_t) * W, pool, s));
    MGT_CUDA(cudaMallocFromPoolAsync(&d_nover, sizeof(unsigned long long), pool, s));
    MGT_CUDA(cudaMallocFromPoolAsync(&d_pt, sizeof(WalkPoint) * m->N, pool, s));
    if (cudaMallocFromPoolAsync(&d_scratch, sizeof(int32_t) * W * K, pool, s) != cudaSuccess) {
        cudaGetLastError();
        d_scratch = nullptr;
        return set_error(MGT_ERR_OOM, "cannot allocate the walk scratch");
    }
    MGT_CUDA(cudaMemsetAsync(m->d_count + 1, 0, 2 * sizeof(unsigned long long), s));
    MGT_CUDA(cudaMemsetAsync(d_nover, 0, sizeof(unsigned long long), s));
    const float inv_Lunit = (float)(1.0 / (m->pos_scale * m->L_unit));
    {
        MGT_KTIMER("k_walk<fused>", s);
        MGT_TRY_STATUS(launch_walk<kWalkFused>(a, W, d_len, nullptr, nullptr, (int32_t)K, m->d_count + 1, d_scratch,
                                               nullptr, m->d_err, ImgWalkArgs{}, s));
    }
    MGT_CUDA(cudaMemsetAsync(d_len + W, 0, sizeof(int64_t), s));
    size_t tmp_bytes = 0;
    MGT_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tmp_bytes, d_len, m->d_ray_off, W + 1, s));
    MGT_CUDA(cudaMallocFromPoolAsync(&tmp, tmp_bytes, pool, s));
    MGT_CUDA(cub::DeviceScan::ExclusiveSum(tmp, tmp_bytes, d_len, m->d_ray_off, W + 1, s));
    // longest half-ray
    MGT_CUDA(cudaMallocFromPoolAsync(&d_max, sizeof(int64_t), pool, s));
    size_t tmp2 = 0;
    MGT_CUDA(cub::DeviceReduce::Max(nullptr, tmp2, d_len, d_max, W, s));
    MGT_CUDA(cudaMallocFromPoolAsync(&tmpb, tmp2, pool, s));
    MGT_CUDA(cub::DeviceReduce::Max(tmpb, tmp2, d_len, d_max, W, s));
    k_walk_overflow<<<ceil_div(W, 256), 256, 0, s>>>(W, d_len, (int32_t)K, d_list, d_nover);
    MGT_LAUNCH_CHECK("k_walk_overflow");
    int64_t total = 0, mx = 0;
    unsigned long long stalls = 0, exact_steps = 0, n_over = 0;
    MGT_CUDA(cudaMemcpyAsync(&total, m->d_ray_off + W, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    MGT_CUDA(cudaMemcpyAsync(&mx, d_max, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    MGT_CUDA(cudaMemcpyAsync(&stalls, m->d_count + 1, sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
    MGT_CUDA(cudaMemcpyAsync(&exact_steps, m->d_count + 2, sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
    MGT_CUDA(cudaMemcpyAsync(&n_over, d_nover, sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
    MGT_CUDA(cudaStreamSynchronize(s));
    MGT_TRY_STATUS(check_device_error(m, s));     // a walk that gave up leaves the lengths unusable
    // the ray buffer comes from the same pool: a model created after another
    // one was destroyed reuses its mapping.  A formal solution on another
    // stream may still read the old buffer, hence the device-wide wait.
    if (m->d_steps32 && total > m->steps32_cap) {
        MGT_CUDA(cudaDeviceSynchronize());
        MGT_CUDA(cudaFreeAsync(m->d_steps32, s));
        m->d_steps32 = nullptr;
    }
    m->steps64_width_mode = -1;                // the FP64 geometry describes the previous rays
    if (!m->d_steps32 && total > 0) {
        cudaError_t e = cudaMallocFromPoolAsync(&m->d_steps32, sizeof(Step32) * total, pool, s);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return set_error(MGT_ERR_OOM, "cannot allocate the ray buffer");
        }
        m->steps32_cap = total;
    }
    m->total_steps = total;
    m->max_half = (int32_t)mx;
    m->n_stalls = (int64_t)stalls;
    m->n_exact_steps = (int64_t)exact_steps;   // the walks of the fused pass
    if (total > 0) {
        {
            // each index read once from its slot and each record written once, plus the offsets
            MGT_KTIMER_BYTES("k_walk_compact", s, 20.0 * (double)total + 8.0 * (double)W);
            k_walk_points<<<ceil_div(m->N, 256), 256, 0, s>>>(m->N, m->d_pos_hl, m->d_vel_hl, m->d_w32, d_pt);
            k_walk_compact<false><<<ceil_div(W * 16, 256), 256, 0, s>>>(a, W, m->d_ray_off, nullptr, (int32_t)K, d_scratch,
                                                                    d_pt, inv_Lunit, m->opts.width_mode, m->d_steps32,
                                                                    m->d_err);
        }
        MGT_LAUNCH_CHECK("k_walk_compact");
        note_launch();                             // k_walk_points
        if (n_over > 0) {
            {
                MGT_KTIMER("k_walk<list>", s);
                MGT_TRY_STATUS(launch_walk<kWalkList>(a, (int64_t)n_over, nullptr, m->d_ray_off, d_list, 0, nullptr,
                                                      nullptr, m->d_steps32, m->d_err, ImgWalkArgs{}, s));
                k_walk_compact<true><<<ceil_div((int64_t)n_over * 16, 256), 256, 0, s>>>(
                    a, (int64_t)n_over, m->d_ray_off, d_list, 0, nullptr, d_pt, inv_Lunit, m->opts.width_mode,
                    m->d_steps32, m->d_err);
            }
            MGT_LAUNCH_CHECK("k_walk_compact<list>");
        }
    }
    m->steps_width_mode = m->opts.width_mode;
    m->rays_p0 = p0;
    m->rays_np = np;
    m->traced = true;
    return MGT_OK;
}

mgt_status build_steps64(mgt_model *m, cudaStream_t s)
{
    if (m->total_steps == 0) return MGT_OK;
    if (m->d_steps64 && m->steps64_cap < m->total_steps) {
        MGT_CUDA(cudaFree(m->d_steps64));
        m->d_steps64 = nullptr;
    }
    if (!m->d_steps64) {
        m->steps64_cap = m->total_steps;
        cudaError_t e = cudaMalloc(&m->d_steps64, sizeof(Step64) * m->total_steps);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return set_error(MGT_ERR_OOM, "cannot allocate the FP64 ray geometry");
        }
    }
    const bool all = m->rays_p0 == 0 && m->rays_np == m->P;
    const int32_t Rw = all ? m->R : 2 * m->rays_np;
    const int64_t W = (int64_t)Rw * m->N;
    k_steps64<<<ceil_div(W, 128), 128, 0, s>>>(m->N, Rw, m->d_ray_off, m->d_steps32, m->d_pos, m->d_vel,
                                               m->d_w64, m->d_dirs, all ? nullptr : m->d_dir_map, 1.0 / m->L_unit,
                                               m->opts.width_mode, m->d_steps64);
    MGT_LAUNCH_CHECK("k_steps64");
    m->steps64_width_mode = m->opts.width_mode;
    return MGT_OK;
}

}  // namespace mgt

namespace mgt {

// ---------------------------------------------------------------------------
// Synthetic image geometry (Listing 3, compute_image_new).  The paper gives
// no algorithm; the image plane, the pixel reference points, the anchor of a
// pixel (the point closest to the pixel line) and the two walks from it follow
// the definition written out in the model-independent form below, in FP64
// with every operation in the order written and no multiply-add contraction.
// ---------------------------------------------------------------------------

// The image plane: basis, and what k_img_plane derives from the projections.
struct ImgPlane {
    double e1[3], e2[3];
    unsigned long long range[4];   // projections' lo1, lo2, hi1, hi2 as ordered integers
    double first1, first2;         // centre minus half-width
    double step1, step2;           // pixel spacings
    double cell, inv_cell;         // the search grid: [first, first + grid cell] on both axes
};

constexpr int kImgThreads = 256;

// Projections (s1, s2) of every point and their range.
__global__ void __launch_bounds__(kImgThreads) k_img_project(int64_t N, const double *__restrict__ pos, ImgPlane *pl,
                                                             double2 *__restrict__ s12)
{
    __shared__ unsigned long long red[4];
    if (threadIdx.x < 4) red[threadIdx.x] = threadIdx.x < 2 ? ~0ull : 0ull;
    __syncthreads();
    unsigned long long v[4] = {~0ull, ~0ull, 0ull, 0ull};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        const double x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2];
        const double s1 = dot3_exact(x, y, z, pl->e1[0], pl->e1[1], pl->e1[2]);
        const double s2 = dot3_exact(x, y, z, pl->e2[0], pl->e2[1], pl->e2[2]);
        s12[i] = make_double2(s1, s2);
        const unsigned long long k1 = order_key(s1), k2 = order_key(s2);
        v[0] = min(v[0], k1);
        v[1] = min(v[1], k2);
        v[2] = max(v[2], k1);
        v[3] = max(v[3], k2);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long w = __shfl_xor_sync(0xffffffffu, v[k], o);
            v[k] = k < 2 ? min(v[k], w) : max(v[k], w);
        }
        if ((threadIdx.x & 31) == 0) k < 2 ? atomicMin(&red[k], v[k]) : atomicMax(&red[k], v[k]);
    }
    __syncthreads();
    if (threadIdx.x < 4)
        threadIdx.x < 2 ? atomicMin(&pl->range[threadIdx.x], red[threadIdx.x])
                        : atomicMax(&pl->range[threadIdx.x], red[threadIdx.x]);
}

// Centre, half-width, pixel spacings and search grid (one thread).
__global__ void k_img_plane(ImgPlane *pl, int32_t npx, int32_t npy, int grid)
{
    const double lo1 = order_value(pl->range[0]), lo2 = order_value(pl->range[1]);
    const double hi1 = order_value(pl->range[2]), hi2 = order_value(pl->range[3]);
    const double c1 = __dmul_rn(0.5, __dadd_rn(lo1, hi1)), c2 = __dmul_rn(0.5, __dadd_rn(lo2, hi2));
    const double w1 = __dsub_rn(hi1, lo1), w2 = __dsub_rn(hi2, lo2);
    const double H = __dmul_rn(0.5, w1 > w2 ? w1 : w2);
    pl->first1 = __dsub_rn(c1, H);
    pl->first2 = __dsub_rn(c2, H);
    pl->step1 = __ddiv_rn(__dmul_rn(2.0, H), (double)npx);
    pl->step2 = __ddiv_rn(__dmul_rn(2.0, H), (double)npy);
    // (all projections in one place: one cell holds everything)
    pl->cell = H > 0.0 ? 2.0 * H / grid : 1e300;
    pl->inv_cell = H > 0.0 ? grid / (2.0 * H) : 0.0;
}

// Reference point of each pixel.
__global__ void k_img_ref(const ImgPlane *__restrict__ pl, int32_t npx, int64_t npix, double *__restrict__ ref)
{
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= npix) return;
    const int64_t j = q / npx, i = q - j * npx;
    const double t1 = __dadd_rn(pl->first1, __dmul_rn((double)i + 0.5, pl->step1));
    const double t2 = __dadd_rn(pl->first2, __dmul_rn((double)j + 0.5, pl->step2));
    for (int k = 0; k < 3; ++k) ref[3 * q + k] = __dadd_rn(__dmul_rn(t1, pl->e1[k]), __dmul_rn(t2, pl->e2[k]));
}

// Search grid over the image plane: cell of each point, points per cell, and
// the points in cell order with what the anchor search reads of them (32 bytes:
// position times pos_scale as float hi + lo, index).
__device__ __forceinline__ int img_cell(double s, double first, const ImgPlane &pl, int grid)
{
    return min(max((int)((s - first) * pl.inv_cell), 0), grid - 1);
}

__global__ void k_img_cells(int64_t N, const double2 *__restrict__ s12, const ImgPlane *__restrict__ pl, int grid,
                            int32_t *__restrict__ count)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double2 v = s12[i];
    atomicAdd(&count[(int64_t)img_cell(v.y, pl->first2, *pl, grid) * grid + img_cell(v.x, pl->first1, *pl, grid)], 1);
}

__global__ void k_img_sort(int64_t N, const double2 *__restrict__ s12, const ImgPlane *__restrict__ pl, int grid,
                           const int32_t *__restrict__ start, int32_t *__restrict__ left,
                           const float *__restrict__ pos_hl, float4 *__restrict__ out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double2 v = s12[i];
    const int64_t c = (int64_t)img_cell(v.y, pl->first2, *pl, grid) * grid + img_cell(v.x, pl->first1, *pl, grid);
    const int64_t at = start[c] + atomicSub(&left[c], 1) - 1;
    const float *h = pos_hl + 6 * i;
    out[2 * at] = make_float4(h[0], h[1], h[2], h[3]);
    out[2 * at + 1] = make_float4(h[4], h[5], __int_as_float((int)i), 0.0f);
}

// Anchor of each pixel: the point whose squared distance to the pixel line
// |(x - p) - ((x - p).n) n|^2 is smallest, ties to the smaller index.  One
// warp per pixel looks at the points in a window of grid cells around the
// pixel: FP32 distances from hi + lo positions with the error bounds ep and e2
// of the walk (its offsets' 2s holds here too: the reference point's scaled
// coordinates are at most 3.1, so hi + lo leaves 4.1 2^-48 out of an offset and
// its low parts round by as much, 3.6 s in all over the three components), an
// FP64 scan of the window (the defining expressions) when the bounds do not
// separate the winner from every other point.  The window grows until every
// point within the winner's upper bound (plus a margin for the projections)
// lies inside it, so no point outside can win or tie.  The margin: a direction
// may be 5e-13 from unit length, e2 = n x e1 with it, and then a pixel lies up to
// 2 x 5e-13 x 2.6 beside its place among the projections (in units of the
// scaled positions).
//
// Every pixel against every point took 5.3 ms for 16,384 pixels and 100k
// points (issue bound, 1.6e9 distances); the grid holds two points per cell on
// average, and a pixel looks at some hundred: a view of 128 x 128 pixels with 32
// channels, new rays and image, went from 6.6 to 0.85 ms.
__global__ void __launch_bounds__(kImgThreads) k_img_anchor(WalkArgs a, const ImgPlane *__restrict__ plane, int grid,
                                                            const int32_t *__restrict__ start,
                                                            const float4 *__restrict__ pts,
                                                            const double *__restrict__ ref, int32_t npx, int64_t npix,
                                                            double n0, double n1, double n2,
                                                            int32_t *__restrict__ anchor)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (q >= npix) return;                                     // whole warp
    const ImgPlane &pl = *plane;
    const double *pr = ref + 3 * q;
    const double sx = pr[0] * a.pos_scale, sy = pr[1] * a.pos_scale, sz = pr[2] * a.pos_scale;
    const float ohx = (float)sx, ohy = (float)sy, ohz = (float)sz;
    const float olx = (float)(sx - (double)ohx), oly = (float)(sy - (double)ohy), olz = (float)(sz - (double)ohz);
    const float f0 = (float)n0, f1 = (float)n1, f2 = (float)n2;
    const int64_t jy = q / npx;
    const double t1 = pl.first1 + ((double)(q - jy * npx) + 0.5) * pl.step1,
                 t2 = pl.first2 + ((double)jy + 0.5) * pl.step2;
    const int cx = img_cell(t1, pl.first1, pl, grid), cy = img_cell(t2, pl.first2, pl, grid);
    const double inv_scale = 1.0 / a.pos_scale;
    const double margin = 1e-11 * inv_scale;       // (far above the rounding of projections and cell edges)
    float bd2, bU, bL, minLo;
    int bi, best = -1;
    // every point of the window, 32 at a time: rows of cells are contiguous
    // runs, 32 rows' runs at a time share the lanes
    auto scan = [&](int x0, int x1, int y0, int y1, auto &&point) {
        for (int yb = y0; yb <= y1; yb += 32) {
            const int y = yb + lane;
            int s = 0, len = 0;
            if (y <= y1) {
                s = start[(int64_t)y * grid + x0];
                len = start[(int64_t)y * grid + x1 + 1] - s;
            }
            int incl = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(full, incl, o);
                if (lane >= o) incl += v;
            }
            const int total = __shfl_sync(full, incl, 31), base = s - (incl - len);
            for (int i0 = 0; i0 < total; i0 += 32) {
                const int i = i0 + lane;
                int r = 0;                          // the row whose run holds item i
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    if (__shfl_sync(full, incl, r + o - 1) <= i) r += o;
                const int at = __shfl_sync(full, base, r & 31) + i;
                if (i < total) point((int64_t)at);
            }
        }
    };
    int x0 = 0, x1 = 0, y0 = 0, y1 = 0;
    for (int k = 1;;) {
        x0 = max(cx - k, 0);
        x1 = min(cx + k, grid - 1);
        y0 = max(cy - k, 0);
        y1 = min(cy + k, grid - 1);
        bd2 = bU = bL = minLo = 3.0e38f;
        bi = 0x7fffffff;
        scan(x0, x1, y0, y1, [&](int64_t at) {
            const Vec8 h = load32(pts + 2 * at);
            const int i = __float_as_int(h.b.z);
            const float dx = (h.a.x - ohx) + (h.a.w - olx), dy = (h.a.y - ohy) + (h.b.x - oly),
                        dz = (h.a.z - ohz) + (h.b.y - olz);
            const float S = fabsf(dx) + fabsf(dy) + fabsf(dz);
            const float Z = fmaf(dz, f2, fmaf(dy, f1, dx * f0));
            const float px = fmaf(-Z, f0, dx), py = fmaf(-Z, f1, dy), pz = fmaf(-Z, f2, dz);
            const float d2 = fmaf(pz, pz, fmaf(py, py, px * px));
            const float ep = fmaf(8e-7f, S, 8.0f * a.pos_slack);
            const float e2 = fmaf(ep, fmaf(2.5f, sqrtf(d2), ep), 4e-7f * d2);
            if (d2 < bd2) {
                minLo = fminf(minLo, bL);
                bd2 = d2;
                bU = d2 + e2;
                bL = d2 - e2;
                bi = i;
            } else {
                minLo = fminf(minLo, d2 - e2);
            }
        });
        // warp winner: smallest d2, then smallest index
        float wd2 = bd2;
        int wi = bi;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float od = __shfl_xor_sync(full, wd2, o);
            const int oi = __shfl_xor_sync(full, wi, o);
            if (od < wd2 || (od == wd2 && oi < wi)) {
                wd2 = od;
                wi = oi;
            }
        }
        const bool mine = bi == wi;
        minLo = fminf(minLo, mine ? 3.0e38f : bL);
        bU = mine ? bU : 3.0e38f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            minLo = fminf(minLo, __shfl_xor_sync(full, minLo, o));
            bU = fminf(bU, __shfl_xor_sync(full, bU, o));
        }
        best = wi;
        if (x0 == 0 && y0 == 0 && x1 == grid - 1 && y1 == grid - 1) break;     // every point was looked at
        if (wd2 >= 3.0e38f) {                                                  // an empty window
            k *= 2;
            continue;
        }
        // distance to the nearest side of the window that is not the grid's own
        double reach = 1e300;
        if (x0 > 0) reach = fmin(reach, t1 - (pl.first1 + x0 * pl.cell));
        if (x1 < grid - 1) reach = fmin(reach, pl.first1 + (x1 + 1) * pl.cell - t1);
        if (y0 > 0) reach = fmin(reach, t2 - (pl.first2 + y0 * pl.cell));
        if (y1 < grid - 1) reach = fmin(reach, pl.first2 + (y1 + 1) * pl.cell - t2);
        const double need = (double)sqrtf(bU) * 1.0001 * inv_scale + margin;
        if (need <= reach) break;
        k = max(k + 1, (int)fmin(need * pl.inv_cell + 2.0, 1e9));
    }
    if (!(bU < minLo)) {
        // FP64, the defining expressions
        double ed2 = 0.0;
        int ei = 0x7fffffff;
        scan(x0, x1, y0, y1, [&](int64_t at) {
            const int i = __float_as_int(pts[2 * at + 1].z);
            const double *x = a.pos + 3 * (int64_t)i;
            const double dx = __dsub_rn(x[0], pr[0]), dy = __dsub_rn(x[1], pr[1]), dz = __dsub_rn(x[2], pr[2]);
            const double Z = dot3_exact(dx, dy, dz, n0, n1, n2);
            const double px = __dsub_rn(dx, __dmul_rn(Z, n0)), py = __dsub_rn(dy, __dmul_rn(Z, n1)),
                         pz = __dsub_rn(dz, __dmul_rn(Z, n2));
            const double d2 = dot3_exact(px, py, pz, px, py, pz);
            if (ei == 0x7fffffff || d2 < ed2 || (d2 == ed2 && i < ei)) {
                ed2 = d2;
                ei = i;
            }
        });
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double od = __shfl_xor_sync(full, ed2, o);
            const int oi = __shfl_xor_sync(full, ei, o);
            if (oi != 0x7fffffff && (ei == 0x7fffffff || od < ed2 || (od == ed2 && oi < ei))) {
                ed2 = od;
                ei = oi;
            }
        }
        best = ei;
    }
    if (lane == 0) anchor[q] = best;
}

// Full-ray sizes (far half, anchor, near half; entry npix: zero), the longest
// full ray and the longest half-ray.
__global__ void __launch_bounds__(kImgThreads) k_img_sizes(int64_t npix, const int64_t *__restrict__ lens,
                                                           int64_t *__restrict__ sizes, int *__restrict__ longest)
{
    __shared__ int red[2];
    if (threadIdx.x < 2) red[threadIdx.x] = 0;
    __syncthreads();
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q < npix) {
        const int64_t a = lens[2 * q], b = lens[2 * q + 1];
        sizes[q] = a + b + 1;
        atomicMax(&red[0], (int)(a + b + 1));
        atomicMax(&red[1], (int)max(a, b));
    } else if (q == npix) {
        sizes[q] = 0;
    }
    __syncthreads();
    if (threadIdx.x < 2 && red[threadIdx.x] > 0) atomicMax(&longest[threadIdx.x], red[threadIdx.x]);
}

// Full rays from the scratch slots, one warp per pixel: the far half reversed,
// the anchor, the near half.
__global__ void __launch_bounds__(kImgThreads) k_img_place(int64_t npix, const int64_t *__restrict__ lens,
                                                           const int64_t *__restrict__ off,
                                                           const int32_t *__restrict__ anchor, int32_t K,
                                                           const int32_t *__restrict__ scratch,
                                                           int32_t *__restrict__ pts)
{
    const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (q >= npix) return;
    const int nf = (int)lens[2 * q], nn = (int)lens[2 * q + 1];
    const int64_t b = off[q];
    if (lane == 0) pts[b + nf] = anchor[q];
    const int32_t *far = scratch + 2 * q * K, *near = far + K;
    if (nf <= K)
        for (int j = lane; j < nf; j += 32) pts[b + nf - 1 - j] = far[j];
    if (nn <= K)
        for (int j = lane; j < nn; j += 32) pts[b + nf + 1 + j] = near[j];
}

// Give the geometry's buffers back to the pool on stream s.  The caller has
// made sure that no other stream still reads them.
static void image_release(ImageGeom &g, cudaStream_t s)
{
    for (void *p : {(void *)g.d_ref, (void *)g.d_anchor, (void *)g.d_off, (void *)g.d_pts})
        if (p) cudaFreeAsync(p, s);
    g = ImageGeom{};
}

// Rays kept from a view four times as large, in buffers that do not go back to
// the library's pool: a new view gets its own.
static bool image_oversized(const ImageGeom &g, int64_t npix)
{
    const int64_t bytes = std::max<int64_t>(24 * g.npix_cap, 4 * g.pts_cap);
    return g.npix_cap > 4 * npix && bytes > (int64_t)kPooledBytes;
}

void image_free(mgt_model *m)          // the device is idle
{
    if (!m->img.d_ref) return;
    image_release(m->img, nullptr);
    cudaStreamSynchronize(nullptr);
}

mgt_status trace_image(mgt_model *m, const double n[3], int32_t npx, int32_t npy, cudaStream_t s)
{
    ImageGeom &g = m->img;
    if (g.valid && g.npx == npx && g.npy == npy && g.n[0] == n[0] && g.n[1] == n[1] && g.n[2] == n[2]) {
        if (s != g.stream || s == cudaStreamPerThread) g.shared = true;
        return MGT_OK;
    }
    // the old rays may still be read on another stream
    if (g.d_ref && (g.shared || s != g.stream || s == cudaStreamPerThread)) MGT_CUDA(cudaDeviceSynchronize());
    g.valid = false;
    g.shared = false;
    g.stream = s;
    const int64_t npix = (int64_t)npx * npy, N = m->N;
    std::vector<void *> tmp;               // this call's temporaries
    struct Guard {
        std::vector<void *> &v;
        cudaStream_t s;
        ~Guard()
        {
            for (void *p : v) cudaFreeAsync(p, s);
        }
    } guard{tmp, s};
    auto temp = [&](auto **p, int64_t count) -> mgt_status {
        const mgt_status st = buffer_alloc(p, count, s);
        if (st == MGT_OK) tmp.push_back((void *)*p);
        return st;
    };
    if (npix > g.npix_cap || image_oversized(g, npix)) {
        image_release(g, s);
        g.stream = s;
        MGT_TRY_STATUS(buffer_alloc(&g.d_ref, 3 * npix, s));
        MGT_TRY_STATUS(buffer_alloc(&g.d_anchor, npix, s));
        MGT_TRY_STATUS(buffer_alloc(&g.d_off, npix + 1, s));
        g.npix_cap = npix;
    }
    // the image plane's basis: e1 = unit(a x n), a the coordinate axis least
    // aligned with n (lowest index on ties), e2 = n x e1
    ImgPlane pl{};
    {
        int ax = 0;
        for (int k = 1; k < 3; ++k)
            if (std::fabs(n[k]) < std::fabs(n[ax])) ax = k;
        double av[3] = {0.0, 0.0, 0.0};
        av[ax] = 1.0;
        const double c[3] = {av[1] * n[2] - av[2] * n[1], av[2] * n[0] - av[0] * n[2], av[0] * n[1] - av[1] * n[0]};
        const double cl = std::sqrt(c[0] * c[0] + c[1] * c[1] + c[2] * c[2]);
        for (int k = 0; k < 3; ++k) pl.e1[k] = c[k] / cl;
        pl.e2[0] = n[1] * pl.e1[2] - n[2] * pl.e1[1];
        pl.e2[1] = n[2] * pl.e1[0] - n[0] * pl.e1[2];
        pl.e2[2] = n[0] * pl.e1[1] - n[1] * pl.e1[0];
        pl.range[0] = pl.range[1] = ~0ull;
    }
    // search grid: two points per cell on average
    const int grid = (int)std::min(2048.0, std::max(1.0, std::ceil(std::sqrt(0.5 * (double)N))));
    const int64_t cells = (int64_t)grid * grid;
    // scratch slot per half-ray, as in trace_range, at most 1 GB in all: above
    // 8.4 million pixels none, and every ray is walked again into its place
    const int64_t usual = ((int64_t)(8.0 * std::cbrt((double)N)) + 16 + 15) / 16 * 16;
    const int32_t K = (int32_t)std::min(usual, ((int64_t)1 << 30) / (8 * npix) / 16 * 16);
    ImgPlane *d_pl = nullptr;
    double2 *d_s12 = nullptr;
    int32_t *d_count = nullptr, *d_start = nullptr, *d_scratch = nullptr;
    float4 *d_sorted = nullptr;
    int64_t *d_lens = nullptr, *d_sizes = nullptr;
    int *d_longest = nullptr;
    unsigned char *d_cub = nullptr;
    size_t cub1 = 0, cub2 = 0;
    MGT_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, cub1, d_count, d_start, (int)(cells + 1), s));
    MGT_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, cub2, d_sizes, g.d_off, npix + 1, s));
    MGT_TRY_STATUS(temp(&d_pl, 1));
    MGT_TRY_STATUS(temp(&d_s12, N));
    MGT_TRY_STATUS(temp(&d_count, cells + 1));
    MGT_TRY_STATUS(temp(&d_start, cells + 1));
    MGT_TRY_STATUS(temp(&d_sorted, 2 * N));
    MGT_TRY_STATUS(temp(&d_scratch, 2 * npix * K));
    MGT_TRY_STATUS(temp(&d_lens, 2 * npix));
    MGT_TRY_STATUS(temp(&d_sizes, npix + 1));
    MGT_TRY_STATUS(temp(&d_longest, 2));
    MGT_TRY_STATUS(temp(&d_cub, std::max<size_t>(std::max(cub1, cub2), 1)));
    MGT_CUDA(cudaMemcpyAsync(d_pl, &pl, sizeof pl, cudaMemcpyHostToDevice, s));
    MGT_CUDA(cudaMemsetAsync(d_count, 0, sizeof(int32_t) * (cells + 1), s));
    MGT_CUDA(cudaMemsetAsync(d_longest, 0, sizeof(int) * 2, s));
    k_img_project<<<(unsigned)std::min<int64_t>(ceil_div(N, kImgThreads), 304), kImgThreads, 0, s>>>(N, m->d_pos, d_pl,
                                                                                                     d_s12);
    MGT_LAUNCH_CHECK("k_img_project");
    k_img_plane<<<1, 1, 0, s>>>(d_pl, npx, npy, grid);
    MGT_LAUNCH_CHECK("k_img_plane");
    k_img_ref<<<ceil_div(npix, kImgThreads), kImgThreads, 0, s>>>(d_pl, npx, npix, g.d_ref);
    MGT_LAUNCH_CHECK("k_img_ref");
    k_img_cells<<<ceil_div(N, kImgThreads), kImgThreads, 0, s>>>(N, d_s12, d_pl, grid, d_count);
    MGT_LAUNCH_CHECK("k_img_cells");
    MGT_CUDA(cub::DeviceScan::ExclusiveSum(d_cub, cub1, d_count, d_start, (int)(cells + 1), s));
    k_img_sort<<<ceil_div(N, kImgThreads), kImgThreads, 0, s>>>(N, d_s12, d_pl, grid, d_start, d_count, m->d_pos_hl,
                                                                d_sorted);
    MGT_LAUNCH_CHECK("k_img_sort");
    WalkArgs a{m->N,        m->R,          m->d_pos,  m->d_nbr_off, m->d_nbrs,   m->d_nbr_pos,
               m->pos_scale, m->d_bnd,     m->d_dirs, m->d_ent,     m->d_ent_row, m->d_pos_hl,
               m->d_dirs32,  m->d_order,   m->pos_slack, m->d_count + 3, m->n_chunks, nullptr};
    k_img_anchor<<<ceil_div(npix * 32, kImgThreads), kImgThreads, 0, s>>>(a, d_pl, grid, d_start, d_sorted, g.d_ref, npx,
                                                                          npix, n[0], n[1], n[2], g.d_anchor);
    MGT_LAUNCH_CHECK("k_img_anchor");
    ImgWalkArgs im{g.d_ref, g.d_anchor, g.d_off, nullptr, npix, {n[0], n[1], n[2]}};
    MGT_TRY_STATUS(launch_walk<kWalkImg>(a, 2 * npix, d_lens, nullptr, nullptr, K, nullptr, d_scratch, nullptr, m->d_err,
                                         im, s));
    k_img_sizes<<<ceil_div(npix + 1, kImgThreads), kImgThreads, 0, s>>>(npix, d_lens, d_sizes, d_longest);
    MGT_LAUNCH_CHECK("k_img_sizes");
    MGT_CUDA(cub::DeviceScan::ExclusiveSum(d_cub, cub2, d_sizes, g.d_off, npix + 1, s));
    int64_t total = 0;
    int longest[2] = {0, 0};
    MGT_CUDA(cudaMemcpyAsync(&total, g.d_off + npix, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    MGT_CUDA(cudaMemcpyAsync(longest, d_longest, sizeof longest, cudaMemcpyDeviceToHost, s));
    MGT_TRY_STATUS(check_device_error(m, s));     // (synchronises) a walk that gave up leaves the lengths unusable
    if (total > g.pts_cap) {
        if (g.d_pts) MGT_CUDA(cudaFreeAsync(g.d_pts, s));
        g.d_pts = nullptr;
        g.pts_cap = 0;
        MGT_TRY_STATUS(buffer_alloc(&g.d_pts, total, s));
        g.pts_cap = total;
    }
    k_img_place<<<ceil_div(npix * 32, kImgThreads), kImgThreads, 0, s>>>(npix, d_lens, g.d_off, g.d_anchor, K, d_scratch,
                                                                         g.d_pts);
    MGT_LAUNCH_CHECK("k_img_place");
    if (longest[1] > K) {
        im.pts = g.d_pts;
        MGT_TRY_STATUS(launch_walk<kWalkImgFill>(a, 2 * npix, d_lens, nullptr, nullptr, 0, nullptr, nullptr, nullptr,
                                                 m->d_err, im, s));
    }
    // complete before another stream may read it
    MGT_TRY_STATUS(check_device_error(m, s));
    g.total = total;
    g.max_len = longest[0];
    g.n[0] = n[0];
    g.n[1] = n[1];
    g.n[2] = n[2];
    g.npx = npx;
    g.npy = npy;
    g.valid = true;
    return MGT_OK;
}

}  // namespace mgt
