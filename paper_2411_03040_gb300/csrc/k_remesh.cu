// Recursive re-meshing of a point cloud (Sec. 4.1): divide a box into 8 equal
// parts while the variation 2 (rho_max - rho_min)/(rho_max + rho_min) of the
// tracer inside it exceeds r_max and the recursion level is below l, crop
// each non-empty part to the bounding box of its points, and represent every
// final box by its centre; then add evenly spaced boundary points on the
// surface of the outermost box.
//
// GPU form: the recursion runs level by level.  The points themselves (position
// and tracer, 32 bytes) are kept in box order, so that every box is one
// contiguous segment; per level every open box's bounds and tracer range are
// reduced (exact in any order), the boxes that divide count their points per
// octant and move them into the children's segments, and the children
// (non-empty octants, in parent order then octant order) are the next level's
// boxes.  Final boxes are written level by level in box order.
//
// The passes over points run on units of at most kRmUnit consecutive points of
// one box, one warp per unit: the first levels (one box of every point) and the
// last ones (10^5 boxes of a few points) both fill the GPU.  With one block per
// box the first levels of a 1M-point cloud ran on 1, 8 and 64 blocks: 47 ms of
// kernels per call, now below 2 ms (12 levels; host to host 100.0 -> 3.06 ms,
// the binding's second call for the count included in the 100.0).  A level's
// passes move about 130 bytes per point, mostly through L2, so what is left is
// launch latency and the copies.  Bounds are compared as integers that order
// like the doubles: this GPU's FP64 pipe takes 16 cycles per warp instruction.
#include <cub/cub.cuh>

#include <algorithm>
#include <cmath>
#include <vector>

#include "mgt_common.cuh"

namespace mgt {

namespace {

constexpr int kRmThreads = 256;
constexpr int kRmUnit = 512;          // points of one warp's unit of work

struct __align__(32) RmPoint {
    double x, y, z, rho;
};

__device__ __forceinline__ double no_negative_zero(double v) { return v == 0.0 ? 0.0 : v; }

__device__ __forceinline__ uint64_t ord_mid(double v) { return order_key(no_negative_zero(v)); }

// A box's bounds and tracer range as ordered integers: lo[3], hi[3], rmin, rmax.
struct RmBox {
    uint64_t v[8];
};

__device__ __forceinline__ void empty_box(RmBox &s)
{
#pragma unroll
    for (int k = 0; k < 8; ++k) s.v[k] = k < 3 || k == 6 ? ~0ull : 0ull;
}

// Per box of a level: how many leaves, children and children's units come
// from it; their exclusive scan places them.
struct RmCounts {
    uint32_t leaf, child, unit;
};

struct RmAdd {
    __host__ __device__ RmCounts operator()(const RmCounts &a, const RmCounts &b) const
    {
        return {a.leaf + b.leaf, a.child + b.child, a.unit + b.unit};
    }
};

__host__ __device__ inline int64_t rm_units(int64_t n) { return (n + kRmUnit - 1) / kRmUnit; }

// Units of a level: unit u covers kRmUnit points of box box[u] from its
// (u - first[box[u]])-th unit on.
struct RmUnits {
    int64_t n;
    const int32_t *box;
    const uint32_t *first;     // [boxes]
    const int32_t *start, *len;
};

// The unit of the calling warp: its box, first point and number of points.
__device__ __forceinline__ bool my_unit(const RmUnits &u, int64_t &b, int64_t &p0, int &n, bool &only)
{
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (w >= u.n) return false;
    b = u.box[w];
    const int64_t k = w - (int64_t)u.first[b], len = u.len[b];
    p0 = u.start[b] + k * kRmUnit;
    n = (int)min((int64_t)kRmUnit, len - k * kRmUnit);
    only = len <= kRmUnit;
    return true;
}

__device__ __forceinline__ RmPoint load_point(const RmPoint *p)
{
    const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    return {a.x, a.y, b.x, b.y};
}

__device__ __forceinline__ int octant(const RmPoint &p, const uint64_t *mid)
{
    return (order_key(p.x) >= mid[0] ? 1 : 0) | (order_key(p.y) >= mid[1] ? 2 : 0) | (order_key(p.z) >= mid[2] ? 4 : 0);
}

// Lanes of the warp whose active point lies in octant `oct`.
__device__ __forceinline__ unsigned octant_mask(int o, bool on, int oct)
{
    const unsigned act = __ballot_sync(0xffffffffu, on);
    unsigned m = act;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const unsigned bit = __ballot_sync(0xffffffffu, (o >> d) & 1);
        m &= (oct >> d) & 1 ? bit : ~bit;
    }
    return m;
}

// Bounds and tracer range over each unit, merged into its box.
__global__ void __launch_bounds__(kRmThreads) k_rm_stats(RmUnits u, const RmPoint *__restrict__ pts,
                                                         RmBox *__restrict__ box)
{
    int64_t b, p0;
    int n;
    bool only;
    if (!my_unit(u, b, p0, n, only)) return;       // whole warp
    const int lane = threadIdx.x & 31;
    RmBox s;
    empty_box(s);
    for (int i = lane; i < n; i += 32) {
        const RmPoint p = load_point(pts + p0 + i);
        const uint64_t c[4] = {order_key(p.x), order_key(p.y), order_key(p.z), order_key(p.rho)};
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            uint64_t &lo = s.v[d < 3 ? d : 6], &hi = s.v[d < 3 ? 3 + d : 7];
            lo = min(lo, c[d]);
            hi = max(hi, c[d]);
        }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        uint64_t v = s.v[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const uint64_t w = __shfl_xor_sync(0xffffffffu, v, o);
            v = k < 3 || k == 6 ? min(v, w) : max(v, w);
        }
        if (lane == 0) {
            unsigned long long *at = reinterpret_cast<unsigned long long *>(&box[b].v[k]);
            if (only)
                *at = v;
            else if (k < 3 || k == 6)
                atomicMin(at, (unsigned long long)v);
            else
                atomicMax(at, (unsigned long long)v);
        }
    }
}

// Division decision and midpoint of every box; the outermost box's bounds.
__global__ void k_rm_decide(int64_t nb, const RmBox *__restrict__ box, double r_max, bool may_divide,
                            uint8_t *__restrict__ divide, double *__restrict__ mids, double *__restrict__ root)
{
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const RmBox s = box[b];
    const double rmin = order_value(s.v[6]), rmax = order_value(s.v[7]);
    const double var = 2.0 * ((rmax - rmin) / (rmax + rmin));
    divide[b] = may_divide && var > r_max ? 1 : 0;
    for (int d = 0; d < 3; ++d) {
        const double lo = order_value(s.v[d]), hi = order_value(s.v[3 + d]);
        mids[3 * b + d] = (lo + hi) * 0.5;
        if (root) {
            root[d] = lo;
            root[3 + d] = hi;
        }
    }
}

// Octant counts of the dividing boxes (zeroed before the launch).
__global__ void __launch_bounds__(kRmThreads) k_rm_count(RmUnits u, const RmPoint *__restrict__ pts,
                                                         const double *__restrict__ mids,
                                                         const uint8_t *__restrict__ divide,
                                                         uint32_t *__restrict__ counts)
{
    int64_t b, p0;
    int n;
    bool only;
    if (!my_unit(u, b, p0, n, only) || !divide[b]) return;      // whole warp
    const int lane = threadIdx.x & 31;
    const uint64_t mid[3] = {ord_mid(mids[3 * b]), ord_mid(mids[3 * b + 1]), ord_mid(mids[3 * b + 2])};
    int c = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const bool on = i0 + lane < n;
        const int o = on ? octant(load_point(pts + p0 + i0 + lane), mid) : 0;
        c += __popc(octant_mask(o, on, lane & 7));
    }
    if (lane < 8) {
        if (only)
            counts[8 * b + lane] = c;
        else
            atomicAdd(&counts[8 * b + lane], (uint32_t)c);
    }
}

__global__ void k_rm_flags(int64_t nb, const uint8_t *__restrict__ divide, const uint32_t *__restrict__ counts,
                           RmCounts *__restrict__ out)
{
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b > nb) return;
    RmCounts r{0, 0, 0};                           // (entry nb: the scan's total)
    if (b < nb) {
        if (!divide[b]) {
            r.leaf = 1;
        } else {
            for (int o = 0; o < 8; ++o) {
                const uint32_t c = counts[8 * b + o];
                r.child += c > 0 ? 1 : 0;
                r.unit += (uint32_t)rm_units(c);
            }
        }
    }
    out[b] = r;
}

// Final boxes of this level -> centres; children of dividing boxes -> the
// next level's segments, units and empty boxes, and the octants' first places
// in place of their counts.
__global__ void k_rm_emit(int64_t nb, const int32_t *__restrict__ start, const double *__restrict__ mids,
                          const uint8_t *__restrict__ divide, uint32_t *__restrict__ counts,
                          const RmCounts *__restrict__ at, int64_t leaf_base, double *__restrict__ out,
                          int32_t *__restrict__ nstart, int32_t *__restrict__ nlen, uint32_t *__restrict__ nfirst,
                          int32_t *__restrict__ unit_box, RmBox *__restrict__ nbox)
{
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const RmCounts w = at[b];
    if (!divide[b]) {
        double *o = out + 3 * (leaf_base + w.leaf);
        for (int d = 0; d < 3; ++d) o[d] = mids[3 * b + d];
        return;
    }
    uint32_t a = (uint32_t)start[b], k = w.child, t = w.unit;
    for (int o = 0; o < 8; ++o) {
        const uint32_t c = counts[8 * b + o];
        counts[8 * b + o] = a;
        if (c > 0) {
            nstart[k] = (int32_t)a;
            nlen[k] = (int32_t)c;
            nfirst[k] = t;
            empty_box(nbox[k]);
            for (int64_t j = rm_units(c); j > 0; --j) unit_box[t++] = (int32_t)k;
            ++k;
        }
        a += c;
    }
}

// Move the points of dividing boxes into their children's segments (any order
// inside a child): a warp counts its unit's octants, takes the places of each
// octant with one addition, then writes.
__global__ void __launch_bounds__(kRmThreads) k_rm_scatter(RmUnits u, const RmPoint *__restrict__ pts,
                                                           RmPoint *__restrict__ out, const double *__restrict__ mids,
                                                           const uint8_t *__restrict__ divide,
                                                           uint32_t *__restrict__ place)
{
    int64_t b, p0;
    int n;
    bool only;
    if (!my_unit(u, b, p0, n, only) || !divide[b]) return;      // whole warp
    const int lane = threadIdx.x & 31;
    const uint64_t mid[3] = {ord_mid(mids[3 * b]), ord_mid(mids[3 * b + 1]), ord_mid(mids[3 * b + 2])};
    uint32_t at = 0;                               // lane o: next place of octant o
    if (only) {
        at = place[8 * b + (lane & 7)];
    } else {
        int c = 0;
        for (int i0 = 0; i0 < n; i0 += 32) {
            const bool on = i0 + lane < n;
            const int o = on ? octant(load_point(pts + p0 + i0 + lane), mid) : 0;
            c += __popc(octant_mask(o, on, lane & 7));
        }
        if (lane < 8)
            at = atomicAdd(&place[8 * b + lane], (uint32_t)c);
    }
    for (int i0 = 0; i0 < n; i0 += 32) {
        const bool on = i0 + lane < n;
        RmPoint p{};
        if (on) p = load_point(pts + p0 + i0 + lane);
        const int o = on ? octant(p, mid) : 0;
        const unsigned all = octant_mask(o, on, lane & 7);       // lane k: octant k & 7's points
        const unsigned same = __shfl_sync(0xffffffffu, all, o);  // my octant's
        const int64_t base = (int64_t)__shfl_sync(0xffffffffu, at, o);
        if (on) {
            double2 *q = reinterpret_cast<double2 *>(out + base + __popc(same & ((1u << lane) - 1u)));
            q[0] = make_double2(p.x, p.y);
            q[1] = make_double2(p.z, p.rho);
        }
        at += __popc(all);
    }
}

// Positions and tracer into points; the first level's one box and its units.
__global__ void k_rm_pack(int64_t n, const double *__restrict__ pos, const double *__restrict__ rho,
                          RmPoint *__restrict__ pts, int32_t *__restrict__ start, int32_t *__restrict__ len,
                          uint32_t *__restrict__ first, int32_t *__restrict__ unit_box, RmBox *__restrict__ box)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    double2 *q = reinterpret_cast<double2 *>(pts + i);
    q[0] = make_double2(no_negative_zero(pos[3 * i]), no_negative_zero(pos[3 * i + 1]));
    q[1] = make_double2(no_negative_zero(pos[3 * i + 2]), rho[i]);
    if (i < rm_units(n)) unit_box[i] = 0;
    if (i == 0) {
        *start = 0;
        *len = (int32_t)n;
        *first = 0;
        empty_box(*box);
    }
}

}  // namespace

}  // namespace mgt

using namespace mgt;

extern "C" mgt_status mgt_remesh(int64_t n_points, const double *pos, const double *rho, double r_max,
                                 int32_t max_level, int32_t n_side, double *out_pos, uint8_t *out_boundary,
                                 int64_t capacity, int64_t *n_out, void *stream)
{
    MGT_RANGE("mgt_remesh");
    if (n_points < 1 || n_points >= ((int64_t)1 << 31)) return set_error(MGT_ERR_ARG, "n_points must be 1..2^31-1");
    if (!pos || !rho || !n_out) return set_error(MGT_ERR_ARG, "pos, rho and n_out are required");
    if (!(r_max >= 0.0) || !std::isfinite(r_max)) return set_error(MGT_ERR_ARG, "r_max must be finite and >= 0");
    if (max_level < 0 || max_level > 30) return set_error(MGT_ERR_ARG, "max_level must be 0..30");
    if (n_side < 2 || n_side > 1024) return set_error(MGT_ERR_ARG, "n_side must be 2..1024");
    for (int64_t i = 0; i < n_points; ++i) {
        if (!(rho[i] > 0.0) || !std::isfinite(rho[i])) return set_error(MGT_ERR_ARG, "rho must be finite and > 0");
        for (int d = 0; d < 3; ++d)
            if (!std::isfinite(pos[3 * i + d])) return set_error(MGT_ERR_ARG, "positions must be finite");
    }
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t N = n_points;
    double *d_out = nullptr, *d_root = nullptr;
    RmPoint *pts = nullptr, *pts2 = nullptr;
    // (N < 2^31: places in the point buffers and counts are 32-bit; the working
    // memory is 253 bytes per point)
    int32_t *start = nullptr, *len = nullptr, *nstart = nullptr, *nlen = nullptr;
    uint32_t *first = nullptr, *nfirst = nullptr, *counts = nullptr;
    int32_t *unit_box = nullptr, *nunit_box = nullptr;
    double *mids = nullptr;
    RmBox *box = nullptr;
    RmCounts *at = nullptr;
    uint8_t *divide = nullptr;
    void *tmp = nullptr;
    size_t tmp_bytes = 0;
    std::vector<void *> owned;
    auto dev = [&](auto **p, size_t n) -> cudaError_t {
        cudaError_t e = cudaMallocAsync((void **)p, sizeof(**p) * (n ? n : 1), s);
        if (e == cudaSuccess) owned.push_back((void *)*p);
        return e;
    };
    struct Release {
        std::vector<void *> &v;
        cudaStream_t s;
        ~Release()
        {
            for (void *p : v) cudaFreeAsync(p, s);
        }
    } release{owned, s};
    // boxes of one level <= N; units <= boxes + N / kRmUnit
    const int64_t max_units = N + rm_units(N);
    MGT_CUDA(dev(&pts, N));
    MGT_CUDA(dev(&pts2, N));
    MGT_CUDA(dev(&d_out, 3 * N));
    MGT_CUDA(dev(&d_root, 6));
    for (int32_t **p : {&start, &len, &nstart, &nlen}) MGT_CUDA(dev(p, N));
    for (uint32_t **p : {&first, &nfirst}) MGT_CUDA(dev(p, N));
    for (int32_t **p : {&unit_box, &nunit_box}) MGT_CUDA(dev(p, max_units));
    MGT_CUDA(dev(&counts, 8 * N));
    MGT_CUDA(dev(&mids, 3 * N));
    MGT_CUDA(dev(&box, N));
    MGT_CUDA(dev(&at, N + 1));
    MGT_CUDA(dev(&divide, N));
    auto scan = [&](size_t &bytes, void *work, int64_t n) {
        return cub::DeviceScan::ExclusiveScan(work, bytes, at, at, RmAdd{}, RmCounts{0, 0, 0}, n, s);
    };
    MGT_CUDA(scan(tmp_bytes, nullptr, N + 1));
    MGT_CUDA(dev((unsigned char **)&tmp, tmp_bytes));
    {
        // the inputs pass through the second point buffer: positions, then the tracer
        double *in = reinterpret_cast<double *>(pts2);
        MGT_CUDA(cudaMemcpyAsync(in, pos, sizeof(double) * 3 * N, cudaMemcpyHostToDevice, s));
        MGT_CUDA(cudaMemcpyAsync(in + 3 * N, rho, sizeof(double) * N, cudaMemcpyHostToDevice, s));
        k_rm_pack<<<ceil_div(N, 256), 256, 0, s>>>(N, in, in + 3 * N, pts, start, len, first, unit_box, box);
        MGT_LAUNCH_CHECK("k_rm_pack");
    }
    int64_t nb = 1, n_units = rm_units(N), n_leaves = 0;
    for (int level = 0; nb > 0; ++level) {
        const RmUnits u{n_units, unit_box, first, start, len};
        const int ublocks = ceil_div(n_units * 32, kRmThreads), bblocks = ceil_div(nb + 1, 256);
        k_rm_stats<<<ublocks, kRmThreads, 0, s>>>(u, pts, box);
        MGT_LAUNCH_CHECK("k_rm_stats");
        k_rm_decide<<<bblocks, 256, 0, s>>>(nb, box, r_max, level < max_level, divide, mids,
                                            level == 0 ? d_root : nullptr);
        MGT_LAUNCH_CHECK("k_rm_decide");
        MGT_CUDA(cudaMemsetAsync(counts, 0, sizeof(uint32_t) * 8 * nb, s));
        k_rm_count<<<ublocks, kRmThreads, 0, s>>>(u, pts, mids, divide, counts);
        MGT_LAUNCH_CHECK("k_rm_count");
        k_rm_flags<<<bblocks, 256, 0, s>>>(nb, divide, counts, at);
        MGT_LAUNCH_CHECK("k_rm_flags");
        MGT_CUDA(scan(tmp_bytes, tmp, nb + 1));
        k_rm_emit<<<bblocks, 256, 0, s>>>(nb, start, mids, divide, counts, at, n_leaves, d_out, nstart, nlen, nfirst,
                                          nunit_box, box);
        MGT_LAUNCH_CHECK("k_rm_emit");
        k_rm_scatter<<<ublocks, kRmThreads, 0, s>>>(u, pts, pts2, mids, divide, counts);
        MGT_LAUNCH_CHECK("k_rm_scatter");
        RmCounts total{};
        MGT_CUDA(cudaMemcpyAsync(&total, at + nb, sizeof(RmCounts), cudaMemcpyDeviceToHost, s));
        MGT_CUDA(cudaStreamSynchronize(s));
        n_leaves += total.leaf;
        nb = total.child;
        n_units = total.unit;
        std::swap(pts, pts2);
        std::swap(start, nstart);
        std::swap(len, nlen);
        std::swap(first, nfirst);
        std::swap(unit_box, nunit_box);
    }
    double root[6];
    MGT_CUDA(cudaMemcpyAsync(root, d_root, sizeof root, cudaMemcpyDeviceToHost, s));
    MGT_CUDA(cudaStreamSynchronize(s));
    // evenly spaced boundary points: the surface nodes of the n_side^3 lattice
    // over the outermost box
    std::vector<double> bnd;
    for (int i = 0; i < n_side; ++i)
        for (int j = 0; j < n_side; ++j)
            for (int k = 0; k < n_side; ++k) {
                if (!(i == 0 || i == n_side - 1 || j == 0 || j == n_side - 1 || k == 0 || k == n_side - 1)) continue;
                const int ijk[3] = {i, j, k};
                for (int d = 0; d < 3; ++d)
                    bnd.push_back(root[d] + (double)ijk[d] / (n_side - 1) * (root[3 + d] - root[d]));
            }
    const int64_t nbnd = (int64_t)bnd.size() / 3;
    *n_out = n_leaves + nbnd;
    if (!out_pos) return MGT_OK;
    if (capacity < *n_out) return set_error(MGT_ERR_ARG, "capacity is below the number of output points (see n_out)");
    MGT_CUDA(cudaMemcpyAsync(out_pos, d_out, sizeof(double) * 3 * n_leaves, cudaMemcpyDeviceToHost, s));
    MGT_CUDA(cudaStreamSynchronize(s));
    std::copy(bnd.begin(), bnd.end(), out_pos + 3 * n_leaves);
    if (out_boundary) {
        std::fill(out_boundary, out_boundary + n_leaves, (uint8_t)0);
        std::fill(out_boundary + n_leaves, out_boundary + *n_out, (uint8_t)1);
    }
    return MGT_OK;
}
