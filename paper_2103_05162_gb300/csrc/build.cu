// Index construction: bounds, space-filling-curve keys, gather into sorted
// order, DenseBox cell classification and leaf layout, Karras LBVH topology
// and the node boxes (Sec. 4.1, 4.2).
#include <algorithm>

#include "build.cuh"

namespace gbd {

// DenseBox grid (Sec. 4.2) from the bounds, in double precision: cell side
// h = f * eps / sqrt(D) (computed by the host), enlarged when the widest axis
// would need more than 2^max_axis_bits - 2 cells (the per-cell guard keeps
// the result exact for any cell size, reading of Sec. 4.2); cmax_k = the
// cell index of hi_k (plus one spare cell for rounding at the top); the key
// interleaves `bits` bits per axis, enough for every cmax_k.
template <int D>
__device__ void make_grid(uint32_t* ctrl, const GridRequest& q)
{
    GridParams g{};
    double h = q.side;
    const double maxcells = (double)(1ull << q.max_axis_bits);
    float lo[D], hi[D];
    double ext_max = 0.0;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        lo[k] = ord2f(__ldcg(&ctrl[CTRL_LO + k]));
        hi[k] = ord2f(__ldcg(&ctrl[CTRL_HI + k]));
        ext_max = fmax(ext_max, (double)hi[k] - (double)lo[k]);
    }
    if (!(ext_max >= 0.0) || isinf(ext_max)) ext_max = 0.0;  // non-finite input: the run is aborted anyway
    if (ext_max / h >= maxcells - 2.0) h = ext_max / (maxcells - 2.0);
    const float inv_h = (float)(1.0 / h);
    int bits = 1;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        g.lo[k] = lo[k];
        double c = floor(((double)hi[k] - (double)lo[k]) * (double)inv_h) + 1.0;
        if (!(c >= 1.0)) c = 1.0;
        if (c > maxcells - 1.0) c = maxcells - 1.0;
        g.cmax[k] = (uint32_t)c;
        bits = max(bits, 32 - __clz((int)g.cmax[k]));
    }
    if (bits > q.max_axis_bits) bits = q.max_axis_bits;
    g.inv_h = inv_h;
    g.bits = bits;
    g.morton = 1;
    *q.gp = g;
    ctrl[CTRL_KEYBITS] = (uint32_t)(bits * D);
}

// ---------------------------------------------------------------------------
// K1: exact fp32 bounding box of the points, plus a flag for NaN/Inf.
// Each thread strides over the flat coordinate array with a stride that is a
// multiple of D, so it always sees the same axis. The kernel also clears the
// scratch that the stages after it find zeroed, and its last block computes
// the DenseBox grids: a memset or a one-thread kernel of its own cost 2 to 7 us
// of a small run each.
// ---------------------------------------------------------------------------
template <int D, int BT = bounds_threads<D>()>
__global__ void __launch_bounds__(BT) k_bounds(const float* __restrict__ pts, int64_t n,
                                               uint32_t* __restrict__ ctrl, BoundsExtra x)
{
    stage_begin(pts);
    __shared__ uint32_t s_lo[D], s_hi[D];
    __shared__ int s_bad, s_last;
    if (threadIdx.x < D) { s_lo[threadIdx.x] = 0xffffffffu; s_hi[threadIdx.x] = 0u; }
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    const int64_t total = n * D;
    const int64_t stride = (int64_t)gridDim.x * BT;
    const int64_t first = blockIdx.x * (int64_t)BT + threadIdx.x;
#pragma unroll
    for (int z = 0; z < 2; ++z)
        for (int64_t i = first; i < x.zero16[z]; i += stride) x.zero[z][i] = make_uint4(0u, 0u, 0u, 0u);
    const int axis = threadIdx.x % D;
    float lo = INFINITY, hi = -INFINITY;
    bool bad = false;
    for (int64_t i = first; i < total; i += stride) {
        float v = __ldcs(pts + i);
        bad |= !isfinite(v);
        lo = fminf(lo, v);
        hi = fmaxf(hi, v);
    }
    if (lo <= hi) {
        atomicMin(&s_lo[axis], f2ord(lo));
        atomicMax(&s_hi[axis], f2ord(hi));
    }
    if (bad) s_bad = 1;
    __syncthreads();
    if (threadIdx.x < D) {
        atomicMin(&ctrl[CTRL_LO + threadIdx.x], s_lo[threadIdx.x]);
        atomicMax(&ctrl[CTRL_HI + threadIdx.x], s_hi[threadIdx.x]);
        __threadfence();
    }
    if (threadIdx.x == 0 && s_bad) atomicOr(&ctrl[CTRL_ABORT], ERR_NONFINITE);
    if (x.grids == 0) return;
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&ctrl[CTRL_TICKET], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last || threadIdx.x != 0) return;
    __threadfence();
    // (the run's own grid last: CTRL_KEYBITS is its)
    for (int q = 0; q < x.grids; ++q) make_grid<D>(ctrl, x.grid[q]);
}

// the run's first kernel (see launch_run_begin)
__global__ void k_run_begin(uint32_t* ctrl, int algo)
{
    stage_begin();
    const int t = threadIdx.x;
    if (t == 0) {
        const uint32_t a = ctrl[CTRL_ABORT];
        if (a) ctrl[CTRL_ERR] |= a;
        ctrl[CTRL_ABORT] = 0u;
        ctrl[CTRL_ALGO] = (uint32_t)algo;
        ctrl[CTRL_M] = 0u;
        ctrl[CTRL_NCELLS] = 0u;
        ctrl[CTRL_TICKET] = 0u;
    }
    if (t < MAX_DIM) {
        ctrl[CTRL_LO + t] = 0xffffffffu;
        ctrl[CTRL_HI + t] = 0u;
    }
}

// ---------------------------------------------------------------------------
// K2: keys. Bit interleaving with axis 0 in the lowest bit.
// ---------------------------------------------------------------------------
// Morton code of each point on a 2^bits grid over the (device-side) bounds;
// u32 keys (FDBSCAN ordering). values = input index.
template <int D>
__global__ void k_morton32(const float* __restrict__ pts, int64_t n, const uint32_t* __restrict__ ctrl, int bits,
                           uint32_t* __restrict__ keys, uint32_t* __restrict__ vals)
{
    stage_begin(pts, ctrl);
    if (!stage_on(ctrl, DBSCAN_ALGO_FDBSCAN)) return;
    float lo[D], scale[D];
    const float cells = (float)(1u << bits);
#pragma unroll
    for (int k = 0; k < D; ++k) {
        lo[k] = ord2f(ctrl[CTRL_LO + k]);
        const float ext = __fsub_rn(ord2f(ctrl[CTRL_HI + k]), lo[k]);
        scale[k] = ext > 0.0f ? __fdiv_rn(cells, ext) : 0.0f;
    }
    const uint32_t cmax = (1u << bits) - 1u;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t c[D];
#pragma unroll
        for (int k = 0; k < D; ++k) {
            c[k] = cell_index(floorf(__fmul_rn(__fsub_rn(pts[i * D + k], lo[k]), scale[k])), cmax);
        }
        keys[i] = (uint32_t)interleave<D>(c);
        vals[i] = (uint32_t)i;
    }
}

// The same with 64-bit keys (FDBSCAN ordering above 3D).
template <int D>
__global__ void k_morton64(const float* __restrict__ pts, int64_t n, const uint32_t* __restrict__ ctrl, int bits,
                           uint64_t* __restrict__ keys, uint32_t* __restrict__ vals)
{
    stage_begin(pts, ctrl);
    if (!stage_on(ctrl, DBSCAN_ALGO_FDBSCAN)) return;
    float lo[D], scale[D];
    const float cells = (float)(1u << bits);
#pragma unroll
    for (int k = 0; k < D; ++k) {
        lo[k] = ord2f(ctrl[CTRL_LO + k]);
        const float ext = __fsub_rn(ord2f(ctrl[CTRL_HI + k]), lo[k]);
        scale[k] = ext > 0.0f ? __fdiv_rn(cells, ext) : 0.0f;
    }
    const uint32_t cmax = (1u << bits) - 1u;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t c[D];
#pragma unroll
        for (int k = 0; k < D; ++k) {
            c[k] = cell_index(floorf(__fmul_rn(__fsub_rn(pts[i * D + k], lo[k]), scale[k])), cmax);
        }
        keys[i] = interleave<D>(c);
        vals[i] = (uint32_t)i;
    }
}

// Grid-cell key of each point (DenseBox, Sec. 4.2): cell index
// floor((x_k - lo_k) * inv_h) clamped to [0, cmax_k], Morton-interleaved (or
// packed axis by axis when `morton` is 0). values = input index.
template <int D>
__device__ __forceinline__ uint64_t cell_key(const float* __restrict__ p, const GridParams& g)
{
    uint32_t c[D];
#pragma unroll
    for (int k = 0; k < D; ++k) c[k] = cell_index(floorf(__fmul_rn(__fsub_rn(p[k], g.lo[k]), g.inv_h)), g.cmax[k]);
    uint64_t key;
    if (g.morton) {
        key = interleave<D>(c);
    } else {
        key = 0;
#pragma unroll
        for (int k = D - 1; k >= 0; --k) key = (key << g.bits) | c[k];
    }
    return key;
}

// Packed for a keys-only sort: key << idx_bits | i in one word (the host
// caps the grid so that key bits + idx_bits <= 64, and n <= 2^idx_bits). The
// words go to the buffer the sort takes its input from (sort_dev_input_alt).
template <int D>
__global__ void k_cellkey_packed(const float* __restrict__ pts, int64_t n, const GridParams* __restrict__ gp,
                                 const uint32_t* __restrict__ ctrl, int idx_bits, int host_passes,
                                 uint64_t* __restrict__ words0, uint64_t* __restrict__ words1)
{
    stage_begin(pts, gp, ctrl);
    if (!stage_on(ctrl, DBSCAN_ALGO_DENSEBOX)) return;
    const GridParams g = *gp;
    // (host_passes 0: no sort runs, n <= 1, and the words stay in words0)
    uint64_t* __restrict__ words =
        host_passes > 0 && sort_dev_input_alt(host_passes, sort_passes((int)ctrl[CTRL_KEYBITS])) ? words1 : words0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        words[i] = (cell_key<D>(pts + i * D, g) << idx_bits) | (uint64_t)i;
}

// ---------------------------------------------------------------------------
// Density estimate for the automatic FDbscan / DenseBox choice: the share of
// points that lie in DenseBox cells holding at least minPts points, from
// EST_SAMPLES strided sample points. Their cells go into an open-addressing
// table; one pass over all points counts the points of each sampled cell
// (per-block shared counters, flushed once); the estimate is the share of
// samples whose cell reaches minPts. Above 2^22 points the counting pass
// reads every stride-th point only and scales its counts by the stride (an
// estimate either way). Keys use at most 63 bits, so the all-ones word marks
// an empty slot.
// ---------------------------------------------------------------------------
constexpr unsigned long long EST_EMPTY = ~0ull;

__device__ __forceinline__ uint32_t est_hash(uint64_t k)
{
    return (uint32_t)((k * 0x9E3779B97F4A7C15ull) >> 52);  // 12 bits: EST_SLOTS = 4096
}

template <int D>
__global__ void k_est_insert(const float* __restrict__ pts, int64_t n, int s, const GridParams* __restrict__ gp,
                             const uint32_t* __restrict__ ctrl, unsigned long long* __restrict__ table,
                             int32_t* __restrict__ slot)
{
    stage_begin(pts, gp, ctrl);
    if (!stage_on(ctrl, -1)) return;
    const GridParams g = *gp;
    for (int j = threadIdx.x; j < s; j += blockDim.x) {
        const int64_t i = (int64_t)j * n / s;
        const unsigned long long key = cell_key<D>(pts + i * D, g);
        uint32_t h = est_hash(key);
        slot[j] = -1;
        for (int probe = 0; probe < EST_SLOTS; ++probe) {  // load <= 1/2: a slot is always found
            const unsigned long long prev = atomicCAS(&table[h], EST_EMPTY, key);
            if (prev == EST_EMPTY || prev == key) {
                slot[j] = (int32_t)h;
                break;
            }
            h = (h + 1) & (EST_SLOTS - 1);
        }
    }
}

template <int D>
__global__ void k_est_count(const float* __restrict__ pts, int64_t n, int64_t stride,
                            const GridParams* __restrict__ gp, const uint32_t* __restrict__ ctrl,
                            const unsigned long long* __restrict__ table, uint32_t* __restrict__ counts)
{
    stage_begin(pts, gp, ctrl, table);
    if (!stage_on(ctrl, -1)) return;
    const GridParams g = *gp;
    __shared__ uint32_t sc[EST_SLOTS];
    for (int t = threadIdx.x; t < EST_SLOTS; t += blockDim.x) sc[t] = 0;
    __syncthreads();
    const int64_t nc = (n + stride - 1) / stride;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nc; j += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long key = cell_key<D>(pts + j * stride * D, g);
        uint32_t h = est_hash(key);
        for (int probe = 0; probe < EST_SLOTS; ++probe) {
            const unsigned long long k = table[h];
            if (k == key) {
                atomicAdd(&sc[h], 1u);
                break;
            }
            if (k == EST_EMPTY) break;
            h = (h + 1) & (EST_SLOTS - 1);
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < EST_SLOTS; t += blockDim.x)
        if (sc[t]) atomicAdd(&counts[t], sc[t]);
}

// out[0] = samples whose cell holds >= min_pts points; out[2..3] = the sum
// over the samples of their cell's point count (64-bit, low word first);
// then the choice: DenseBox if the dense share reaches auto_fraction or the
// mean occupancy auto_occupancy, else FDbscan (CTRL_ALGO, estimates in
// CTRL_EST_FRAC / CTRL_EST_OCC). One block.
__global__ void k_est_result(const int32_t* __restrict__ slot, int s, const uint32_t* __restrict__ counts,
                             int64_t n, int64_t stride, int min_pts, float auto_fraction, float auto_occupancy,
                             uint32_t* __restrict__ out, uint32_t* __restrict__ ctrl)
{
    stage_begin(slot, counts);
    if (!stage_on(ctrl, -1)) return;
    uint32_t c = 0;
    unsigned long long occ = 0;
    for (int j = threadIdx.x; j < s; j += blockDim.x) {
        if (slot[j] < 0) continue;
        // the sample itself once, the other counted points of its cell scaled
        // by the stride (the sample is among the counted points iff its index
        // is a multiple of the stride)
        const int64_t i = (int64_t)j * n / s;
        const unsigned long long self = (i % stride == 0) ? 1ull : 0ull;
        const unsigned long long others = (unsigned long long)counts[slot[j]] - self;
        const unsigned long long k = 1ull + others * (unsigned long long)stride;
        if (k >= (unsigned long long)min_pts) ++c;
        occ += k;
    }
    atomicAdd(out, c);
    atomicAdd(reinterpret_cast<unsigned long long*>(out + 2), occ);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence_block();
        const uint32_t dense = *(volatile uint32_t*)out;
        const unsigned long long occ_sum = *(volatile unsigned long long*)(out + 2);
        const float frac = (float)dense / (float)s;
        const float mean_occ = (float)((double)occ_sum / (double)s);
        ctrl[CTRL_EST_FRAC] = __float_as_uint(frac);
        ctrl[CTRL_EST_OCC] = __float_as_uint(mean_occ);
        ctrl[CTRL_ALGO] = (frac >= auto_fraction || mean_occ >= auto_occupancy) ? (uint32_t)DBSCAN_ALGO_DENSEBOX
                                                                               : (uint32_t)DBSCAN_ALGO_FDBSCAN;
    }
}

// generic Morton codes with host-side bounds (component entry point)
template <int D>
__global__ void k_morton_generic(const float* __restrict__ pts, int64_t n, GridParams g, uint64_t* __restrict__ out)
{
    stage_begin(pts);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t c[D];
#pragma unroll
        for (int k = 0; k < D; ++k) {
            c[k] = cell_index(floorf(__fmul_rn(__fsub_rn(pts[i * D + k], g.lo[k]), g.scale[k])), g.cmax[k]);
        }
        uint64_t key = 0;
        for (int b = 0; b < g.bits; ++b)
            for (int k = 0; k < D; ++k) key |= (uint64_t)((c[k] >> b) & 1u) << (b * D + k);
        out[i] = key;
    }
}

// ---------------------------------------------------------------------------
// K4: gather the points into sorted order (structure of points, one 16-byte
// (3D) or 8-byte (2D) record per point).
// ---------------------------------------------------------------------------
template <int D>
__global__ void k_gather(const float* __restrict__ pts, const uint32_t* __restrict__ perm, int64_t n,
                         typename Traits<D>::Point* __restrict__ sp, const uint32_t* __restrict__ ctrl, int algo)
{
    stage_begin(pts, perm, ctrl);
    // a sort that gave up leaves stale words in perm: never index with them
    if (!stage_on(ctrl, algo)) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        sp[i] = Traits<D>::load_point(pts, perm[i]);
}

// A 3D input point (12 bytes at float index 3j) read in aligned pieces: the
// 16-byte block that holds it when it lies in one (one load), else an 8-byte
// and a 4-byte piece (two loads), never past the end of the array (n points).
// The input must be 16-byte aligned.
__device__ __forceinline__ float4 load_point3_aligned(const float* __restrict__ pts, uint32_t j, int64_t n)
{
    const int64_t f = 3 * (int64_t)j;
    const int64_t b = f & ~(int64_t)3;
    const int o = (int)(f - b);
    if (o == 1 || (o == 0 && b + 4 <= 3 * n)) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(pts + b));
        return o == 0 ? make_float4(v.x, v.y, v.z, 0.0f) : make_float4(v.y, v.z, v.w, 0.0f);
    }
    if (o == 3) {
        const float2 yz = __ldg(reinterpret_cast<const float2*>(pts + f + 1));
        return make_float4(__ldg(pts + f), yz.x, yz.y, 0.0f);
    }
    // o == 2, or the last point of the array at o == 0
    const float2 xy = __ldg(reinterpret_cast<const float2*>(pts + f));
    return make_float4(xy.x, xy.y, __ldg(pts + f + 2), 0.0f);
}

template <int D, bool A16>
__device__ __forceinline__ typename Traits<D>::Point gather_point(const float* __restrict__ pts, uint32_t j, int64_t n)
{
    if constexpr (D == 3 && A16) return load_point3_aligned(pts, j, n);
    else return Traits<D>::load_point(pts, j);
}

// The same from sorted packed words, which it splits into the permutation
// and the sorted keys: two sorted positions per thread and step, so that two
// independent input reads are in flight (the words, keys and permutation are
// 16- and 8-byte aligned workspace arrays).
template <int D, bool A16>
__global__ void k_gather_packed(const float* __restrict__ pts, const uint64_t* __restrict__ words, int64_t n,
                                int idx_bits, typename Traits<D>::Point* __restrict__ sp,
                                uint32_t* __restrict__ perm, uint64_t* __restrict__ keys,
                                const uint32_t* __restrict__ ctrl)
{
    stage_begin(pts, words, ctrl);
    using P = typename Traits<D>::Point;
    if (!stage_on(ctrl, DBSCAN_ALGO_DENSEBOX)) return;  // (a sort that gave up: stale index bits)
    const uint64_t mask = (1ull << idx_bits) - 1ull;
    const int64_t pairs = n >> 1;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < pairs; t += stride) {
        // the words are read once and the permutation is next read by the
        // last stages: both stream through L2 with evict-first priority, so
        // that more of the randomly read input points stay cached
        const ulonglong2 w = __ldcs(reinterpret_cast<const ulonglong2*>(words) + t);
        const uint32_t j0 = (uint32_t)(w.x & mask), j1 = (uint32_t)(w.y & mask);
        const P p0 = gather_point<D, A16>(pts, j0, n);
        const P p1 = gather_point<D, A16>(pts, j1, n);
        __stcs(reinterpret_cast<uint2*>(perm) + t, make_uint2(j0, j1));
        reinterpret_cast<ulonglong2*>(keys)[t] = make_ulonglong2(w.x >> idx_bits, w.y >> idx_bits);
        sp[2 * t] = p0;
        sp[2 * t + 1] = p1;
    }
    if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) {
        const int64_t i = n - 1;
        const uint64_t w = words[i];
        const uint32_t j = (uint32_t)(w & mask);
        perm[i] = j;
        keys[i] = w >> idx_bits;
        sp[i] = gather_point<D, A16>(pts, j, n);
    }
}

// ---------------------------------------------------------------------------
// K5/K6: DenseBox classification. Cells are runs of equal keys in sorted
// order. A cell is dense iff it holds at least minPts points AND the squared
// distance between the corners of the exact bounding box of its points passes
// the eps test: by monotone rounding every pair inside then passes too, so
// "all points core and in one cluster" (Sec. 4.2) holds exactly, whatever
// rounding the grid arithmetic suffered (the precision hazard of Sec. 4.2 is
// turned into a per-cell check instead of an abort).
//
// One pass: the thread at the first point of a run checks with one load
// whether the run reaches minPts points, and walks it if it does. Runs of up
// to CELL_THREAD points end there, all lanes at once; the block collects the
// longer ones of a round of its steps, its warps take those of up to CELL_WARP
// points, and the whole block the rest: the end by a 256-way search, the box
// with four loads in flight per thread. The points of a dense cell are marked
// 1 (fits in a tile) or 2 (larger: a leaf of its own), with the run's first
// point, and the box of a cell larger than a tile goes to dbox[first point /
// 32] (more than 32 points: no two such cells share a slot) for the leaf boxes.
// Bound by the latency of its loads. Batch of 512 instances (cells of up to
// 29,000 points): 376 us, one warp walking one run after another 932, a thread
// per run of up to 64 points 840, groups of 8 lanes 428; 3.9M 2D blob points
// (few large cells): the leaves stage 215 us instead of 2300; 16.8M halos 127
// instead of 85. The leaf boxes, which walked the large cells again, fell from
// 511 to 38 us on the batch and from 119 to 76 on the halos, with the topology
// that is now in the same launch. pdense must be zero on entry.
//
// Batches: the key's bits from lb up are the instance, whose minPts and eps^2
// are read from mps and e2s (null: min_pts and e2).
// ---------------------------------------------------------------------------
constexpr int CELL_THREADS = 256;
constexpr int CELL_STEPS = 16;    // at most, per round
constexpr int CELL_THREAD = 8;    // a multiple of 4
constexpr int CELL_WARP = 1024;   // a multiple of 64
// runs of more than so many points that start in one round, at most
constexpr int CELL_RUNS_WARP = CELL_STEPS * CELL_THREADS / (CELL_THREAD + 1) + 1;
constexpr int CELL_RUNS_BLOCK = CELL_STEPS * CELL_THREADS / (CELL_WARP + 1) + 1;

template <int D>
__global__ void __launch_bounds__(CELL_THREADS)
    k_dense_classify(const uint64_t* __restrict__ keys, const typename Traits<D>::Point* __restrict__ sp, int64_t n,
                     int min_pts, float e2, const int32_t* __restrict__ mps, const float* __restrict__ e2s, int lb,
                     uint8_t* __restrict__ pdense, int32_t* __restrict__ dstart,
                     typename Traits<D>::Box* __restrict__ dbox, uint32_t* __restrict__ ctrl, int algo, int steps)
{
    stage_begin(keys, sp, mps, e2s);
    using T = Traits<D>;
    using Box = typename T::Box;
    if (!stage_on(ctrl, algo)) return;
    __shared__ int64_t s_run[CELL_RUNS_WARP];  // first points of the runs for the warps,
    __shared__ int64_t s_long[CELL_RUNS_BLOCK];   // and for the block
    __shared__ int s_n[2];
    __shared__ long long s_end;
    __shared__ Box s_box[CELL_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t chunk = (int64_t)steps * CELL_THREADS;
    for (int64_t base = blockIdx.x * chunk; base < n; base += gridDim.x * chunk) {  // whole blocks together
        if (threadIdx.x < 2) s_n[threadIdx.x] = 0;
        __syncthreads();
        for (int step = 0; step < steps; ++step) {
            const int64_t i = base + step * CELL_THREADS + threadIdx.x;
            uint64_t k = 0;
            bool cand = false;
            if (i < n) {
                k = keys[i];
                const int64_t j = i + (mps ? mps[k >> lb] : min_pts) - 1;
                cand = j < n && keys[j] == k && (i == 0 || keys[i - 1] != k);
            }
            bool dense = false;
            if (cand) {
                Box b = T::empty_box();
                int len = 0;
                bool more = true;
                while (more && len < CELL_THREAD) {
                    // four points at a time (past the run's end: its first point again)
                    bool in[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) in[u] = i + len + u < n && keys[i + len + u] == k;
#pragma unroll
                    for (int u = 1; u < 4; ++u) in[u] = in[u] && in[u - 1];
#pragma unroll
                    for (int u = 0; u < 4; ++u) T::grow(b, sp[in[u] ? i + len + u : i]);
                    len += in[0] + in[1] + in[2] + in[3];
                    more = in[3];
                }
                if (more && i + len < n && keys[i + len] == k) {
                    s_run[atomicAdd(&s_n[0], 1)] = i;
                } else if (T::diag2(b) <= (mps ? e2s[k >> lb] : e2)) {  // the guard: provably one clique
                    dense = true;
                    for (int t = 0; t < len; ++t) {
                        pdense[i + t] = 1;
                        dstart[i + t] = (int32_t)i;
                    }
                }
            }
            const unsigned dm = __ballot_sync(FULL, dense);
            if (lane == 0 && dm) atomicAdd(&ctrl[CTRL_NCELLS], (uint32_t)__popc(dm));
        }
        __syncthreads();
        const int nr = s_n[0];
        for (int q = warp; q < nr; q += CELL_THREADS / 32) {
            const int64_t c0 = s_run[q];
            const uint64_t k = keys[c0];
            Box b = T::empty_box();
            int len = 0;
            bool more = true;
            while (more && len < CELL_WARP) {
                // two points per lane (past the run's end: its first point again)
                const int64_t t0 = c0 + len + lane, t1 = t0 + 32;
                const bool in0 = t0 < n && keys[t0] == k, in1 = t1 < n && keys[t1] == k;
                T::grow(b, sp[in0 ? t0 : c0]);
                T::grow(b, sp[in1 ? t1 : c0]);
                const unsigned m1 = __ballot_sync(FULL, in1);
                len += __popc(__ballot_sync(FULL, in0)) + __popc(m1);
                more = m1 == FULL;
            }
            if (more && c0 + len < n && keys[c0 + len] == k) {
                if (lane == 0) s_long[atomicAdd(&s_n[1], 1)] = c0;
                continue;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) T::merge(b, T::shfl_xor(b, o));
            if (T::diag2(b) > (mps ? e2s[k >> lb] : e2)) continue;
            if (lane == 0) {
                if (len > TILE) dbox[c0 >> 5] = b;
                atomicAdd(&ctrl[CTRL_NCELLS], 1u);
            }
            for (int t = lane; t < len; t += 32) {
                pdense[c0 + t] = len > TILE ? 2 : 1;
                dstart[c0 + t] = (int32_t)c0;
            }
        }
        __syncthreads();
        const int nl = s_n[1];
        for (int q = 0; q < nl; ++q) {
            const int64_t c0 = s_long[q];
            const uint64_t kk = keys[c0];
            // the run's end: lo is in the run, hi is not (or is n)
            int64_t lo = c0 + CELL_WARP, hi = n;
            while (hi - lo > 1) {
                const int64_t step = (hi - lo + CELL_THREADS - 1) / CELL_THREADS;
                const int64_t p = lo + (threadIdx.x + 1) * step;
                // the last probe in the run
                if (threadIdx.x == 0) s_end = lo;
                __syncthreads();
                if (p < hi && keys[p] == kk) atomicMax(&s_end, (long long)p);
                __syncthreads();
                const int64_t last = s_end;
                __syncthreads();
                lo = last;
                hi = hi < last + step ? hi : last + step;
            }
            const int64_t e = hi;
            Box b = T::empty_box();
            for (int64_t t = c0 + threadIdx.x; t < e; t += 4 * CELL_THREADS) {
                typename T::Point p[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int64_t at = t + u * CELL_THREADS;
                    p[u] = sp[at < e ? at : t];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) T::grow(b, p[u]);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) T::merge(b, T::shfl_xor(b, o));
            if (lane == 0) s_box[warp] = b;
            __syncthreads();
            b = s_box[0];
            for (int w = 1; w < CELL_THREADS / 32; ++w) T::merge(b, s_box[w]);
            if (T::diag2(b) <= (mps ? e2s[kk >> lb] : e2)) {
                if (threadIdx.x == 0) {
                    dbox[c0 >> 5] = b;
                    atomicAdd(&ctrl[CTRL_NCELLS], 1u);
                }
                for (int64_t t = c0 + threadIdx.x; t < e; t += CELL_THREADS) {
                    pdense[t] = 2;
                    dstart[t] = (int32_t)c0;
                }
            }
            __syncthreads();  // s_box and s_end are used again
        }
        __syncthreads();  // (all have read the counts)
    }
}

template <typename K>
__device__ __forceinline__ K shfl_key(K v, int src)
{
    if constexpr (sizeof(K) == 8) {
        const uint32_t lo = __shfl_sync(FULL, (uint32_t)v, src), hi = __shfl_sync(FULL, (uint32_t)(v >> 32), src);
        return (K)(((uint64_t)hi << 32) | lo);
    } else {
        return (K)__shfl_sync(FULL, (uint32_t)v, src);
    }
}

// Leaves. A new leaf starts at point i where the node of the points' radix
// tree (Karras: keys with position tie-break) that splits i - 1 from i covers
// more than TILE points -- tiles are then the maximal subtrees of at most TILE
// points, spatially compact unlike fixed runs in Morton order; and at the
// first point of every dense cell larger than a tile, after such a cell, and
// (batches) where the instance changes.
// With e[i] the prefix length delta(i - 1, i), that node covers the run of
// splits around i of prefix length at least e[i] (the common prefix of two
// sorted keys is the smallest adjacent one between them): it covers more than
// TILE points iff some TILE consecutive splits that include i have no smaller
// prefix than e[i], i.e. iff the largest over those windows of their smallest
// prefix reaches e[i] -- a sliding minimum and a sliding maximum of width 32,
// five doubling steps of warp shuffles each. (Probes of the keys 15 and 31
// positions away with ballots for the undecided took 233 us on 16.8M halos.)
//
// Two kernels over the same split of the positions into contiguous parts, one
// per warp (at most LF_BLOCKS blocks, so that every block can add up the counts
// of those before it): k_leaf_flags writes the starts as bit words and counts
// them, k_leaf_records numbers them and writes the leaf records, a leaf's end
// by the thread that finds the next start. Flags by key probes and ballots, a
// three-kernel scan, starts and records took 284 us on 16.8M halos in seven
// launches; these take 112 and 63. (One kernel with a decoupled look-back took 186:
// the blocks stood at its barrier while their offsets came.)
constexpr int LEAF_T = TILE;
static_assert(LEAF_T == 32, "windows of one warp");
constexpr int LF_THREADS = 256;
constexpr int LF_WARPS = LF_THREADS / 32;
constexpr int LF_BLOCKS = LEAF_BLOCKS;
constexpr int LF_MIN_WINDOWS = 4;  // windows of 32 positions per warp, an even number

// Sliding minima and maxima of two windows at once, one in each 16-bit half
// (prefix lengths are at most 96, -1 outside the points).
__device__ __forceinline__ unsigned pack2(int lo, int hi) { return __byte_perm((unsigned)lo, (unsigned)hi, 0x5410); }
__device__ __forceinline__ int half_lo(unsigned v) { return (int)(short)v; }
__device__ __forceinline__ int half_hi(unsigned v) { return (int)v >> 16; }
// the smallest of e[s .. s + 31], for s in the window a (this lane: s), which
// the window b follows
__device__ __forceinline__ unsigned window_min(unsigned a, unsigned b, int lane)
{
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        // (within b, positions past its end repeat its last one: a's minima
        // never reach them)
        const unsigned x = __shfl_sync(FULL, a, (lane + k) & 31), y = __shfl_sync(FULL, b, (lane + k) & 31);
        b = __vmins2(b, __shfl_down_sync(FULL, b, k));
        a = __vmins2(a, lane + k < 32 ? x : y);
    }
    return a;
}
// the largest of v[s - 31 .. s], for s in the window b, which follows a
__device__ __forceinline__ unsigned window_max(unsigned a, unsigned b, int lane)
{
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        const unsigned x = __shfl_sync(FULL, a, (lane - k) & 31), y = __shfl_sync(FULL, b, (lane - k) & 31);
        a = __vmaxs2(a, __shfl_up_sync(FULL, a, k));
        b = __vmaxs2(b, lane >= k ? y : x);
    }
    return b;
}

template <typename K>
__global__ void __launch_bounds__(LF_THREADS)
    k_leaf_flags(const K* __restrict__ keys, const int32_t* __restrict__ dstart, const uint8_t* __restrict__ pdense,
                 int64_t n, int windows, int id_shift, uint32_t* __restrict__ words, uint32_t* __restrict__ counts,
                 const uint32_t* __restrict__ ctrl, int algo)
{
    stage_begin(keys, dstart, pdense, ctrl);
    if (!stage_on(ctrl, algo)) return;
    const int lane = threadIdx.x & 31;
    const int warp = blockIdx.x * LF_WARPS + (threadIdx.x >> 5);
    const int64_t base64 = (int64_t)warp * (32 * windows);
    const int base = base64 < n ? (int)base64 : (int)n;  // (positions fit 31 bits)
    const int np = (int)n;

    // the splits' prefix lengths of the window at p (e[p + lane]; -1 outside
    // the points), given its keys and the last key before it
    auto key_at = [&](int i) { return (unsigned)i < (unsigned)np ? keys[i] : K(0); };
    auto splits = [&](int p, K k, K before) {
        K kp = shfl_key(k, (lane + 31) & 31);
        if (lane == 0) kp = before;
        const int i = p + lane;
        constexpr int KB = 8 * (int)sizeof(K);
        const int d = k != kp ? (sizeof(K) == 8 ? __clzll((long long)(k ^ kp)) : __clz((int)(k ^ kp)))
                              : KB + __clz(i ^ (i - 1));
        return i >= 1 && i < np ? d : -1;
    };
    uint32_t count = 0;
    if (base < np) {
        K kc = key_at(base + lane), k1 = key_at(base + 32 + lane), k2 = key_at(base + 64 + lane);
        const K kp = key_at(base - 32 + lane);
        int ec = splits(base, kc, shfl_key(kp, 31));
        int wp = half_lo(window_min(pack2(splits(base - 32, kp, key_at(base - 33)), 0), pack2(ec, 0), lane));
        K kprev = shfl_key(kp, 31);  // the key before the current window
        unsigned carry = pdense && base > 0 && pdense[base - 1] == 2;
#pragma unroll 1
        for (int w = 0; w < windows && base + 32 * (int64_t)w < n; w += 2) {
            const int p = base + 32 * w;
            const int e1 = splits(p + 32, k1, shfl_key(kc, 31)), e2 = splits(p + 64, k2, shfl_key(k1, 31));
            const K k3 = key_at(p + 96 + lane), k4 = key_at(p + 128 + lane);  // (in flight during this step)
            const unsigned wc = window_min(pack2(ec, e1), pack2(e1, e2), lane);
            const unsigned mx = window_max(pack2(wp, half_lo(wc)), wc, lane);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = p + 32 * h + lane;
                const bool in = i < np;
                unsigned word = __ballot_sync(FULL, in && (h ? half_hi(mx) >= e1 : half_lo(mx) >= ec));
                if (id_shift < 64) {
                    const K k = h ? k1 : kc, before = h ? shfl_key(kc, 31) : kprev;
                    K kl = shfl_key(k, (lane + 31) & 31);
                    if (lane == 0) kl = before;
                    word |= __ballot_sync(FULL, in && ((uint64_t)k >> id_shift) != ((uint64_t)kl >> id_shift));
                }
                if (pdense) {
                    // dense cells larger than a tile: only their first point
                    // starts a leaf, and the point after them does
                    const unsigned d2 = __ballot_sync(FULL, in && pdense[in ? i : 0] == 2);
                    if (d2 | carry) {
                        const unsigned st = __ballot_sync(FULL, ((d2 >> lane) & 1u) && dstart[in ? i : 0] == i);
                        const unsigned valid = __ballot_sync(FULL, in);
                        word = ((word | ((d2 << 1) | carry)) & ~d2 & valid) | st;
                    }
                    carry = d2 >> 31;
                }
                if (p + 32 * h == 0) word |= 1u;
                if (lane == 0 && p + 32 * h < np) words[(p >> 5) + h] = word;
                count += __popc(word);
            }
            kprev = shfl_key(k1, 31);
            kc = k2;
            k1 = k3;
            k2 = k4;
            ec = e2;
            wp = half_hi(wc);
        }
    }

    if (lane == 0) counts[warp] = count;
}

template <typename K>
__global__ void __launch_bounds__(LF_THREADS)
    k_leaf_records(const K* __restrict__ keys, const uint8_t* __restrict__ pdense, int64_t n, int windows, int id_shift,
                   const uint32_t* __restrict__ words, const uint32_t* __restrict__ counts, int2* __restrict__ leafr,
                   uint64_t* __restrict__ lkey, int32_t* __restrict__ linst, uint32_t* __restrict__ ctrl, int algo)
{
    stage_begin(keys, pdense, words, counts);
    // (skipped -- aborted run, or the other algorithm's chain --: m stays 0
    // and every later stage finds no leaves)
    if (!stage_on(ctrl, algo)) return;
    __shared__ uint32_t s_sum[LF_WARPS];
    const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5;
    const int warp = blockIdx.x * LF_WARPS + wb;
    // the starts before this block: all counts before it, by all threads
    uint32_t sum = 0;
    for (int j = threadIdx.x; j < blockIdx.x * LF_WARPS; j += LF_THREADS) sum += counts[j];
    sum = __reduce_add_sync(FULL, sum);
    if (lane == 0) s_sum[wb] = sum;
    __syncthreads();
    uint32_t o = 0;
#pragma unroll
    for (int w = 0; w < LF_WARPS; ++w) o += s_sum[w];
    for (int w = 0; w < wb; ++w) o += counts[blockIdx.x * LF_WARPS + w];
    const int64_t base = (int64_t)warp * (32 * windows);
    const unsigned lt = (1u << lane) - 1u;
    unsigned mine = 0;
    for (int w = 0; w < windows && base + 32 * (int64_t)w < n; ++w) {
        if ((w & 31) == 0) {  // the next 32 words, one per lane
            const int64_t at = (base >> 5) + w + lane;
            mine = w + lane < windows && 32 * at < n ? words[at] : 0u;
        }
        const unsigned word = __shfl_sync(FULL, mine, w & 31);
        if (!word) continue;
        const int64_t i = base + 32 * w + lane;
        if ((word >> lane) & 1u) {
            const uint32_t l = o + __popc(word & lt);
            const uint64_t k = (uint64_t)keys[i];
            leafr[l].x = (int32_t)i;
            lkey[l] = k;
            if (linst) linst[l] = (int32_t)(k >> id_shift);
            if (l > 0) leafr[l - 1].y = (int32_t)((uint32_t)i | (pdense && pdense[i - 1] == 2 ? 0x80000000u : 0u));
        }
        o += __popc(word);
    }
    // the warp of the last position: the last leaf's end and the number of leaves
    if (lane == 0 && base < n && base + 32 * (int64_t)windows >= n) {
        leafr[o - 1].y = (int32_t)((uint32_t)n | (pdense && pdense[n - 1] == 2 ? 0x80000000u : 0u));
        ctrl[CTRL_M] = o;
    }
}

// Higher block summaries: level k (k >= 2) entry j is the union of level-1
// entries [32^(k-1) j, 32^(k-1) (j + 1)), i.e. of 32^k consecutive leaves;
// the levels follow each other in `sum` (level 1 first; sizes and count as
// sum_level_size / sum_levels_entries). One warp per entry, reading level 1
// directly, so no level waits for another.
template <int D>
__global__ void k_box_levels(const uint32_t* __restrict__ ctrl, typename Traits<D>::Box* __restrict__ sum)
{
    stage_begin(ctrl);
    using T = Traits<D>;
    const int lane = threadIdx.x & 31;
    const int64_t m = ctrl[CTRL_M];
    if (m <= 1) return;
    const int64_t n1 = sum_level_size(m, 1);
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int64_t off = n1;   // start of level 2
    int64_t span = 32;  // level-1 entries per entry of level k
    for (int k = 2; k <= SUM_LEVELS && sum_level_size(m, k - 1) > SUM_DIRECT; ++k, span <<= 5) {
        const int64_t nk = sum_level_size(m, k);
        for (int64_t j = warp; j < nk; j += nwarps) {
            typename T::Box b = T::empty_box();
            const int64_t e0 = j * span, e1 = min(e0 + span, n1);
            for (int64_t i = e0 + lane; i < e1; i += 32) T::merge(b, sum[i]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) T::merge(b, T::shfl_xor(b, o));
            if (lane == 0) sum[off + j] = b;
        }
        off += nk;
    }
}

// ---------------------------------------------------------------------------
// K7: Karras (2012) LBVH topology. For internal node i the direction, the far
// end of its range and the split come from the common-prefix length delta of
// the sorted leaf keys; equal keys are told apart by the leaf index.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int kdelta(const uint64_t* k, int64_t m, int64_t i, int64_t j)
{
    if (j < 0 || j >= m) return -1;
    const uint64_t a = k[i], b = k[j];
    if (a != b) return __clzll((long long)(a ^ b));
    return 64 + __clz((int)((uint32_t)i ^ (uint32_t)j));
}

__device__ __forceinline__ void karras(const uint64_t* lkey, int64_t m, int4* __restrict__ nmeta,
                                       int2* __restrict__ child_out, int2* __restrict__ range_out,
                                       int32_t* __restrict__ first_out, unsigned block, unsigned blocks)
{
    for (int64_t i = block * (int64_t)blockDim.x + threadIdx.x; i < m - 1; i += (int64_t)blocks * blockDim.x) {
        const int d = (kdelta(lkey, m, i, i + 1) - kdelta(lkey, m, i, i - 1)) > 0 ? 1 : -1;
        const int dmin = kdelta(lkey, m, i, i - d);
        int64_t lmax = 2;
        while (kdelta(lkey, m, i, i + lmax * d) > dmin) lmax <<= 1;
        int64_t l = 0;
        for (int64_t t = lmax >> 1; t >= 1; t >>= 1)
            if (kdelta(lkey, m, i, i + (l + t) * d) > dmin) l += t;
        const int64_t j = i + l * d;
        const int dnode = kdelta(lkey, m, i, j);
        int64_t s = 0, t = l;
        do {
            t = (t + 1) >> 1;
            if (kdelta(lkey, m, i, i + (s + t) * d) > dnode) s += t;
        } while (t > 1);
        const int64_t gamma = i + s * d + (d < 0 ? -1 : 0);
        const int64_t first = i < j ? i : j, last = i < j ? j : i;
        const int32_t left = (int32_t)(first == gamma ? (m - 1) + gamma : gamma);
        const int32_t right = (int32_t)(last == gamma + 1 ? (m - 1) + gamma + 1 : gamma + 1);
        nmeta[i] = make_int4(left, right, (int32_t)gamma, (int32_t)last);
        if (child_out) child_out[i] = make_int2(left, right);
        if (range_out) range_out[i] = make_int2((int32_t)first, (int32_t)last);
        if (first_out) first_out[i] = (int32_t)first;
    }
}

// the topology alone (component entry point)
__global__ void k_karras(const uint64_t* __restrict__ lkey, int64_t m, int4* __restrict__ nmeta,
                         int2* __restrict__ child_out, int2* __restrict__ range_out)
{
    stage_begin(lkey);
    karras(lkey, m, nmeta, child_out, range_out, nullptr, blockIdx.x, gridDim.x);
}

// ---------------------------------------------------------------------------
// Leaf boxes: exact min/max of each leaf's points. A thread takes a leaf of
// at most TILE points (reading its contiguous points, four loads in flight;
// consecutive threads' ranges share cache lines); the boxes of the leaves
// larger than that (dense cells) come from the classification (dbox). Each
// warp also writes the union of its 32 leaves' boxes, the first level of the
// block summaries that the refit reads (sum1[w]: leaves 32 w .. 32 w + 31).
// The topology (K7) needs nothing of them, nor they of it: the odd blocks of
// the same launch do it. Both are chains of loads: one after the other in the
// same threads took 17 us on 16,384 blob points (12 on 1,000, 91 on 16.8M
// halos), this takes 10 (9, 76).
// ---------------------------------------------------------------------------
template <int D>
__global__ void k_leaf_boxes(const typename Traits<D>::Point* __restrict__ sp, const int2* __restrict__ leafr,
                             const uint32_t* __restrict__ ctrl, const typename Traits<D>::Box* __restrict__ dbox,
                             typename Traits<D>::Box* __restrict__ leafbox, typename Traits<D>::Box* __restrict__ sum1,
                             const uint64_t* __restrict__ lkey, int4* __restrict__ nmeta,
                             int2* __restrict__ range_out, int32_t* __restrict__ first_out, int shared_keys)
{
    stage_begin(sp, leafr, ctrl, dbox, lkey);
    using T = Traits<D>;
    const int lane = threadIdx.x & 31;
    const int64_t m = ctrl[CTRL_M];
    const unsigned block = blockIdx.x >> 1, blocks = gridDim.x >> 1;
    if (blockIdx.x & 1) {
        // the topology's searches are chains of dependent loads of keys: where all
        // of them fit, they are read from shared memory
        if (m <= shared_keys) {
            extern __shared__ __align__(16) unsigned char smem[];
            uint64_t* keys = reinterpret_cast<uint64_t*>(smem);
            if ((int64_t)block * blockDim.x >= m - 1) return;  // no node for this block
            for (int64_t i = threadIdx.x; i < m; i += blockDim.x) keys[i] = lkey[i];
            __syncthreads();
            karras(keys, m, nmeta, nullptr, range_out, first_out, block, blocks);
        } else {
            karras(lkey, m, nmeta, nullptr, range_out, first_out, block, blocks);
        }
        return;
    }
    const int64_t stride = (int64_t)blocks * blockDim.x;
    for (int64_t base = block * (int64_t)blockDim.x + threadIdx.x - lane; base < m; base += stride) {
        const int64_t l = base + lane;
        int s = 0, e = 0;
        if (l < m) {
            const int2 r = leafr[l];
            s = r.x;
            e = r.y & 0x7fffffff;
        }
        const bool small = l < m && e - s <= TILE;
        typename T::Box mine = T::empty_box();
        if (small) {
            typename T::Box b = T::empty_box();
            int j = s;
            if constexpr (D == 3) {
                // two 16-byte points per 256-bit load from an even index on
                if ((j & 1) && j < e) T::grow(b, sp[j++]);
#pragma unroll 4
                for (; j + 1 < e; j += 2) {
                    float4 p0, p1;
                    ldg256(&sp[j], p0, p1);
                    T::grow(b, p0);
                    T::grow(b, p1);
                }
            }
#pragma unroll 4
            for (; j < e; ++j) T::grow(b, sp[j]);
            leafbox[l] = b;
            mine = b;
        }
        if (l < m && !small) {
            mine = dbox[s >> 5];
            leafbox[l] = mine;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) T::merge(mine, T::shfl_xor(mine, o));
        if (lane == 0) sum1[base >> 5] = mine;
    }
}

// ---------------------------------------------------------------------------
// K8: refit. The box of a node is the exact min/max of the boxes of the
// leaves it covers, a contiguous range: node i covers leaves [first_i,
// last_i], its left child [first_i, split_i] and its right child [split_i +
// 1, last_i]. So each node's child boxes are computed directly from the leaf
// boxes, with no dependency between nodes (no climbing, counters or fences):
// min and max are exact in any order, so the boxes are the bottom-up ones
// bit for bit. A node covering at most RF_SMALL leaves is done by its thread;
// longer ranges by the whole warp, from the partial blocks at both ends of
// each summary level and the full blocks of the next one (at most 64 loads a
// lane per level).
// ---------------------------------------------------------------------------
constexpr int RF_SMALL = 32;

template <int D>
__device__ __forceinline__ typename Traits<D>::Box ld_box(const typename Traits<D>::Box* b)
{
    typename Traits<D>::Box r;
    if constexpr (sizeof(typename Traits<D>::Box) == 32) ld256(b, r.lo, r.hi);
    else r = *b;
    return r;
}

// union of leaf boxes a..b (inclusive), by the whole warp (all lanes, same a, b)
template <int D>
__device__ typename Traits<D>::Box range_box(const typename Traits<D>::Box* leafbox,
                                             const typename Traits<D>::Box* sum, int64_t m, int64_t a,
                                             int64_t b, int lane)
{
    using T = Traits<D>;
    typename T::Box acc = T::empty_box();
    const typename T::Box* arr = leafbox;
    int64_t off = 0, nk = sum_level_size(m, 1);
    for (int level = 0; a <= b && level <= SUM_LEVELS; ++level) {
        if (b - a < SUM_DIRECT || level == SUM_LEVELS) {
            for (int64_t j = a + lane; j <= b; j += 32) T::merge(acc, ld_box<D>(arr + j));
            break;
        }
        // the partial blocks at both ends at this level, the full blocks
        // between them at the next
        const int64_t ha = a + lane, tb = (b & ~(int64_t)31) + lane;
        if (ha <= (a | 31)) T::merge(acc, ld_box<D>(arr + ha));
        if (tb <= b) T::merge(acc, ld_box<D>(arr + tb));
        a = (a >> 5) + 1;
        b = (b >> 5) - 1;
        arr = sum + off;
        off += nk;
        nk = (nk + 31) >> 5;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) T::merge(acc, T::shfl_xor(acc, o));
    return acc;
}

template <int D>
__global__ void k_refit(uint32_t* __restrict__ ctrl, const int4* __restrict__ nmeta,
                        const int32_t* __restrict__ nfirst, const typename Traits<D>::Box* __restrict__ leafbox,
                        const typename Traits<D>::Box* __restrict__ sum, typename Traits<D>::Node* __restrict__ nodes)
{
    stage_begin(nmeta, nfirst, leafbox, sum);
    using T = Traits<D>;
    using Box = typename T::Box;
    const int lane = threadIdx.x & 31;
    const int64_t m = ctrl[CTRL_M];
    if (m <= 1) return;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // whole warps iterate together (the long ranges take all lanes)
    for (int64_t base = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; base < m - 1; base += stride) {
        const int64_t p = base + lane;
        int4 mt = make_int4(0, 0, 0, 0);
        int first = 0;
        bool ok = false;
        if (p < m - 1) {
            mt = nmeta[p];
            first = nfirst[p];
            // a range outside the leaves means a corrupt topology
            ok = first >= 0 && first <= mt.z && mt.z < mt.w && mt.w < m;
            if (!ok) atomicOr(&ctrl[CTRL_ERR], ERR_STACK);
        }
        const bool small = ok && mt.w - first < RF_SMALL;
        if (small) {
            Box L = T::empty_box(), R = T::empty_box();
            int j = first;
#pragma unroll 4
            for (; j <= mt.z; ++j) T::merge(L, ld_box<D>(leafbox + j));
#pragma unroll 4
            for (; j <= mt.w; ++j) T::merge(R, ld_box<D>(leafbox + j));
            nodes[p] = T::make_node(L, R, mt.x, mt.y, mt.z, mt.w);
        }
        unsigned big = __ballot_sync(FULL, ok && !small);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const int f = __shfl_sync(FULL, first, src), g = __shfl_sync(FULL, mt.z, src),
                      w = __shfl_sync(FULL, mt.w, src);
            const Box L = range_box<D>(leafbox, sum, m, f, g, lane);
            const Box R = range_box<D>(leafbox, sum, m, (int64_t)g + 1, w, lane);
            if (lane == src) nodes[p] = T::make_node(L, R, mt.x, mt.y, mt.z, mt.w);
        }
    }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
cudaError_t launch_density_estimate(const float* points, int64_t n, int dim, const GridParams* g, int min_pts,
                                   float auto_fraction, float auto_occupancy, const EstBuffers& eb, uint32_t* ctrl,
                                   cudaStream_t s)
{
    cudaError_t e;
    if ((e = cudaMemsetAsync(eb.table, 0xff, sizeof(unsigned long long) * EST_SLOTS, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(eb.counts, 0, sizeof(uint32_t) * EST_SLOTS, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(eb.result, 0, 4 * sizeof(uint32_t), s)) != cudaSuccess) return e;
    const int smp = n < EST_SAMPLES ? (int)n : EST_SAMPLES;
    const int64_t stride = n > (int64_t(1) << 22) ? n >> 22 : 1;
    int64_t gb = (n / stride + 255) / 256;
    if (gb > 152 * 4) gb = 152 * 4;
#define EST_LAUNCH(D)                                                                      \
    do {                                                                                   \
        launch(k_est_insert<D>, 1, 1024, 0, s, points, n, smp, g, ctrl, eb.table, eb.slot);   \
        launch(k_est_count<D>, (unsigned)gb, 256, 0, s, points, n, stride, g, ctrl, eb.table, eb.counts); \
    } while (0)
    GBD_DIM_SWITCH(dim, EST_LAUNCH)
#undef EST_LAUNCH
    launch(k_est_result, 1, 1024, 0, s, eb.slot, smp, eb.counts, n, stride, min_pts, auto_fraction, auto_occupancy,
                                    eb.result, ctrl);
    note_launches(3);
    return cudaGetLastError();
}

static inline unsigned grid_for(int64_t work, int threads, int max_blocks)
{
    int64_t b = (work + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > max_blocks) b = max_blocks;
    return (unsigned)b;
}

void launch_bounds(const float* pts, int64_t n, int dim, uint32_t* ctrl, const BoundsExtra& x, cudaStream_t s)
{
#define BOUNDS_LAUNCH(D)                                                                            \
    launch(k_bounds<D>, grid_for(n * D, bounds_threads<D>(), 152 * 8), bounds_threads<D>(), 0, s, pts, n, ctrl, x)
    GBD_DIM_SWITCH(dim, BOUNDS_LAUNCH)
#undef BOUNDS_LAUNCH
    note_launches(1);
}

void launch_run_begin(uint32_t* ctrl, int algo, cudaStream_t s)
{
    launch(k_run_begin, 1, 32, 0, s, ctrl, algo);
    note_launches(1);
}

void launch_morton32(const float* pts, int64_t n, int dim, const uint32_t* ctrl, int bits, uint32_t* keys,
                     uint32_t* vals, cudaStream_t s)
{
    const unsigned g = grid_for(n, 256, 152 * 16);
    if (dim == 3) launch(k_morton32<3>, g, 256, 0, s, pts, n, ctrl, bits, keys, vals);
    else launch(k_morton32<2>, g, 256, 0, s, pts, n, ctrl, bits, keys, vals);
    note_launches(1);
}

void launch_morton64(const float* pts, int64_t n, int dim, const uint32_t* ctrl, int bits, uint64_t* keys,
                     uint32_t* vals, cudaStream_t s)
{
    const unsigned g = grid_for(n, 256, 152 * 16);
#define M64_LAUNCH(D) launch(k_morton64<D>, g, 256, 0, s, pts, n, ctrl, bits, keys, vals)
    GBD_DIM_SWITCH(dim, M64_LAUNCH)
#undef M64_LAUNCH
    note_launches(1);
}

void launch_cellkey_packed(const float* pts, int64_t n, int dim, const GridParams* gp, const uint32_t* ctrl,
                           int idx_bits, int host_passes, uint64_t* words0, uint64_t* words1, cudaStream_t s)
{
    const unsigned g = grid_for(n, 256, 152 * 16);
#define CKP_LAUNCH(D) \
    launch(k_cellkey_packed<D>, g, 256, 0, s, pts, n, gp, ctrl, idx_bits, host_passes, words0, words1)
    GBD_DIM_SWITCH(dim, CKP_LAUNCH)
#undef CKP_LAUNCH
    note_launches(1);
}

void launch_gather_packed(const float* pts, const uint64_t* words, int64_t n, int dim, int idx_bits, void* sp,
                          uint32_t* perm, uint64_t* keys, const uint32_t* ctrl, cudaStream_t s)
{
    const unsigned g = grid_for((n + 1) / 2, 256, 152 * 16);
    const bool a16 = (reinterpret_cast<uintptr_t>(pts) & 15) == 0;
#define GP_LAUNCH(D)                                                                                          \
    do {                                                                                                      \
        auto* spd = static_cast<typename Traits<D>::Point*>(sp);                                              \
        if (a16) launch(k_gather_packed<D, true>, g, 256, 0, s, pts, words, n, idx_bits, spd, perm, keys, ctrl);  \
        else launch(k_gather_packed<D, false>, g, 256, 0, s, pts, words, n, idx_bits, spd, perm, keys, ctrl);    \
    } while (0)
    GBD_DIM_SWITCH(dim, GP_LAUNCH)
#undef GP_LAUNCH
    note_launches(1);
}

void launch_morton_generic(const float* pts, int64_t n, int dim, const GridParams& gp, uint64_t* out, cudaStream_t s)
{
    const unsigned g = grid_for(n, 256, 152 * 16);
    if (dim == 3) launch(k_morton_generic<3>, g, 256, 0, s, pts, n, gp, out);
    else launch(k_morton_generic<2>, g, 256, 0, s, pts, n, gp, out);
    note_launches(1);
}

void launch_gather(const float* pts, const uint32_t* perm, int64_t n, int dim, void* sp, const uint32_t* ctrl,
                   int algo, cudaStream_t s)
{
    const unsigned g = grid_for(n, 256, 152 * 16);
#define GATHER_LAUNCH(D) \
    launch(k_gather<D>, g, 256, 0, s, pts, perm, n, static_cast<typename Traits<D>::Point*>(sp), ctrl, algo)
    GBD_DIM_SWITCH(dim, GATHER_LAUNCH)
#undef GATHER_LAUNCH
    note_launches(1);
}

// Leaves of n sorted keys: records and keys, and m into ctrl
template <typename K>
cudaError_t launch_leaves(const K* keys, const int32_t* dstart, const uint8_t* pdense, int64_t n, int id_shift,
                          const DenseBoxTemps& t, int2* leafr, uint64_t* lkey, int32_t* linst, uint32_t* ctrl, int algo,
                          cudaStream_t s)
{
    const int64_t per = (int64_t)LF_BLOCKS * LF_THREADS * 2;
    int64_t w2 = (n + per - 1) / per;
    if (w2 < LF_MIN_WINDOWS / 2) w2 = LF_MIN_WINDOWS / 2;
    const int windows = (int)(2 * w2);
    const unsigned g = (unsigned)((n + (int64_t)LF_THREADS * windows - 1) / ((int64_t)LF_THREADS * windows));
    launch(k_leaf_flags<K>, g, LF_THREADS, 0, s, keys, dstart, pdense, n, windows, id_shift, t.lf, t.lfc, ctrl, algo);
    launch(k_leaf_records<K>, g, LF_THREADS, 0, s, keys, pdense, n, windows, id_shift, t.lf, t.lfc, leafr, lkey, linst, ctrl,
                                               algo);
    note_launches(2);
    return cudaGetLastError();
}

void launch_dense_classify(const uint64_t* keys, const void* sp, int64_t n, int dim, int min_pts, float e2,
                           const int32_t* mps, const float* e2s, int lb, const DenseBoxTemps& t, uint32_t* ctrl,
                           int algo, cudaStream_t s)
{
    int64_t steps = (n + (int64_t)152 * 16 * CELL_THREADS - 1) / ((int64_t)152 * 16 * CELL_THREADS);
    if (steps > CELL_STEPS) steps = CELL_STEPS;
    const unsigned g = grid_for(n, (int)steps * CELL_THREADS, 152 * 16);
#define DC_LAUNCH(D)                                                                                              \
    launch(k_dense_classify<D>, g, CELL_THREADS, 0, s, keys, static_cast<const typename Traits<D>::Point*>(sp), n,     \
                                                   min_pts, e2, mps, e2s, lb, t.pdense, t.dstart,                  \
                                                   static_cast<typename Traits<D>::Box*>(t.dbox), ctrl, algo,       \
                                                   (int)steps)
    GBD_DIM_SWITCH(dim, DC_LAUNCH)
#undef DC_LAUNCH
    note_launches(1);
}

cudaError_t launch_densebox_leaves(const uint64_t* keys, const void* sp, int64_t n, int dim, int min_pts, float e2,
                                   const DenseBoxTemps& t, int2* leafr, uint64_t* lkey, uint32_t* ctrl,
                                   cudaStream_t s)
{
    const int A = DBSCAN_ALGO_DENSEBOX;
    launch_dense_classify(keys, sp, n, dim, min_pts, e2, nullptr, nullptr, 64, t, ctrl, A, s);
    return launch_leaves<uint64_t>(keys, t.dstart, t.pdense, n, 64, t, leafr, lkey, nullptr, ctrl, A, s);
}

// Leaves of a batch: keys carry the instance in their bits from id_shift up;
// tiles never cross instances. pdense/dstart come from the batch's dense-cell
// classification (null for FDBSCAN).
cudaError_t launch_batch_leaves(const uint64_t* keys, int64_t n, int id_shift, const DenseBoxTemps& t, int2* leafr,
                                uint64_t* lkey, int32_t* linst, uint32_t* ctrl, cudaStream_t s)
{
    return launch_leaves<uint64_t>(keys, t.dstart, t.pdense, n, id_shift, t, leafr, lkey, linst, ctrl, -1, s);
}

cudaError_t launch_tile_leaves(const uint32_t* keys32, int64_t n, const DenseBoxTemps& t, int2* leafr,
                               uint64_t* lkey, uint32_t* ctrl, cudaStream_t s)
{
    return launch_leaves<uint32_t>(keys32, nullptr, nullptr, n, 64, t, leafr, lkey, nullptr, ctrl,
                                   DBSCAN_ALGO_FDBSCAN, s);
}

cudaError_t launch_tile_leaves64(const uint64_t* keys, int64_t n, const DenseBoxTemps& t, int2* leafr,
                                 uint64_t* lkey, uint32_t* ctrl, cudaStream_t s)
{
    return launch_leaves<uint64_t>(keys, nullptr, nullptr, n, 64, t, leafr, lkey, nullptr, ctrl, DBSCAN_ALGO_FDBSCAN,
                                   s);
}

void launch_lbvh(const void* sp, int dim, const int2* leafr, const uint64_t* lkey, const void* dbox, int64_t m_cap,
                 uint32_t* ctrl, int4* nmeta, int32_t* nfirst, void* leafbox, void* nsum, void* nodes, cudaStream_t s,
                 int2* range_out)
{
    const unsigned g = grid_for(m_cap, 256, 152 * 16);
    const unsigned gl = grid_for(sum_levels_entries(m_cap) * 32, 256, 152 * 4);
    // leaf keys that a block of the topology takes into shared memory: in runs
    // of up to 64K points, which seldom have more tiles than that; larger runs
    // keep the shared memory free for more blocks
    const int keys = m_cap <= (1 << 16) ? (int)std::min<int64_t>(m_cap, 4096) : 0;
    // (the levels from 2 on: none while level 1 is read directly)
    const bool levels = sum_level_size(m_cap, 1) > SUM_DIRECT;
#define LB_LAUNCH(D)                                                                                                  \
    do {                                                                                                              \
        using Bx = typename Traits<D>::Box;                                                                           \
        launch(k_leaf_boxes<D>, 2 * g, 256, sizeof(uint64_t) * keys, s, static_cast<const typename Traits<D>::Point*>(sp), leafr, ctrl, \
                                          static_cast<const Bx*>(dbox), static_cast<Bx*>(leafbox),                    \
                                          static_cast<Bx*>(nsum), lkey, nmeta, range_out, nfirst, keys);      \
        if (levels) launch(k_box_levels<D>, gl, 256, 0, s, ctrl, static_cast<Bx*>(nsum));                                 \
    } while (0)
    GBD_DIM_SWITCH(dim, LB_LAUNCH)
#undef LB_LAUNCH
#define RF_LAUNCH(D)                                                                                         \
    launch(k_refit<D>, g, 256, 0, s, ctrl, nmeta, nfirst, static_cast<typename Traits<D>::Box*>(leafbox),          \
                                 static_cast<const typename Traits<D>::Box*>(nsum),                            \
                                 static_cast<typename Traits<D>::Node*>(nodes))
    GBD_DIM_SWITCH(dim, RF_LAUNCH)
#undef RF_LAUNCH
    note_launches(levels ? 3 : 2);
}

void launch_karras_only(const uint64_t* lkey, int64_t m, int4* nmeta, int2* child_out,
                        int2* range_out, cudaStream_t s)
{
    launch(k_karras, grid_for(m, 256, 152 * 16), 256, 0, s, lkey, m, nmeta, child_out, range_out);
    note_launches(1);
}

}  // namespace gbd
