// Adaptive assignment of the occupied voxels to n networks (Alg. 1 stage
// II, Sec. "Adaptive Radiance Fields Slimming and Fine-tuning"): network k
// takes the smallest unassigned voxel (lexicographic (z, y, x), i.e. the
// smallest linear index) as its anchor plus the s - 1 unassigned voxels
// nearest to it (squared distance in voxel units, ties to the smaller linear
// index), s = S / n; the last network takes what remains.
//
// The networks are built one after the other (each depends on the voxels
// the earlier ones took), so what counts is the latency of one network.  Two
// forms:
//
// k_assign_bricks (small networks of voxels that lie together; the line is
// assign_from_bricks): one cluster of 8 blocks builds every network in one
// launch.  The unassigned voxels are kept in lists by 8^3 brick (each block owns
// every eighth brick).  Per network: a
// histogram of the bricks' largest distance to the anchor, weighted by their
// voxels, bounds the distance of the last voxel wanted; only bricks that reach
// below that bound are candidates; a histogram of their voxels' squared
// distances narrows the last voxel's key to one bin, and that bin's keys are
// ranked directly.  The candidates' keys stay in registers between these steps
// (up to four per thread; else they are formed again, a thread per brick of a
// few voxels, a warp per brick of many), histograms are pushed into every block's copy
// through distributed shared memory, so a network costs four cluster barriers
// and a few L2 latencies, and touches about as many voxels as it takes (instead
// of every unassigned voxel once per launch of the general form).
//
// The general form, for larger networks and scattered voxels: per network
//   k_hist_select  per digit of the key (squared distance << 27 | rank), a
//                  histogram of the candidates matching the digits fixed so
//                  far (shared-memory bins, then global atomics);
//                  the block that finishes last picks the bin holding the
//                  wanted rank, growing the key prefix by one digit (4
//                  digits of 12 bits; 5 where squared distances reach 2^21)
//   k_take_anchor  every unassigned voxel whose key is <= the selected key
//                  joins the network; the block that finishes last finds the
//                  next network's anchor (the first unassigned voxel from a
//                  cursor; k_anchor for the first network)
// Five or six launches per network, with no waiting between blocks: the serial
// parts run in whichever block finishes last (a counter of finished blocks).
// Keys are unique (the rank is part of them), so exactly s voxels are taken.
// All state stays on the device: no host synchronisation per network.
#include <cooperative_groups.h>

#include "internal.cuh"

namespace cg = cooperative_groups;

namespace roam {

namespace {

constexpr int kDigitBits = 12;
constexpr int kBins = 1 << kDigitBits;
constexpr int kRankBits = 27;               // ranks below 2^27 (512^3 grids hold < 2^27 occupied voxels)
constexpr uint16_t kFree = 0xffffu;

struct AssignState {
    uint32_t cursor;       // every rank before it is assigned
    uint32_t anchor;       // rank of the current anchor
    uint32_t ax, ay, az;   // its voxel coordinates
    uint32_t rank_left;    // rank still to locate within the current prefix
    unsigned long long prefix;   // key digits fixed so far
    uint32_t status;
    uint32_t done;               // blocks finished in the current launch (the last one does the serial part)
};

__global__ void k_occupied_list(const uint2 *cells, int64_t n_words, uint32_t *vox)
{
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < n_words;
         w += (int64_t)gridDim.x * blockDim.x) {
        const uint2 cell = cells[w];
        uint32_t word = cell.x, r = cell.y;
        while (word) {
            const int b = __ffs(word) - 1;
            vox[r++] = (uint32_t)(w * 32 + b);
            word &= word - 1u;
        }
    }
}

// the first unassigned voxel from the cursor: the new anchor (one block)
__device__ void find_anchor(const uint16_t *field, uint32_t S, const uint32_t *vox, int gx, int gy, AssignState *st,
                            uint32_t s_minus_1)
{
    __shared__ uint32_t found;
    if (threadIdx.x == 0) found = 0xffffffffu;
    __syncthreads();
    for (uint32_t base = st->cursor; base < S; base += blockDim.x) {
        const uint32_t i = base + threadIdx.x;
        if (i < S && __ldcg(&field[i]) == kFree) atomicMin(&found, i);     // past L1: other blocks just wrote
        __syncthreads();
        if (found != 0xffffffffu) break;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const uint32_t a = found;
        st->cursor = a;
        st->anchor = a;
        if (a < S) {
            const uint32_t v = vox[a];
            st->ax = v % (uint32_t)gx;
            st->ay = (v / (uint32_t)gx) % (uint32_t)gy;
            st->az = v / ((uint32_t)gx * (uint32_t)gy);
        } else {
            st->status = 1u;
        }
        st->rank_left = s_minus_1;
        st->prefix = 0ull;
    }
}

__global__ void __launch_bounds__(1024) k_anchor(const uint16_t *field, uint32_t S, const uint32_t *vox, int gx,
                                                 int gy, AssignState *st, uint32_t s_minus_1)
{
    find_anchor(field, S, vox, gx, gy, st, s_minus_1);
}

// true in the one block that finishes last (after every block's global
// writes of this launch are visible)
__device__ __forceinline__ bool last_block(AssignState *st)
{
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&st->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last) __threadfence();
    return last;
}

__device__ __forceinline__ unsigned long long key_of(const AssignState &st, uint32_t v, uint32_t rank, int gx, int gy)
{
    const int x = (int)(v % (uint32_t)gx), y = (int)((v / (uint32_t)gx) % (uint32_t)gy),
              z = (int)(v / ((uint32_t)gx * (uint32_t)gy));
    const long long dx = x - (int)st.ax, dy = y - (int)st.ay, dz = z - (int)st.az;
    const unsigned long long d2 = (unsigned long long)(dx * dx + dy * dy + dz * dz);
    return (d2 << kRankBits) | rank;
}

// Histogram of the keys' digit at `shift` (`first`: the most significant) over
// the keys matching the prefix (shared-memory bins, then global atomics); then,
// in the block that finishes last, the select: the bin holding rank_left extends
// the prefix by one digit (512 threads, 8 bins each), and the histogram is cleared.
__global__ void __launch_bounds__(512) k_hist_select(const uint16_t *field, uint32_t S, const uint32_t *vox, int gx,
                                                     int gy, AssignState *st, int shift, bool first, uint32_t *hist)
{
    __shared__ uint32_t sh[kBins];
    for (int b = threadIdx.x; b < kBins; b += blockDim.x) sh[b] = 0u;
    __syncthreads();
    {
        const AssignState sv = *st;
        // eight candidates per thread per round, their loads issued together
        // (one dependent load after another per voxel would leave the SMs
        // waiting on L2 latency)
        constexpr int kU = 8;
        const uint32_t stride = gridDim.x * blockDim.x;
        for (uint32_t i0 = sv.cursor + blockIdx.x * blockDim.x + threadIdx.x; i0 < S; i0 += kU * stride) {
            uint16_t fv[kU];
            uint32_t vv[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const uint32_t i = i0 + (uint32_t)u * stride;
                fv[u] = i < S ? field[i] : (uint16_t)0;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const uint32_t i = i0 + (uint32_t)u * stride;
                vv[u] = fv[u] == kFree && i < S ? vox[i] : 0u;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const uint32_t i = i0 + (uint32_t)u * stride;
                if (fv[u] != kFree || i >= S) continue;
                const unsigned long long k = key_of(sv, vv[u], i, gx, gy);
                if (!first && (k >> (shift + kDigitBits)) != sv.prefix) continue;
                atomicAdd(&sh[(k >> shift) & (kBins - 1)], 1u);
            }
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kBins; b += blockDim.x)
        if (sh[b]) atomicAdd(&hist[b], sh[b]);
    if (!last_block(st)) return;
    // select: the bin holding rank_left (hist read from L2, where the atomics landed)
    const int t = threadIdx.x;
    const uint32_t want = st->rank_left;
    uint32_t c[8], sum = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) { c[q] = __ldcg(&hist[8 * t + q]); sum += c[q]; }
    uint32_t *part = sh;                      // reuse: the block's histogram is flushed
    __syncthreads();
    part[t] = sum;
    __syncthreads();
    for (int o = 1; o < 512; o <<= 1) {
        const uint32_t v = t >= o ? part[t - o] : 0u;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    const uint32_t before = t > 0 ? part[t - 1] : 0u;
    if (want >= before && want < part[t]) {
        uint32_t acc = before;
        for (int q = 0; q < 8; ++q) {
            if (want < acc + c[q]) {
                st->prefix = (st->prefix << kDigitBits) | (unsigned long long)(8 * t + q);
                st->rank_left = want - acc;
                break;
            }
            acc += c[q];
        }
    }
    if (t == 511 && want >= part[511]) st->status = 1u;      // fewer candidates than asked for
#pragma unroll
    for (int q = 0; q < 8; ++q) hist[8 * t + q] = 0u;
    if (t == 0) st->done = 0u;
}

// every unassigned voxel whose key is <= the selected key joins network
// `net`; then, in the block that finishes last, the next network's anchor
__global__ void __launch_bounds__(1024) k_take_anchor(uint16_t *field, uint32_t S, const uint32_t *vox, int gx, int gy,
                                                      AssignState *st, uint16_t net, uint32_t s_minus_1)
{
    {
        const AssignState sv = *st;
        const unsigned long long thr = sv.prefix;
        for (uint32_t i = sv.cursor + blockIdx.x * blockDim.x + threadIdx.x; i < S; i += gridDim.x * blockDim.x) {
            if (field[i] != kFree) continue;
            if (key_of(sv, vox[i], i, gx, gy) <= thr) field[i] = net;
        }
    }
    if (!last_block(st)) return;
    if (threadIdx.x == 0) st->done = 0u;
    find_anchor(field, S, vox, gx, gy, st, s_minus_1);
}

__global__ void k_take_rest(uint16_t *field, uint32_t S, uint16_t net)
{
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < S; i += gridDim.x * blockDim.x)
        if (field[i] == kFree) field[i] = net;
}

// Voxels in rank order: neighbours mostly belong to one network, so a warp
// reduces each network it meets and its first lane updates the box (one lane
// per voxel updating it directly took 328 us of a 500,000-voxel assignment:
// six atomics per voxel on a few hundred addresses).
__global__ void k_boxes(const uint16_t *field, uint32_t S, const uint32_t *vox, int gx, int gy, int32_t *boxes)
{
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); i0 < S; i0 += stride) {
        const uint32_t i = i0 + (threadIdx.x & 31u);
        const bool in = i < S;
        const uint32_t v = in ? vox[i] : 0u, f = in ? field[i] : 0u;
        const int x = (int)(v % (uint32_t)gx), y = (int)((v / (uint32_t)gx) % (uint32_t)gy),
                  z = (int)(v / ((uint32_t)gx * (uint32_t)gy));
        unsigned todo = __ballot_sync(0xffffffffu, in);
        while (todo) {
            const uint32_t lead = __shfl_sync(0xffffffffu, f, __ffs(todo) - 1);
            const bool mine = in && f == lead;
            todo &= ~__ballot_sync(0xffffffffu, mine);
            const int lx = __reduce_min_sync(0xffffffffu, mine ? x : 0x7fffffff);
            const int ly = __reduce_min_sync(0xffffffffu, mine ? y : 0x7fffffff);
            const int lz = __reduce_min_sync(0xffffffffu, mine ? z : 0x7fffffff);
            const int hx = __reduce_max_sync(0xffffffffu, mine ? x + 1 : 0);
            const int hy = __reduce_max_sync(0xffffffffu, mine ? y + 1 : 0);
            const int hz = __reduce_max_sync(0xffffffffu, mine ? z + 1 : 0);
            if ((threadIdx.x & 31u) == 0) {
                int32_t *b = boxes + 6 * (int64_t)lead;
                atomicMin(&b[0], lx); atomicMin(&b[1], ly); atomicMin(&b[2], lz);
                atomicMax(&b[3], hx); atomicMax(&b[4], hy); atomicMax(&b[5], hz);
            }
        }
    }
}

__global__ void k_boxes_init(int32_t *boxes, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        boxes[6 * i + 0] = boxes[6 * i + 1] = boxes[6 * i + 2] = 0x7fffffff;
        boxes[6 * i + 3] = boxes[6 * i + 4] = boxes[6 * i + 5] = 0;
    }
}

// ---- networks from brick lists ---------------------------------------------

constexpr int kCluster = 8;
constexpr int kAT = 1024;                   // threads per block
constexpr int kABins = 1024;                // one per thread
constexpr int kListMax = 1024;              // keys ranked directly
constexpr int kCandMax = 1536;              // candidate bricks of one block kept in shared memory
constexpr int kVox = 4;                     // ... and voxels per thread kept in registers

struct BrickLists {
    uint32_t *n;           // [2]: bricks with voxels, voxels
    uint32_t *coord;       // [NB] bx | by << 8 | bz << 16 (grids are at most 2048^3: 256 bricks per axis)
    uint32_t *count;       // [NB] unassigned voxels
    uint32_t *start;       // [NB] first entry
    uint32_t *spill;       // [NB + 8] candidate bricks past a block's table (ceil(NB / 8) words per block)
    uint32_t *rank;        // [S] ranks, brick after brick
    uint16_t *loc;         // [S] voxel within its brick: x | y << 3 | z << 6
};

// one warp per brick: its occupied voxels, appended to the lists (bricks in
// any order: the networks do not depend on it)
__global__ void __launch_bounds__(256) k_brick_lists(const uint2 *__restrict__ cells, int gx, int gy, int gz, BrickLists L)
{
    const int bx_n = gx >> 3, by_n = gy >> 3, bz_n = gz >> 3, wpr = gx >> 5, lane = threadIdx.x & 31;
    const uint32_t n_b = (uint32_t)bx_n * by_n * bz_n;
    for (uint32_t b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; b < n_b; b += (gridDim.x * blockDim.x) >> 5) {
        const int bx = (int)(b % bx_n), by = (int)((b / bx_n) % by_n), bz = (int)(b / ((uint32_t)bx_n * by_n));
        uint32_t m[2], base[2];
        int own = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = lane + 32 * h, y = by * 8 + (r & 7), z = bz * 8 + (r >> 3);     // row r of the brick
            const uint32_t w = ((uint32_t)z * gy + y) * wpr + (bx >> 2);
            const uint2 cell = cells[w];
            const uint32_t sh = (uint32_t)(bx & 3) * 8;
            m[h] = (cell.x >> sh) & 0xffu;
            base[h] = cell.y + (uint32_t)__popc(cell.x & ((1u << sh) - 1u));
            own += __popc(m[h]);
        }
        int incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        if (total == 0) continue;
        uint32_t slot = 0, first = 0;
        if (lane == 0) {
            slot = atomicAdd(&L.n[0], 1u);
            first = atomicAdd(&L.n[1], (uint32_t)total);
            L.coord[slot] = (uint32_t)bx | (uint32_t)by << 8 | (uint32_t)bz << 16;
            L.count[slot] = (uint32_t)total;
            L.start[slot] = first;
        }
        first = __shfl_sync(0xffffffffu, first, 0);
        uint32_t at = first + (uint32_t)(incl - own);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t q = m[h], k = 0;
            while (q) {
                const uint32_t x = (uint32_t)__ffs(q) - 1u;
                L.rank[at] = base[h] + k;
                L.loc[at] = (uint16_t)(x | (uint32_t)(lane + 32 * h) << 3);
                ++at;
                ++k;
                q &= q - 1u;
            }
        }
    }
}

// inclusive scan of one value per thread over the block (scratch: 32 words)
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t *scratch)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    if (lane == 31) scratch[wid] = v;
    __syncthreads();
    if (wid == 0) {
        uint32_t s = scratch[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        scratch[lane] = s;
    }
    __syncthreads();
    if (wid > 0) v += scratch[wid - 1];
    return v;
}

__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kAT, 1)
    k_assign_bricks(uint16_t *field, uint32_t S, const uint32_t *vox, int gx, int gy, AssignState *st, BrickLists L,
                    int n, uint32_t per)
{
    cg::cluster_group cluster = cg::this_cluster();
    // a block's own histogram, and the cluster's sum of one (every block's copy)
    __shared__ uint32_t hist[kABins], sum[2][kABins], scratch[32];
    __shared__ unsigned long long list[kListMax];         // block 0's is the cluster's
    __shared__ uint32_t list_n, sel_bin, sel_before, sel_count;
    __shared__ unsigned long long thr_s, anchor_s, cand_s;
    // candidate bricks, and where each one's voxels start among the candidates'
    __shared__ uint32_t cand[kCandMax], cand_at[kCandMax], cand_kept[kCandMax];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster.block_rank(), n_bricks = L.n[0];
    uint32_t *const spill = L.spill + rank * ((n_bricks + kCluster - 1) / kCluster);

    hist[tid] = sum[0][tid] = sum[1][tid] = 0u;
    if (tid == 0) {
        list_n = 0u;
        cand_s = 0ull;
    }
    cluster.sync();
    // adds the block's histogram to every block's copy of the cluster's sum h
    // (a push: after the cluster's barrier nothing is read across blocks), and clears it
    auto share = [&](uint32_t *h) {
        __syncthreads();
        const uint32_t v = hist[tid];
        if (v) {
#pragma unroll
            for (int q = 0; q < kCluster; ++q) atomicAdd(&cluster.map_shared_rank(h, q)[tid], v);
            hist[tid] = 0u;
        }
        cluster.sync();
    };
    // the bin that holds item `want` (0-based) of the summed histogram, which is
    // cleared; every block finds the same.  False: fewer items.
    auto select = [&](uint32_t *h, uint32_t want) -> bool {
        if (tid == 0) sel_bin = 0xffffffffu;
        const uint32_t c = h[tid], incl = block_scan(c, scratch);
        h[tid] = 0u;
        if (want >= incl - c && want < incl) {
            sel_bin = (uint32_t)tid;
            sel_before = incl - c;
            sel_count = c;
        }
        __syncthreads();
        return sel_bin != 0xffffffffu;
    };

    uint32_t cursor = 0;
    for (int net = 0; net + 1 < n; ++net) {
        // ---- anchor: the first unassigned rank from the cursor (every block looks) ----
        for (uint32_t base = cursor;; base += kAT) {
            if (tid == 0) anchor_s = ~0ull;
            __syncthreads();
            const uint32_t i = base + (uint32_t)tid;
            const uint32_t v = i < S ? __ldg(&vox[i]) : 0u;
            const unsigned m = __ballot_sync(0xffffffffu, i < S && __ldcg(&field[i]) == kFree);
            if (m && lane == __ffs(m) - 1) atomicMin(&anchor_s, (unsigned long long)i << 32 | v);
            __syncthreads();
            if (anchor_s != ~0ull || base + kAT >= S) break;
            __syncthreads();
        }
        const unsigned long long found = anchor_s;
        if (found == ~0ull) {                               // (the same in every block)
            if (rank == 0 && tid == 0) st->status = 1u;
            break;
        }
        cursor = (uint32_t)(found >> 32);
        const uint32_t av = (uint32_t)found;
        const int ax = (int)(av % (uint32_t)gx), ay = (int)((av / (uint32_t)gx) % (uint32_t)gy),
                  az = (int)(av / ((uint32_t)gx * (uint32_t)gy));
        // smallest and largest squared distance of a brick's voxels to the anchor
        auto reach = [&](uint32_t c, uint32_t &lo, uint32_t &hi) {
            lo = hi = 0u;
            const int b[3] = {(int)(c & 255u) * 8 - ax, (int)((c >> 8) & 255u) * 8 - ay, (int)((c >> 16) & 255u) * 8 - az};
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int d0 = b[q], d1 = b[q] + 7;         // the range of the axis' difference
                const int far = max(abs(d0), abs(d1)), near = d0 > 0 ? d0 : (d1 < 0 ? -d1 : 0);
                lo += (uint32_t)(near * near);
                hi += (uint32_t)(far * far);
            }
        };
        auto dist_bin = [&](uint32_t d2) { return min((uint32_t)sqrtf((float)d2), (uint32_t)kABins - 1u); };

        // ---- the bound: voxels of bricks by their largest distance ----
        for (uint32_t b = rank + (uint32_t)tid * kCluster; b < n_bricks; b += kAT * kCluster) {
            const uint32_t c = L.count[b];
            if (!c) continue;
            uint32_t lo, hi;
            reach(L.coord[b], lo, hi);
            atomicAdd(&hist[dist_bin(hi)], c);
        }
        share(sum[0]);
        const bool enough = select(sum[0], per - 1u);
        if (!enough) {                                      // fewer voxels than asked for
            if (rank == 0 && tid == 0) st->status = 1u;
            break;
        }
        // squared distances below this hold the last voxel wanted (one more in
        // the root for the rounding of sqrtf; the last bin is open)
        const uint32_t root = sel_bin + 2u;
        const uint32_t bound = sel_bin == (uint32_t)kABins - 1u ? 0xffffffffu : root * root;
        // ---- candidate bricks, and the histogram of their voxels' distances ----
        const unsigned long long bound_key = (unsigned long long)bound << kRankBits;
        const int bits_d2 = bound == 0xffffffffu ? 24 : 32 - __clz(bound);      // (d2 < 3 * 2048^2 < 2^24)
        const int sh = max(0, bits_d2 - 10);
        for (uint32_t b = rank + (uint32_t)tid * kCluster; b < n_bricks; b += kAT * kCluster) {
            if (!L.count[b]) continue;
            uint32_t lo, hi;
            reach(L.coord[b], lo, hi);
            if (lo >= bound) continue;
            // its place in the table and its voxels' places, both in one counter
            const unsigned long long at = atomicAdd(&cand_s, 1ull << 32 | L.count[b]);
            const uint32_t q = (uint32_t)(at >> 32);
            if (q < (uint32_t)kCandMax) {
                cand[q] = b;
                cand_at[q] = (uint32_t)at;
                cand_kept[q] = 0u;
            } else {
                spill[q] = b;
            }
        }
        __syncthreads();
        const uint32_t nc = (uint32_t)(cand_s >> 32), nv = (uint32_t)cand_s;
        auto cand_of = [&](uint32_t q) { return q < (uint32_t)kCandMax ? cand[q] : spill[q]; };
        // a few voxels per thread: their keys stay in registers
        const bool few = nc <= (uint32_t)kCandMax && nv <= kVox * (uint32_t)kAT;
        unsigned long long vk[kVox];
        uint32_t vq[kVox];
        uint16_t vl[kVox];
        if (few) {
#pragma unroll
            for (int u = 0; u < kVox; ++u) {
                const uint32_t e = (uint32_t)(u * kAT + tid);
                vk[u] = ~0ull;
                if (e >= nv) continue;
                uint32_t q0 = 0, q1 = nc;                    // the last candidate at or before e
                while (q1 - q0 > 1) {
                    const uint32_t mid = (q0 + q1) / 2;
                    if (cand_at[mid] <= e) q0 = mid; else q1 = mid;
                }
                const uint32_t b = cand[q0], c = L.coord[b], at = L.start[b] + (e - cand_at[q0]);
                const uint32_t l = L.loc[at], r = L.rank[at];
                const int dx = (int)(c & 255u) * 8 - ax + (int)(l & 7u), dy = (int)((c >> 8) & 255u) * 8 - ay + (int)((l >> 3) & 7u),
                          dz = (int)((c >> 16) & 255u) * 8 - az + (int)(l >> 6);
                vk[u] = (unsigned long long)(uint32_t)(dx * dx + dy * dy + dz * dz) << kRankBits | r;
                vq[u] = q0;
                vl[u] = (uint16_t)l;
            }
        }
        // a brick's voxels as keys
        struct Brick {
            uint32_t n, first;
            int x, y, z;
        };
        auto open = [&](uint32_t b) {
            const uint32_t c = L.coord[b];
            return Brick{L.count[b], L.start[b], (int)(c & 255u) * 8 - ax, (int)((c >> 8) & 255u) * 8 - ay,
                         (int)((c >> 16) & 255u) * 8 - az};
        };
        auto key = [&](const Brick &o, uint32_t e) -> unsigned long long {
            const uint32_t l = L.loc[e];
            const int dx = o.x + (int)(l & 7u), dy = o.y + (int)((l >> 3) & 7u), dz = o.z + (int)(l >> 6);
            return (unsigned long long)(uint32_t)(dx * dx + dy * dy + dz * dz) << kRankBits | L.rank[e];
        };
        // else a thread goes over each of its block's candidates where these hold
        // a few voxels each, a warp where they hold many
        const bool sparse = nv < 6u * nc;
        auto each_key = [&](auto f) {
            if (few) {
#pragma unroll
                for (int u = 0; u < kVox; ++u)
                    if (vk[u] < bound_key) f(vk[u]);
            } else if (sparse) {
                for (uint32_t q = (uint32_t)tid; q < nc; q += kAT) {
                    const Brick o = open(cand_of(q));
                    for (uint32_t e = o.first; e < o.first + o.n; ++e) {
                        const unsigned long long k = key(o, e);
                        if (k < bound_key) f(k);
                    }
                }
            } else {
                for (uint32_t q = (uint32_t)warp; q < nc; q += kAT / 32) {
                    const Brick o = open(cand_of(q));
                    for (uint32_t e = (uint32_t)lane; e < o.n; e += 32) {
                        const unsigned long long k = key(o, o.first + e);
                        if (k < bound_key) f(k);
                    }
                }
            }
        };
        each_key([&](unsigned long long k) { atomicAdd(&hist[(uint32_t)(k >> (kRankBits + sh))], 1u); });
        share(sum[1]);
        uint32_t want = per - 1u;
        select(sum[1], want);
        want -= sel_before;
        // the wanted key lies in [lo_key, lo_key + 2^shift)
        int shift = sh + kRankBits;
        unsigned long long lo_key = (unsigned long long)sel_bin << shift;
        uint32_t left = sel_count;
        // ---- narrow until the bin's keys can be ranked directly (rarely needed) ----
        while (left > (uint32_t)kListMax) {
            cluster.sync();                                 // every block has read and cleared its sum
            const int ns = max(0, shift - 10);
            each_key([&](unsigned long long k) {
                if (k >= lo_key && (k - lo_key) >> shift == 0ull) atomicAdd(&hist[(uint32_t)((k - lo_key) >> ns)], 1u);
            });
            share(sum[1]);
            select(sum[1], want);
            want -= sel_before;
            lo_key += (unsigned long long)sel_bin << ns;
            shift = ns;
            left = sel_count;
            __syncthreads();
        }
        // ---- the bin's keys, in block 0's list ----
        {
            uint32_t *ln = cluster.map_shared_rank(&list_n, 0);
            unsigned long long *lp = cluster.map_shared_rank(list, 0);
            each_key([&](unsigned long long k) {
                if (k >= lo_key && (k - lo_key) >> shift == 0ull) {
                    const uint32_t at = atomicAdd(ln, 1u);
                    if (at < (uint32_t)kListMax) lp[at] = k;
                }
            });
        }
        cluster.sync();
        if (rank != 0 && (uint32_t)tid < left) list[tid] = cluster.map_shared_rank(list, 0)[tid];
        __syncthreads();
        if ((uint32_t)tid < left) {
            const unsigned long long k = list[tid];
            uint32_t below = 0;
#pragma unroll 4
            for (uint32_t q = 0; q < left; ++q) below += list[q] < k;
            if (below == want) thr_s = k;
        }
        __syncthreads();
        const unsigned long long thr = thr_s;
        // ---- take: keys up to the threshold join the network; each brick's list closes up ----
        if (few) {
            // (every entry was read above: the kept ones close up in any order)
#pragma unroll
            for (int u = 0; u < kVox; ++u) {
                if (vk[u] == ~0ull) continue;
                const uint32_t r = (uint32_t)vk[u] & ((1u << kRankBits) - 1u);
                if (vk[u] <= thr) {
                    __stcg(&field[r], (uint16_t)net);
                } else {
                    const uint32_t at = L.start[cand[vq[u]]] + atomicAdd(&cand_kept[vq[u]], 1u);
                    L.rank[at] = r;
                    L.loc[at] = vl[u];
                }
            }
            __syncthreads();
            for (uint32_t q = (uint32_t)tid; q < nc; q += kAT) L.count[cand[q]] = cand_kept[q];
        } else if (!sparse) {
            for (uint32_t q = (uint32_t)warp; q < nc; q += kAT / 32) {
                const uint32_t b = cand_of(q);
                const Brick o = open(b);
                uint32_t kept = 0;
                for (uint32_t e0 = 0; e0 < o.n; e0 += 32) {
                    const uint32_t e = o.first + e0 + (uint32_t)lane;
                    const bool in = e0 + (uint32_t)lane < o.n;
                    const uint32_t r = in ? L.rank[e] : 0u;
                    const uint16_t l = in ? L.loc[e] : (uint16_t)0;
                    const bool take = in && key(o, in ? e : o.first) <= thr;
                    const unsigned km = __ballot_sync(0xffffffffu, in && !take);
                    if (take) __stcg(&field[r], (uint16_t)net);
                    __syncwarp();
                    if (in && !take) {
                        const uint32_t at = o.first + kept + (uint32_t)__popc(km & ((1u << lane) - 1u));
                        L.rank[at] = r;
                        L.loc[at] = l;
                    }
                    __syncwarp();
                    kept += (uint32_t)__popc(km);
                }
                if (lane == 0) L.count[b] = kept;
            }
        } else {
            for (uint32_t q = (uint32_t)tid; q < nc; q += kAT) {
                const uint32_t b = cand_of(q);
                const Brick o = open(b);
                uint32_t kept = 0;
                for (uint32_t e = o.first; e < o.first + o.n; ++e) {
                    const uint32_t r = L.rank[e];
                    const uint16_t l = L.loc[e];
                    if (key(o, e) <= thr) {
                        __stcg(&field[r], (uint16_t)net);
                    } else {
                        L.rank[o.first + kept] = r;
                        L.loc[o.first + kept] = l;
                        ++kept;
                    }
                }
                L.count[b] = kept;
            }
        }
        __syncthreads();
        if (tid == 0) cand_s = 0ull;
        cluster.sync();                                     // the labels and lists are in place; block 0's list is read
        if (rank == 0 && tid == 0) list_n = 0u;
    }
    cluster.sync();                                         // no block leaves while others read its shared memory
}

}  // namespace

// state and histogram, then the lists
size_t assign_scratch_bytes(uint32_t S, int64_t n_bricks, bool lists)
{
    return sizeof(AssignState) + kBins * sizeof(uint32_t) + 16 +
           (lists ? (size_t)n_bricks * 16 + 4 * kCluster + (size_t)S * 6 : 0);
}

void launch_assign(const uint2 *cells, int64_t n_words, int gx, int gy, int gz, uint32_t S, int64_t n_bricks,
                   int n, bool lists, uint32_t *vox, uint16_t *field, int32_t *boxes, void *scratch, int n_sm,
                   cudaStream_t s)
{
    AssignState *st = reinterpret_cast<AssignState *>(scratch);
    uint32_t *hist = reinterpret_cast<uint32_t *>(reinterpret_cast<uint8_t *>(scratch) + sizeof(AssignState));
    // (16 more bytes: the lists' two counters)
    cudaMemsetAsync(scratch, 0, sizeof(AssignState) + kBins * sizeof(uint32_t) + 16, s);
    cudaMemsetAsync(field, 0xff, (size_t)S * sizeof(uint16_t), s);
    k_occupied_list<<<n_sm * 8, 256, 0, s>>>(cells, n_words, vox);
    const uint32_t per = S / (uint32_t)n;
    const int grid = n_sm * 4;
    if (n > 1 && lists) {
        const size_t nb = (size_t)n_bricks;
        BrickLists L;
        L.n = hist + kBins;
        L.coord = L.n + 4;
        L.count = L.coord + nb;
        L.start = L.count + nb;
        L.spill = L.start + nb;
        L.rank = L.spill + nb + kCluster;
        L.loc = reinterpret_cast<uint16_t *>(L.rank + S);
        k_brick_lists<<<n_sm * 8, 256, 0, s>>>(cells, gx, gy, gz, L);
        k_assign_bricks<<<kCluster, kAT, 0, s>>>(field, S, vox, gx, gy, st, L, n, per);
    } else if (n > 1) {
        // per network: a pass per digit (histogram, then the select in the block
        // that finishes last) and the take (then the next anchor, likewise);
        // 4 digits hold squared distances below 2^21, larger grids take 5
        const uint64_t far = (uint64_t)gx * gx + (uint64_t)gy * gy + (uint64_t)gz * gz;
        const int n_digits = far >> (4 * kDigitBits - kRankBits) ? 5 : 4;
        k_anchor<<<1, 1024, 0, s>>>(field, S, vox, gx, gy, st, per - 1u);
        for (int k = 0; k + 1 < n; ++k) {
            // one block per SM: fewer blocks flushing their shared histograms
            // (the first digits fall in a few bins, whose global atomics collide)
            for (int d = n_digits - 1; d >= 0; --d)
                k_hist_select<<<n_sm, 512, 0, s>>>(field, S, vox, gx, gy, st, d * kDigitBits, d == n_digits - 1, hist);
            k_take_anchor<<<grid, 1024, 0, s>>>(field, S, vox, gx, gy, st, (uint16_t)k, per - 1u);
        }
    }
    k_take_rest<<<grid, 256, 0, s>>>(field, S, (uint16_t)(n - 1));
    if (boxes) {
        k_boxes_init<<<(n + 255) / 256, 256, 0, s>>>(boxes, n);
        k_boxes<<<grid, 256, 0, s>>>(field, S, vox, gx, gy, boxes);
    }
}

uint32_t assign_status(const void *scratch)
{
    AssignState st{};
    cudaMemcpy(&st, scratch, sizeof(st), cudaMemcpyDeviceToHost);
    return st.status;
}

}  // namespace roam
