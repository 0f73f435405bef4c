// FP32 SIMT evaluation of the per-field tiny MLPs (the plain FP32 form of
// querying many MLPs at once): a block of 8 warps (4 at W = 32) takes one tile of
// 128 samples of one field at a time, each layer a register-tiled FP32 product.
//
// What bounds it: the FP32 FMA pipe, and beside it the register writes of the
// shared-memory loads (a float4 read from shared memory costs the FMA pipe of
// its sub-partition about 5 cycles).  So a thread owns TS samples x TN outputs
// (8 x 4 at W = 32, 4 x 8 at W = 64, 8 x 8 at W = 128) as packed FMAs; the
// layer's input sits in shared memory feature-major (rows of 128 samples,
// padded by 4), and its outputs replace it in place.  The weights (transposed
// copy, [in][out]) stream through a ring of 16-row stages copied asynchronously
// two stages ahead, so a tile needs 62 KB (W = 64) without its field's 92 KB of
// weights beside it, and two or three blocks share an SM: while one waits at
// a barrier or encodes, the others multiply.  Measured (GB300), against the
// field's weights beside two tiles of 4 warps in one block per SM: 8.2 M samples
// of a render at W = 64 / H = 3 8.83 -> 7.86 ms (0.58 of the FP32 peak), 8.4 M at
// W = 32 / H = 2 3.29 -> 2.86 ms, 8.2 M at W = 128 / H = 3 28.6 -> 23.2 ms; 5,000
// points of 1024 fields at W = 64 / H = 3 235 -> 109 us.  Where fields have long
// runs, so that the replaced form rarely reloaded its weights, the two are level:
// 32.7 M samples of 64 fields at W = 32 / H = 4 13.73 and 13.74 ms, 1 M points of
// one field there 430 and 446 us.
#include "simt_common.cuh"

namespace roam {

namespace {

constexpr int kTile = 128;            // samples per tile
constexpr int XS = kTile + 4;         // row stride of the activations
constexpr int kRingRows = 16, kStages = 3;

template <int W, int H>
struct SimtShape {
    static constexpr int kThreads = W == 32 ? 128 : 256;
    static constexpr int TS = W == 64 ? 4 : 8;                   // samples per thread
    static constexpr int TN = kTile * W / (kThreads * TS);       // outputs per thread
    static constexpr int SB = kTile / (8 * TS);                  // warps along the samples
    // warps without samples in a part-filled tile skip its products (at W = 128
    // the test spills more accumulators: 2 % of full tiles)
    static constexpr bool kSkip = W < 128;
    static constexpr int NH = round4(1 + W);
    static constexpr int rX = W >= 64 ? 0 : round4(W + kPeD);    // rows of F(x): beside those of [h; F(d)] at W = 32
    static constexpr int kRows = W >= 64 ? W + kPeD : rX + kPeX;
    static constexpr int kStage = kRingRows * NH > 4 * W + 4 ? kRingRows * NH : 4 * W + 4;
    // ring stages per tile: every matrix layer, then the output layer with its bias
    static constexpr int kPer = (kPeX + kRingRows - 1) / kRingRows + H * ((W + kRingRows - 1) / kRingRows) +
                                (W + kPeD + kRingRows - 1) / kRingRows + 1;
    static constexpr size_t kSmem = (size_t)(kRows * XS + kStages * kStage + 4 * kTile) * sizeof(float);
    // per SM: what shared memory holds (W = 32), or registers without spilling
    // the accumulators (at W = 64 a third block at 80 registers measured 0.5 %
    // faster on a full chip and 7 % slower on few tiles)
    static constexpr int kBlocks = W == 32 ? 3 : 2;
    static_assert(kRows >= kPeX && TN % 4 == 0, "whole float4 runs per thread");
};

__device__ __forceinline__ float softplus_f(float s) { return s > 20.f ? s : log1pf(expf(s)); }
__device__ __forceinline__ float sigmoid_f(float s) { return 1.f / (1.f + expf(-s)); }

template <int W, int H>
__global__ void __launch_bounds__(SimtShape<W, H>::kThreads, SimtShape<W, H>::kBlocks)
    k_mlp_simt(MlpWeights w, SampleSrc src, BucketBufs b, Counters *ctr, float4 *out)
{
    using F = SimtShape<W, H>;
    constexpr int TS = F::TS, TN = F::TN, G = TS / 4, KC = W + kPeD, kThreads = F::kThreads;
    constexpr int NP = kThreads / kTile;               // threads per sample in the gather and the output layer
    constexpr TLayout TL(W, H);
    extern __shared__ float4 smem4[];
    __shared__ int2 entries[F::kPer];                  // a tile's ring stages: offset in wt, 16-byte pieces
    float *X = reinterpret_cast<float *>(smem4);
    float *ring = X + F::kRows * XS;
    float *red = ring + kStages * F::kStage;           // [4][128]: the outputs' partial sums, the density logit
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int e = tid; e < F::kPer; e += kThreads) {
        int at = 0;
        int2 en = make_int2(0, 0);
        auto piece = [&](int64_t off, int n_rows, int ld, int per_stage) {
            const int n = (n_rows + per_stage - 1) / per_stage, r = e - at;
            at += n;
            if (r < 0 || r >= n) return;
            en = make_int2((int)off + r * per_stage * ld, min(per_stage, n_rows - r * per_stage) * ld / 4);
        };
        piece(TL.l1, kPeX, W, kRingRows);
        for (int l = 1; l < H; ++l) piece(TL.hid + (int64_t)(l - 1) * (W * W + W), W, W, kRingRows);
        piece(TL.head, W, F::NH, kRingRows);
        piece(TL.col, KC, W, kRingRows);
        piece(TL.out, W + 1, 4, W + 1);
        entries[e] = en;
    }
    __syncthreads();
    pdl_begin();

    // tiles of the width class split evenly over the blocks, in order
    const uint32_t c0 = ctr->class_tiles[w.cls], n_tiles = ctr->class_tiles[w.cls + 1] - c0;
    const uint32_t t0 = c0 + (uint32_t)((uint64_t)n_tiles * blockIdx.x / gridDim.x);
    const uint32_t t1 = c0 + (uint32_t)((uint64_t)n_tiles * (blockIdx.x + 1) / gridDim.x);
    if (t0 >= t1) return;

    // the ring's feed: stage j of the run is entry j mod kPer of its tile's list
    Tile tl = b.tiles[t0];                              // the next tile
    uint32_t issue_s = 0, issue_e = 0, issue_t = t0;
    const float *issue_w = w.wt + (int64_t)((int)tl.field - w.field_base) * w.Pt;
    auto feed = [&]() {
        if (issue_t < t1) {
            const int2 en = entries[issue_e];
            float *dst = ring + issue_s * F::kStage;
            for (int c = tid; c < en.y; c += kThreads) cp_async16(dst + 4 * c, issue_w + en.x + 4 * c);
            if (++issue_s == (uint32_t)kStages) issue_s = 0;
            if (++issue_e == (uint32_t)F::kPer) {
                issue_e = 0;
                ++issue_t;                              // (a tile has more entries than the ring has stages)
                issue_w = w.wt + (int64_t)((int)tl.field - w.field_base) * w.Pt;
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int j = 0; j + 1 < kStages; ++j) feed();
    uint32_t slot = 0;
    // the stage has landed for every thread, and every thread is past the stage
    // before it, whose slot takes the next copy; returns this stage
    auto next_stage = [&]() -> const float * {
        cp_async_wait<kStages - 2>();
        __syncthreads();
        feed();
        const float *p = ring + slot * F::kStage;
        if (++slot == (uint32_t)kStages) slot = 0;
        return p;
    };

    // a warp covers 8 TS samples x 4 TN outputs: lane = 8 sample groups x 4
    // output groups; the thread's samples are s0 + 32 g + q, g < G, q < 4
    const int sg = lane & 7, og = lane >> 3;
    const int s0 = (warp % F::SB) * 8 * TS + 4 * sg;
    const int n0 = (warp / F::SB) * 4 * TN + og * TN;
    const bool dens_warp = warp / F::SB == 0;           // the warps that also form the density logit
    bool live = true;                                   // the warp's samples reach into the tile

    // rows [0, K) x [K][LD] weights -> acc; kDens: also dens from column W
    auto dense = [&](auto KK, auto LDc, auto DENS, const float *x, float2 (&acc)[SimtShape<W, H>::TS][SimtShape<W, H>::TN / 2], float (&dens)[SimtShape<W, H>::TS]) {
        constexpr int K = decltype(KK)::value, LD = decltype(LDc)::value;
        constexpr bool kDens = decltype(DENS)::value != 0;
        auto rows = [&](auto NR, int k0) {
            const float *st = next_stage();
            const float *wr = st + n0, *xr = x + (int64_t)k0 * XS + s0;
#pragma unroll
            for (int k = 0; k < decltype(NR)::value; ++k) {
                float2 wv[TN / 2];
                ld_row<TN>(wr + k * LD, wv);
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const float4 x4 = *reinterpret_cast<const float4 *>(xr + k * XS + 32 * g);
                    const float xv[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int j = 0; j < TN / 2; ++j)
                            acc[4 * g + q][j] = __ffma2_rn(wv[j], make_float2(xv[q], xv[q]), acc[4 * g + q][j]);
                    if constexpr (kDens)
                        if (dens_warp) {
                            const float wd = st[k * LD + W];
#pragma unroll
                            for (int q = 0; q < 4; ++q) dens[4 * g + q] = fmaf(wd, xv[q], dens[4 * g + q]);
                        }
                }
            }
        };
        if (F::kSkip && !live) {                        // (the stages' barriers are everyone's)
#pragma unroll 1
            for (int k0 = 0; k0 < K; k0 += kRingRows) next_stage();
            return;
        }
#pragma unroll 1
        for (int k0 = 0; k0 + kRingRows <= K; k0 += kRingRows) rows(Int<kRingRows>{}, k0);
        if constexpr (K % kRingRows != 0) rows(Int<K % kRingRows>{}, K - K % kRingRows);
    };

    const int smp = tid & (kTile - 1), part = tid / kTile;
    SimtPending pend{};
    simt_index(pend, b, tl, smp, true);
    simt_record(pend, src);
    simt_ray(pend, src);
    for (uint32_t t = t0; t < t1; ++t) {
        const Tile tc = tl;
        const SimtPending me = pend;
        const bool more = t + 1 < t1;
        if (more) tl = b.tiles[t + 1];
        const float *wf = w.wt + (int64_t)((int)tc.field - w.field_base) * w.Pt;
        // a layer's biases of this thread's outputs, loaded a layer ahead
        float2 bias[TN / 2];
        auto load_bias = [&](int64_t off) {
#pragma unroll
            for (int j = 0; j < TN / 4; ++j) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(wf + off + n0) + j);
                bias[2 * j] = make_float2(v.x, v.y);
                bias[2 * j + 1] = make_float2(v.z, v.w);
            }
        };
        load_bias(TL.l1 + kPeX * W);
        const float bd = __ldg(wf + TL.head + W * F::NH + W);
        live = (uint32_t)((warp % F::SB) * 8 * TS) < tc.count;
        if (!F::kSkip || (uint32_t)(smp & ~31) < tc.count)
            simt_encode<NP, XS>(me, src, w.affine + 6 * (int64_t)tc.field, X + F::rX * XS + smp, X + W * XS + smp, part);
        float dens[TS];
        // one layer in place: rows [0, W) become its outputs (the first stage's
        // barrier orders them after what wrote the input)
        auto layer = [&](auto KK, auto LDc, auto DENS, const float *x, bool relu, int64_t next_bias) {
            float2 acc[TS][TN / 2];
#pragma unroll
            for (int q = 0; q < TS; ++q)
#pragma unroll
                for (int j = 0; j < TN / 2; ++j) acc[q][j] = bias[j];
            if (next_bias >= 0) load_bias(next_bias);
            dense(KK, LDc, DENS, x, acc, dens);
            __syncthreads();                               // every thread has read the input
#pragma unroll
            for (int j = 0; j < TN; ++j)
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    float v[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        v[q] = (j & 1) ? acc[4 * g + q][j / 2].y : acc[4 * g + q][j / 2].x;
                        if (relu) v[q] = fmaxf(v[q], 0.f);
                    }
                    *reinterpret_cast<float4 *>(X + (n0 + j) * XS + s0 + 32 * g) = make_float4(v[0], v[1], v[2], v[3]);
                }
        };
        // ---- L1, hidden layers, head (features and the density logit), colour ----
        layer(Int<kPeX>{}, Int<W>{}, Int<0>{}, X + F::rX * XS, true,
              H > 1 ? TL.hid + W * W : TL.head + (int64_t)W * F::NH);
        simt_index(pend, b, tl, smp, more);
#pragma unroll 1
        for (int l = 1; l < H; ++l)
            layer(Int<W>{}, Int<W>{}, Int<0>{}, X, true,
                  l + 1 < H ? TL.hid + (int64_t)l * (W * W + W) + W * W : TL.head + (int64_t)W * F::NH);
        simt_record(pend, src);
#pragma unroll
        for (int q = 0; q < TS; ++q) dens[q] = bd;
        layer(Int<W>{}, Int<F::NH>{}, Int<1>{}, X, false, TL.col + (int64_t)KC * W);
        if (dens_warp && og == 0) {
#pragma unroll
            for (int g = 0; g < G; ++g)
                *reinterpret_cast<float4 *>(red + 3 * kTile + s0 + 32 * g) =
                    make_float4(dens[4 * g], dens[4 * g + 1], dens[4 * g + 2], dens[4 * g + 3]);
        }
        layer(Int<KC>{}, Int<W>{}, Int<0>{}, X, true, -1);
        simt_ray(pend, src);
        // ---- rgb = sigmoid(Wo g + bo): a sample's threads take their shares of the sums ----
        {
            const float4 *wo = reinterpret_cast<const float4 *>(next_stage());     // [W][4], then bias[4]
            float z[3] = {0.f, 0.f, 0.f};
            if (part == 0) {
                const float4 bo = wo[W];
                z[0] = bo.x;
                z[1] = bo.y;
                z[2] = bo.z;
            }
            const float *g = X + part * (W / NP) * XS + smp;
#pragma unroll 8
            for (int k = 0; k < W / NP; ++k) {
                const float4 wk = wo[part * (W / NP) + k];
                const float gk = g[k * XS];
                z[0] = fmaf(wk.x, gk, z[0]);
                z[1] = fmaf(wk.y, gk, z[1]);
                z[2] = fmaf(wk.z, gk, z[2]);
            }
            if (NP > 1 && part == 1) {
#pragma unroll
                for (int c = 0; c < 3; ++c) red[c * kTile + smp] = z[c];
            }
            __syncthreads();
            if (part == 0 && me.on) {
                const float sl = red[3 * kTile + smp];
                const float sigma = w.sigma_scale * (w.act == ROAM_RELU ? fmaxf(sl, 0.f) : softplus_f(sl));
                if constexpr (NP > 1) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) z[c] += red[c * kTile + smp];
                }
                out[me.idx] = make_float4(sigma, sigmoid_f(z[0]), sigmoid_f(z[1]), sigmoid_f(z[2]));
            }
        }
    }
}

}  // namespace

template <int W, int H>
static void launch_t(const MlpWeights &w, const SampleSrc &src, const BucketBufs &b, Counters *ctr, float4 *out,
                     int n_sm, cudaStream_t s)
{
    using F = SimtShape<W, H>;
    static int smem_set[kMaxDevices] = {};
    raise_smem_limit((const void *)k_mlp_simt<W, H>, (int)F::kSmem, smem_set);
    // one wave of resident blocks; each takes a contiguous run of tiles
    launch_pdl(k_mlp_simt<W, H>, n_sm * F::kBlocks, F::kThreads, F::kSmem, s, w, src, b, ctr, out);
}

void launch_mlp_simt(const MlpWeights &w, const SampleSrc &src, const BucketBufs &b, Counters *ctr, float4 *out,
                     int n_sm, cudaStream_t s)
{
#define ROAM_CASE(WW, HH) \
    if (w.W == WW && w.H == HH) { launch_t<WW, HH>(w, src, b, ctr, out, n_sm, s); return; }
    ROAM_CASE(32, 1) ROAM_CASE(32, 2) ROAM_CASE(32, 3) ROAM_CASE(32, 4)
    ROAM_CASE(64, 1) ROAM_CASE(64, 2) ROAM_CASE(64, 3) ROAM_CASE(64, 4)
    ROAM_CASE(128, 1) ROAM_CASE(128, 2) ROAM_CASE(128, 3) ROAM_CASE(128, 4)
#undef ROAM_CASE
}

}  // namespace roam
