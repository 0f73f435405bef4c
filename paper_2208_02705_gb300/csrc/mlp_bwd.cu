// FP32 adjoint of the per-field tiny MLPs for the fine-tuning step (Sec.
// "Adaptive Radiance Fields Slimming and Fine-tuning": L2 loss on rendered
// pixels) and the distillation step (Eq. 7), as register-tiled SIMT products;
// the Adam update and the losses.
//
// A CTA walks a contiguous run of tiles of kS samples of one field.  Per tile
// it recomputes the encoding and every activation (nothing is stored between
// the passes), then walks the layers backwards:
//   dgrad  dX[k][s]  = sum_n W[n][k] dZ[n][s]
//   wgrad  dW[n][k] += sum_s dZ[n][s] X[k][s],  db[n] += sum_s dZ[n][s]
// What bounds it: the FP32 FMA pipe (2 x (3 MACs - 63 W) FLOP per sample,
// 126 kFLOP at W = 64 / H = 3).  So
//  - every activation of the tile stays in shared memory, feature-major
//    ([k][kS samples], rows kS + 4 apart: consecutive rows start 4 banks
//    apart, which keeps the wgrad's loads along s conflict-free); dZ of a
//    layer overwrites the activations it belongs to, so no second buffer;
//  - a thread owns 4 samples x TN outputs (forward, all 8 warps) or
//    4 samples x 2 TN (dgrad, warps 0-3), while warps 4-7 form the same
//    layer's wgrad (W/8 outputs x 4 inputs per thread, reduced over s in
//    pairs): both have about the same work and share the FMA pipe;
//  - the weights stream through a ring of shared-memory stages (16 rows each),
//    copied asynchronously by warps 0-3 a few stages ahead, one barrier per
//    stage: they are read once per tile and would not fit beside the gradient
//    (bulk copies issued by one thread took ~400 cycles each out of its
//    warp's products; a producer warp would cap the others at 168 registers);
//  - the field's gradient accumulates in shared memory and goes to global
//    memory (one atomic per parameter) when the field changes.
// kS is what shared memory holds: 64 samples at W = 64 (H <= 3), 32 at
// W = 64 / H = 4, 128 at W = 32.
#include <cooperative_groups.h>

#include "simt_common.cuh"

namespace cg = cooperative_groups;

namespace roam {

namespace {

constexpr int kThreads = 256;
constexpr int kRingRows = 16;       // weight rows per ring stage

template <int W, int H>
struct FbShape {
    static constexpr int S = W == 32 ? 128 : (H <= 3 ? 64 : 32);    // samples per tile
    static constexpr int XS = S + 4;                                  // row stride of the activations
    static constexpr int TN = W * S / 1024;                           // forward outputs per thread
    static constexpr int TD = 2 * TN;                                 // dgrad inputs per thread
    static constexpr int KC = W + kPeD;
    static constexpr int NH = round4(1 + W);
    // activation rows: F(x), h_1 .. h_H, [feat; F(d)], g
    static constexpr int rX = 0;
    __host__ __device__ static constexpr int rH(int j) { return kPeX + (j - 1) * W; }    // h_j, j >= 1
    static constexpr int rC = kPeX + H * W;
    static constexpr int rG = rC + KC;
    static constexpr int kRows = rG + W;
    // gradient accumulators: rows of each matrix 4 or -4 banks apart
    static constexpr int SA = 68, SH = W + 4, SC = W == 64 ? 92 : 60;
    static constexpr int gA = 0;
    static constexpr int gHid = gA + W * SA;
    static constexpr int gHead = gHid + (H - 1) * W * SH;    // W feature rows
    static constexpr int gCol = gHead + W * SH;
    static constexpr int gDen = gCol + W * SC;               // the head's density row, W
    static constexpr int gOut = gDen + W;                    // 3 x W
    static constexpr int gB = gOut + 3 * W;                  // biases: (H + 2) x W (L1, hidden, head features, colour)
    static constexpr int gBd = gB + (H + 2) * W;             // density bias, then 3 output biases
    static constexpr int kGrad = round4(gBd + 4);
    // the field's small tables: biases as above, density weights, output
    // weights, density bias and output biases
    static constexpr int tB = 0;
    static constexpr int tDen = tB + (H + 2) * W;
    static constexpr int tOut = tDen + W;
    static constexpr int tBd = tOut + 3 * W;
    static constexpr int kTab = round4(tBd + 4);
    static constexpr int kStage = kRingRows * NH;            // floats of one ring stage
    static constexpr int kFixed = kRows * XS + kGrad + kTab + 4 * S;     // + dz of the 3 outputs and the density
    static constexpr int kStages = ((227 * 1024 - 1024) / 4 - kFixed) / kStage < 6
                                       ? ((227 * 1024 - 1024) / 4 - kFixed) / kStage : 6;
    static constexpr size_t kSmem = (size_t)(kFixed + kStages * kStage) * sizeof(float);
    // ring stages per tile: forward rows of every layer, then the dgrad's
    static constexpr int kPer = (kPeX + kRingRows - 1) / kRingRows + H * (W / kRingRows) +
                                (KC + kRingRows - 1) / kRingRows + (H + 1) * (W / kRingRows);
    static_assert(kStages >= 4, "the weight ring keeps a few stages in flight");
    static_assert(TN == 2 || TN == 4, "forward tiles of 2 or 4 outputs");
};

template <int W, int H>
__global__ void __launch_bounds__(kThreads, 1)
    k_mlp_bwd_simt(MlpWeights w, SampleSrc src, BucketBufs b, Counters *ctr, const float4 *gsr, float *grad)
{
    using F = FbShape<W, H>;
    constexpr int S = F::S, XS = F::XS, KC = F::KC, NST = F::kStages;
    constexpr ApiLayout A(W, H);
    constexpr RLayout RL(W, H);
    constexpr TLayout TL(W, H);
    extern __shared__ float4 smem4[];
    __shared__ int2 entries[F::kPer];      // a tile's ring stages: offset in wt (or -1 - offset in wr), 16-byte pieces
    float *X = reinterpret_cast<float *>(smem4);
    float *ring = X + F::kRows * XS;
    float *tab = ring + NST * F::kStage;
    float *dzo = tab + F::kTab;                       // [3][S] d loss / d output logit, then [S] of the density's
    float *gacc = dzo + 4 * S;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int q = tid; q < F::kGrad; q += kThreads) gacc[q] = 0.f;
    // the order in which a tile reads its weight rows
    for (int e = tid; e < F::kPer; e += kThreads) {
        int at = 0;
        int2 en = make_int2(0, 0);
        auto piece = [&](int64_t off, bool dgrad, int n_rows, int ld) {
            const int n = (n_rows + kRingRows - 1) / kRingRows, r = e - at;
            at += n;
            if (r < 0 || r >= n) return;
            const int o = (int)off + r * kRingRows * ld;
            en = make_int2(dgrad ? -1 - o : o, min(kRingRows, n_rows - r * kRingRows) * ld / 4);
        };
        piece(TL.l1, false, kPeX, W);
        for (int l = 1; l < H; ++l) piece(TL.hid + (int64_t)(l - 1) * (W * W + W), false, W, W);
        piece(TL.head, false, W, F::NH);
        piece(TL.col, false, KC, W);
        piece(RL.col, true, W, W);
        piece(RL.head, true, W, W);
        for (int l = H - 1; l >= 1; --l) piece(RL.hid + (int64_t)(l - 1) * W * W, true, W, W);
        entries[e] = en;
    }
    __syncthreads();

    const uint32_t n_tiles = ctr->n_tiles;
    const uint32_t t0 = (uint32_t)((uint64_t)n_tiles * blockIdx.x / gridDim.x);
    const uint32_t t1 = (uint32_t)((uint64_t)n_tiles * (blockIdx.x + 1) / gridDim.x);

    Tile tl{0u, 0u, 0u, 0u};                        // the next tile
    // the ring's feed, by warps 0-3: stage j of the run is entry j mod kPer of
    // its tile's list, into slot j mod NST
    uint32_t issue_s = 0, issue_e = 0, issue_t = t0, issue_f = 0u;
    auto feed = [&]() {
        if (issue_t < t1) {
            const int2 en = entries[issue_e];
            const float *rows = en.x >= 0 ? w.wt + (int64_t)issue_f * w.Pt + en.x : w.wr + (int64_t)issue_f * w.Pr + (-1 - en.x);
            float *dst = ring + issue_s * F::kStage;
            for (int c = tid; c < en.y; c += 128) cp_async16(dst + 4 * c, rows + 4 * c);
            if (++issue_s == (uint32_t)NST) issue_s = 0;
            if (++issue_e == (uint32_t)F::kPer) {
                issue_e = 0;
                ++issue_t;
                issue_f = tl.field;                 // (a tile has more entries than the ring has stages)
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (warp < 4 && t0 < t1) {
        issue_f = b.tiles[t0].field;
#pragma unroll 1
        for (int j = 0; j + 1 < NST; ++j) feed();
    }

    // forward and dgrad: a warp covers 32 samples x 4 TN (TD) outputs, lane =
    // 8 sample groups of 4 x 4 output groups
    constexpr int SB = S / 32;
    const int sg = lane & 7, og = lane >> 3;
    const int sF = (warp % SB) * 32 + 4 * sg;                       // first sample
    const int nF = (warp / SB) * 4 * F::TN + og * F::TN;            // first forward output
    const int kD = ((warp & 3) / SB) * 4 * F::TD + og * F::TD;      // first dgrad input (warps 0-3)
    uint32_t slot = 0;                                              // ring slot of the next stage to consume
    auto sync = [&]() { bar_sync(1, kThreads); };

    // acc[s][j] += sum over the next K ring rows of x[k][sF + s] row[col + j]
    // (by TH threads: all, or warps 0-3)
    auto dense = [&](auto KK, auto LDc, auto TT, auto THc, const float *x, int col,
                     float2 (&acc)[4][decltype(TT)::value / 2]) {
        constexpr int K = decltype(KK)::value, LD = decltype(LDc)::value, T = decltype(TT)::value,
                      TH = decltype(THc)::value;
        auto rows = [&](auto NR, int k0) {
            // the stage has landed for every loader, and every consumer is past
            // the stage before it, whose slot takes the next copy
            if (warp < 4) cp_async_wait<NST - 2>();
            bar_sync(TH == 256 ? 1 : 2, TH);
            if (warp < 4) feed();
            const float *wrow = ring + slot * F::kStage + col;
            const float *xr = x + (int64_t)k0 * XS + sF;
#pragma unroll
            for (int kk = 0; kk < decltype(NR)::value; ++kk) {
                float2 wv[T / 2];
                ld_row<T>(wrow + kk * LD, wv);
                const float4 xv = *reinterpret_cast<const float4 *>(xr + kk * XS);
                const float2 xx[4] = {make_float2(xv.x, xv.x), make_float2(xv.y, xv.y), make_float2(xv.z, xv.z),
                                      make_float2(xv.w, xv.w)};
#pragma unroll
                for (int j = 0; j < T / 2; ++j)
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[q][j] = __ffma2_rn(wv[j], xx[q], acc[q][j]);
            }
            if (++slot == (uint32_t)NST) slot = 0;
        };
#pragma unroll 1
        for (int k0 = 0; k0 + kRingRows <= K; k0 += kRingRows) rows(Int<kRingRows>{}, k0);
        if constexpr (K % kRingRows != 0) rows(Int<K % kRingRows>{}, K - K % kRingRows);
    };
    // rows r .. of the activations from this thread's outputs, 4 samples at once
    auto store = [&](auto TT, float *row, const float2 (&acc)[4][decltype(TT)::value / 2], bool relu) {
#pragma unroll
        for (int j = 0; j < decltype(TT)::value; ++j) {
            float4 v = (j & 1) ? make_float4(acc[0][j / 2].y, acc[1][j / 2].y, acc[2][j / 2].y, acc[3][j / 2].y)
                               : make_float4(acc[0][j / 2].x, acc[1][j / 2].x, acc[2][j / 2].x, acc[3][j / 2].x);
            if (relu) v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
            *reinterpret_cast<float4 *>(row + j * XS + sF) = v;
        }
    };
    // wgrad of K inputs of a layer by 4 warps (wi = this warp's index among
    // them) over samples [s0, s0 + NS): g[n][k] += sum_s dz[n][s] x[k][s]; a
    // lane owns outputs ln + 8 i and inputs kb + lk + 4 j, a warp W x 4 TK.
    // (at most W inputs at a time: every float4 loaded from shared memory costs
    // the FMA pipe ~5 cycles, so small TK is slow, and past TK = 4 the
    // accumulators spill; `last` adds after the other half of the block)
    auto wgrad = [&](auto KK, auto NSc, int wi, const float *dz, const float *x, float *g, int ldg, int s0, bool last) {
        constexpr int K = decltype(KK)::value, TNW = W / 8, TK = (K + 15) / 16, NS = decltype(NSc)::value;
        const int ln = lane & 7, lk = lane >> 3, kb = wi * 4 * TK + lk;
        float2 acc[TNW][TK];
#pragma unroll
        for (int i = 0; i < TNW; ++i)
#pragma unroll
            for (int j = 0; j < TK; ++j) acc[i][j] = make_float2(0.f, 0.f);
        const float *dzr = dz + ln * XS;
        const float *xr[TK];
#pragma unroll
        for (int j = 0; j < TK; ++j) xr[j] = x + min(kb + 4 * j, K - 1) * XS;    // (rows past K: computed, not kept)
#pragma unroll 2
        for (int s = s0; s < s0 + NS; s += 4) {
            float4 xv[TK];
#pragma unroll
            for (int j = 0; j < TK; ++j) xv[j] = *reinterpret_cast<const float4 *>(xr[j] + s);
#pragma unroll
            for (int i = 0; i < TNW; ++i) {
                const float4 d = *reinterpret_cast<const float4 *>(dzr + 8 * i * XS + s);
#pragma unroll
                for (int j = 0; j < TK; ++j) {
                    acc[i][j] = __ffma2_rn(make_float2(d.x, d.y), make_float2(xv[j].x, xv[j].y), acc[i][j]);
                    acc[i][j] = __ffma2_rn(make_float2(d.z, d.w), make_float2(xv[j].z, xv[j].w), acc[i][j]);
                }
            }
        }
        if (last) sync();
#pragma unroll
        for (int j = 0; j < TK; ++j) {
            const int k = kb + 4 * j;
            if (k >= K) continue;
#pragma unroll
            for (int i = 0; i < TNW; ++i) g[(ln + 8 * i) * ldg + k] += acc[i][j].x + acc[i][j].y;
        }
    };
    // row sums over the samples: out[n] += sum_s v[n][s] m[s] (m may be null: 1),
    // n < W, by the 128 threads of a half (ht = thread within it)
    auto row_sums = [&](int ht, const float *v, const float *m, float *out) {
        constexpr int PT = 128 / W;
        const int n = ht / PT, p = ht % PT;
        float a = 0.f;
#pragma unroll 4
        for (int s = 4 * p; s < S; s += 4 * PT) {
            const float4 q = *reinterpret_cast<const float4 *>(v + n * XS + s);
            if (m) {
                const float4 e = *reinterpret_cast<const float4 *>(m + s);
                a = fmaf(q.x, e.x, a);
                a = fmaf(q.y, e.y, a);
                a = fmaf(q.z, e.z, a);
                a = fmaf(q.w, e.w, a);
            } else {
                a += (q.x + q.y) + (q.z + q.w);
            }
        }
#pragma unroll
        for (int o = 1; o < PT; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (p == 0) out[n] += a;
    };
    // the accumulated gradient of field f to global memory, and cleared
    auto flush_part = [&](float *gf, float *rows, int n_out, int n_in, int ld) {
#pragma unroll 4
        for (int n = warp; n < n_out; n += 8) {
#pragma unroll 3
            for (int k = lane; k < n_in; k += 32) {
                const float v = rows[n * ld + k];
                if (v != 0.f) atomicAdd(gf + n * n_in + k, v);
                rows[n * ld + k] = 0.f;
            }
        }
    };
    auto flush = [&](uint32_t f) {
        float *gf = grad + (int64_t)f * w.P;
        flush_part(gf + A.l1, gacc + F::gA, W, kPeX, F::SA);
        flush_part(gf + A.l1 + W * kPeX, gacc + F::gB, 1, W, W);
        for (int l = 1; l < H; ++l) {
            const int64_t o = A.hid + (int64_t)(l - 1) * (W * W + W);
            flush_part(gf + o, gacc + F::gHid + (l - 1) * W * F::SH, W, W, F::SH);
            flush_part(gf + o + W * W, gacc + F::gB + l * W, 1, W, W);
        }
        flush_part(gf + A.head, gacc + F::gDen, 1, W, W);
        flush_part(gf + A.head + W, gacc + F::gHead, W, W, F::SH);
        flush_part(gf + A.head + (1 + W) * W, gacc + F::gBd, 1, 1, 1);
        flush_part(gf + A.head + (1 + W) * W + 1, gacc + F::gB + H * W, 1, W, W);
        flush_part(gf + A.col, gacc + F::gCol, W, KC, F::SC);
        flush_part(gf + A.col + W * KC, gacc + F::gB + (H + 1) * W, 1, W, W);
        flush_part(gf + A.out, gacc + F::gOut, 3, W, W);
        flush_part(gf + A.out + 3 * W, gacc + F::gBd + 1, 1, 3, 3);
    };

    uint32_t cur = 0xffffffffu;
    const int smp = tid % S;                     // this thread's sample in the gather and the encoding
    constexpr int NP = kThreads / S;             // threads per sample
    const int part = tid / S;
    SimtPending pend{};
    if (t0 < t1) {
        tl = b.tiles[t0];
        simt_index(pend, b, tl, smp, true);
        simt_record(pend, src);
        simt_ray(pend, src);
    }
    for (uint32_t t = t0; t < t1; ++t) {
        const Tile tc = tl;
        const SimtPending me = pend;
        const bool more = t + 1 < t1;
        if (more) tl = b.tiles[t + 1];
        // (every thread is past the previous tile's last reads: the barrier below)
        sync();
        if (tc.field != cur) {
            if (cur != 0xffffffffu) flush(cur);
            cur = tc.field;
            const float *wf = w.w32 + (int64_t)cur * w.P;
            for (int q = tid; q < F::kTab; q += kThreads) {
                float v = 0.f;
                if (q < F::tDen) {
                    const int l = q / W, n = q % W;
                    v = l == 0 ? wf[A.l1 + W * kPeX + n]
                               : (l < H ? wf[A.hid + (int64_t)(l - 1) * (W * W + W) + W * W + n]
                                        : (l == H ? wf[A.head + (1 + W) * W + 1 + n] : wf[A.col + W * KC + n]));
                } else if (q < F::tOut) v = wf[A.head + (q - F::tDen)];
                else if (q < F::tBd) v = wf[A.out + (q - F::tOut)];
                else if (q == F::tBd) v = wf[A.head + (1 + W) * W];
                else if (q < F::tBd + 4) v = wf[A.out + 3 * W + (q - F::tBd - 1)];
                tab[q] = v;
            }
        }
        // ---- encode: the sample's frequencies split over its NP threads ----
        const float4 gv = me.on ? gsr[me.idx] : make_float4(0.f, 0.f, 0.f, 0.f);
        simt_encode<NP, XS>(me, src, w.affine + 6 * (int64_t)tc.field, X + F::rX * XS + smp, X + (F::rC + W) * XS + smp,
                            part);
        sync();

        // ---- forward recompute ----
        auto forward = [&](auto KK, auto LDc, int layer, const float *x, float *y, bool relu) {
            float2 acc[4][F::TN / 2];
#pragma unroll
            for (int j = 0; j < F::TN / 2; ++j) {
                const float2 bb = *reinterpret_cast<const float2 *>(tab + F::tB + layer * W + nF + 2 * j);
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[q][j] = bb;
            }
            dense(KK, LDc, Int<F::TN>{}, Int<256>{}, x, nF, acc);
            store(Int<F::TN>{}, y + nF * XS, acc, relu);
            sync();
        };
        forward(Int<kPeX>{}, Int<W>{}, 0, X + F::rX * XS, X + F::rH(1) * XS, true);
        simt_index(pend, b, tl, smp, more);
#pragma unroll 1
        for (int l = 1; l < H; ++l)
            forward(Int<W>{}, Int<W>{}, l, X + F::rH(l) * XS, X + F::rH(l + 1) * XS, true);
        forward(Int<W>{}, Int<F::NH>{}, H, X + F::rH(H) * XS, X + F::rC * XS, false);
        simt_record(pend, src);
        forward(Int<KC>{}, Int<W>{}, H + 1, X + F::rC * XS, X + F::rG * XS, true);
        simt_ray(pend, src);

        // ---- outputs and the loss gradient at their logits: rgb by parts
        // 0 .. 2, the density by part 3 (a sample's parts go round its threads) ----
#pragma unroll 1
        for (int e = part; e < 4; e += NP) {
            const float *row = (e < 3 ? X + F::rG * XS : X + F::rH(H) * XS) + smp;
            const float *wv = tab + (e < 3 ? F::tOut + e * W : F::tDen);
            float z = tab[F::tBd + (e < 3 ? 1 + e : 0)];
#pragma unroll 16
            for (int k = 0; k < W; ++k) z = fmaf(wv[k], row[k * XS], z);
            if (e < 3) {
                const float c = 1.f / (1.f + expf(-z));
                dzo[e * S + smp] = (e == 0 ? gv.y : (e == 1 ? gv.z : gv.w)) * c * (1.f - c);
            } else {
                dzo[3 * S + smp] = gv.x * w.sigma_scale *
                                   (w.act == ROAM_RELU ? (z > 0.f ? 1.f : 0.f) : 1.f / (1.f + expf(-z)));
            }
        }
        sync();

        // ---- output layer: its wgrad, and dZ of the colour layer in g's place ----
        {
            constexpr int PT = kThreads / W;
            const int n = tid / PT, p = tid % PT;
            const float w0 = tab[F::tOut + n], w1 = tab[F::tOut + W + n], w2 = tab[F::tOut + 2 * W + n];
            float a0 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll 2
            for (int s = 4 * p; s < S; s += 4 * PT) {
                float4 *gp = reinterpret_cast<float4 *>(X + (F::rG + n) * XS + s);
                const float4 g4 = *gp;
                const float4 z0 = *reinterpret_cast<const float4 *>(dzo + s),
                             z1 = *reinterpret_cast<const float4 *>(dzo + S + s),
                             z2 = *reinterpret_cast<const float4 *>(dzo + 2 * S + s);
                const float gg[4] = {g4.x, g4.y, g4.z, g4.w}, y0[4] = {z0.x, z0.y, z0.z, z0.w},
                            y1[4] = {z1.x, z1.y, z1.z, z1.w}, y2[4] = {z2.x, z2.y, z2.z, z2.w};
                float dz[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    a0 = fmaf(y0[q], gg[q], a0);
                    a1 = fmaf(y1[q], gg[q], a1);
                    a2 = fmaf(y2[q], gg[q], a2);
                    const float d = fmaf(w2, y2[q], fmaf(w1, y1[q], w0 * y0[q]));
                    dz[q] = gg[q] > 0.f ? d : 0.f;
                }
                *gp = make_float4(dz[0], dz[1], dz[2], dz[3]);
            }
#pragma unroll
            for (int o = 1; o < PT; o <<= 1) {
                a0 += __shfl_xor_sync(0xffffffffu, a0, o);
                a1 += __shfl_xor_sync(0xffffffffu, a1, o);
                a2 += __shfl_xor_sync(0xffffffffu, a2, o);
            }
            if (p == 0) {
                gacc[F::gOut + n] += a0;
                gacc[F::gOut + W + n] += a1;
                gacc[F::gOut + 2 * W + n] += a2;
            }
            if (warp < 4) {
                // the output biases (warps 0-2) and the density's (warp 3)
                float a = 0.f;
#pragma unroll
                for (int s = lane; s < S; s += 32) a += dzo[warp * S + s];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
                if (lane == 0) gacc[F::gBd + (warp == 3 ? 0 : 1 + warp)] += a;
            }
        }
        sync();

        // ---- colour, head and hidden layers: dgrad by warps 0-3 beside
        // wgrad by warps 4-7; then dX, masked, over the layer's input ----
        auto backward = [&](int layer, const float *dz, float *x, float *g, int ldg, int kind) {
            float2 acc[4][F::TD / 2];
            if (warp < 4) {
                // the head's density row first (kind 1), as the layer's output 0
#pragma unroll
                for (int j = 0; j < F::TD / 2; ++j)
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[q][j] = make_float2(0.f, 0.f);
                if (kind == 1) {
                    float2 wv[F::TD / 2];
                    ld_row<F::TD>(tab + F::tDen + kD, wv);
                    const float4 d = *reinterpret_cast<const float4 *>(dzo + 3 * S + sF);
                    const float dd[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
                    for (int j = 0; j < F::TD / 2; ++j)
#pragma unroll
                        for (int q = 0; q < 4; ++q) acc[q][j] = make_float2(wv[j].x * dd[q], wv[j].y * dd[q]);
                }
                dense(Int<W>{}, Int<W>{}, Int<F::TD>{}, Int<128>{}, dz, kD, acc);
                row_sums(tid, dz, nullptr, gacc + F::gB + layer * W);
                // the colour layer's F(d) inputs beside its features' wgrad
                if (kind == 0) wgrad(Int<kPeD>{}, Int<S>{}, warp, dz, x + W * XS, g + W, ldg, 0, false);
                if (kind == 1) row_sums(tid, x, dzo + 3 * S, gacc + F::gDen);
            } else {
                wgrad(Int<W>{}, Int<S>{}, warp - 4, dz, x, g, ldg, 0, false);
                slot = (slot + W / kRingRows) % NST;
            }
            sync();
            if (warp < 4) {
                if (kind != 0) {
#pragma unroll
                    for (int j = 0; j < F::TD; ++j) {
                        const float4 h = *reinterpret_cast<const float4 *>(x + (kD + j) * XS + sF);
                        float *c[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) c[q] = (j & 1) ? &acc[q][j / 2].y : &acc[q][j / 2].x;
                        if (!(h.x > 0.f)) *c[0] = 0.f;
                        if (!(h.y > 0.f)) *c[1] = 0.f;
                        if (!(h.z > 0.f)) *c[2] = 0.f;
                        if (!(h.w > 0.f)) *c[3] = 0.f;
                    }
                }
                store(Int<F::TD>{}, x + kD * XS, acc, false);
            }
            sync();
        };
        // (kind 0: the features carry no activation)
        backward(H + 1, X + F::rG * XS, X + F::rC * XS, gacc + F::gCol, F::SC, 0);
        backward(H, X + F::rC * XS, X + F::rH(H) * XS, gacc + F::gHead, F::SH, 1);
#pragma unroll 1
        for (int l = H - 1; l >= 1; --l)
            backward(l, X + F::rH(l + 1) * XS, X + F::rH(l) * XS,
                            gacc + F::gHid + (l - 1) * W * F::SH, F::SH, 2);
        // ---- layer 1: wgrad only, half of the samples by each half of the block ----
        wgrad(Int<kPeX>{}, Int<S / 2>{}, warp & 3, X + F::rH(1) * XS, X + F::rX * XS, gacc + F::gA, F::SA,
              warp < 4 ? 0 : S / 2, warp >= 4);
        if (warp < 4) sync();
        if (warp < 4) row_sums(tid, X + F::rH(1) * XS, nullptr, gacc + F::gB);
    }
    sync();
    if (cur != 0xffffffffu) flush(cur);
}

__global__ void k_adam(float *__restrict__ w, float *__restrict__ m, float *__restrict__ v,
                       const float *__restrict__ g, int64_t n, float lr, float b1, float b2, float eps, float bc1,
                       float bc2)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = fmaf(b1, m[i], (1.f - b1) * gi);
        const float vi = fmaf(b2, v[i], (1.f - b2) * gi * gi);
        m[i] = mi;
        v[i] = vi;
        const float mh = mi / bc1, vh = vi / bc2;
        w[i] -= lr * mh / (sqrtf(vh) + eps);
    }
}

// The losses: one cluster of 8 blocks, the sum in a fixed order (per-thread
// strided sums, a fixed tree over the warp, the block and then the cluster,
// through distributed shared memory), so the same inputs give the same bits on
// every run, without scratch memory or a second launch.  One block alone took
// 34 us for 65,536 rays: its 32 warps cannot keep enough loads in flight.
constexpr int kLossBlocks = 8;

// every thread's sum over the cluster, in block 0's thread 0
__device__ __forceinline__ float cluster_sum(float acc)
{
    __shared__ float part[32];
    cg::cluster_group cluster = cg::this_cluster();
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = part[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (lane == 0) part[0] = acc;
    }
    cluster.sync();
    float v = 0.f;
    if (cluster.block_rank() == 0 && threadIdx.x == 0)
        for (int q = 0; q < kLossBlocks; ++q) v += cluster.map_shared_rank(part, q)[0];
    cluster.sync();                                   // no block leaves while its sum is read
    return v;
}

// L2 photometric loss of the fine-tuning stage: loss = sum (rgb - target)^2
// / norm over the rays, and dl/drgb = 2 (rgb - target) / norm (kVec: the three
// arrays are 16-byte aligned).
template <bool kVec>
__global__ void __cluster_dims__(kLossBlocks, 1, 1) __launch_bounds__(1024)
    k_l2_loss(int64_t n3, const float *__restrict__ rgb, const float *__restrict__ target, float inv_norm,
              float *__restrict__ dl, float *__restrict__ loss)
{
    float acc = 0.f;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    auto one = [&](float a, float b) {
        const float e = a - b;
        acc = fmaf(e * inv_norm, e, acc);
        return 2.f * e * inv_norm;
    };
    const int64_t n4 = kVec ? n3 / 4 : 0;
#pragma unroll 4
    for (int64_t i = t; i < n4; i += stride) {
        const float4 a = reinterpret_cast<const float4 *>(rgb)[i], b = reinterpret_cast<const float4 *>(target)[i];
        float4 d;
        d.x = one(a.x, b.x);
        d.y = one(a.y, b.y);
        d.z = one(a.z, b.z);
        d.w = one(a.w, b.w);
        reinterpret_cast<float4 *>(dl)[i] = d;
    }
    for (int64_t i = 4 * n4 + t; i < n3; i += stride) dl[i] = one(rgb[i], target[i]);
    acc = cluster_sum(acc);
    if (t == 0 && loss) *loss = acc;
}

template <int W, int H>
void launch_bwd_t(const MlpWeights &w, const SampleSrc &src, const BucketBufs &b, Counters *ctr, const float4 *gsr,
                  float *grad, int grid, cudaStream_t s)
{
    static int smem_set[kMaxDevices] = {};
    raise_smem_limit((const void *)k_mlp_bwd_simt<W, H>, (int)FbShape<W, H>::kSmem, smem_set);
    k_mlp_bwd_simt<W, H><<<grid, kThreads, FbShape<W, H>::kSmem, s>>>(w, src, b, ctr, gsr, grad);
}

#define ROAM_FB_CASES                                                          \
    ROAM_CASE(32, 1) ROAM_CASE(32, 2) ROAM_CASE(32, 3) ROAM_CASE(32, 4) \
    ROAM_CASE(64, 1) ROAM_CASE(64, 2) ROAM_CASE(64, 3) ROAM_CASE(64, 4)

}  // namespace

bool mlp_bwd_supported(int W, int H) { return (W == 32 || W == 64) && H >= 1 && H <= 4; }

int mlp_bwd_simt_tile(int W, int H)
{
#define ROAM_CASE(WW, HH) \
    if (W == WW && H == HH) return FbShape<WW, HH>::S;
    ROAM_FB_CASES
#undef ROAM_CASE
    return 128;
}

void launch_mlp_bwd_simt(const MlpWeights &w, const SampleSrc &src, const BucketBufs &b, Counters *ctr,
                         const float4 *gsr, float *grad, int grid, cudaStream_t s)
{
#define ROAM_CASE(WW, HH) \
    if (w.W == WW && w.H == HH) { launch_bwd_t<WW, HH>(w, src, b, ctr, gsr, grad, grid, s); return; }
    ROAM_FB_CASES
#undef ROAM_CASE
}

// Eq. 7 over samples: sum [(sigma_s - sigma_t)^2 + |c_s - c_t|^2] / I, its
// gradient 2 (student - teacher) / I per component.
__global__ void __cluster_dims__(kLossBlocks, 1, 1) __launch_bounds__(1024)
    k_distill_loss(int64_t n, const float4 *__restrict__ st, const float4 *__restrict__ te, float inv_I,
                   float4 *__restrict__ dl, float *__restrict__ loss)
{
    float acc = 0.f;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
#pragma unroll 4
    for (int64_t i = t; i < n; i += stride) {
        const float4 a = st[i], b = te[i];
        const float e0 = a.x - b.x, e1 = a.y - b.y, e2 = a.z - b.z, e3 = a.w - b.w;
        dl[i] = make_float4(2.f * e0 * inv_I, 2.f * e1 * inv_I, 2.f * e2 * inv_I, 2.f * e3 * inv_I);
        acc = fmaf(e0 * inv_I, e0, acc);
        acc = fmaf(e1 * inv_I, e1, acc);
        acc = fmaf(e2 * inv_I, e2, acc);
        acc = fmaf(e3 * inv_I, e3, acc);
    }
    acc = cluster_sum(acc);
    if (t == 0 && loss) *loss = acc;
}

void launch_distill_loss(int64_t n, const float4 *student, const float4 *teacher, float I, float4 *dl, float *loss,
                         cudaStream_t s)
{
    k_distill_loss<<<kLossBlocks, 1024, 0, s>>>(n, student, teacher, 1.0f / I, dl, loss);
}

void launch_l2_loss(int64_t n_rays, const float *rgb, const float *target, float norm, float *dl, float *loss,
                    cudaStream_t s)
{
    const bool vec = (((uintptr_t)rgb | (uintptr_t)target | (uintptr_t)dl) & 15) == 0;
    (vec ? k_l2_loss<true> : k_l2_loss<false>)<<<kLossBlocks, 1024, 0, s>>>(3 * n_rays, rgb, target, 1.0f / norm, dl, loss);
}

void launch_adam(float *w32, float *m, float *v, const float *g, int64_t n, float lr, float b1, float b2, float eps,
                 float bc1, float bc2, cudaStream_t s)
{
    k_adam<<<2048, 256, 0, s>>>(w32, m, v, g, n, lr, b1, b2, eps, bc1, bc2);
}

}  // namespace roam
