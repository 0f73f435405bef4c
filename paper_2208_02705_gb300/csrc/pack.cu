// The derived copies of the fields' FP32 masters (API layout), in one pass: the
// transposed copy of the FP32 kernels, the dgrad copy of the FP32 adjoint, and
// the tensor-core images (BF16, and E4M3 with one FP32 scale per output
// channel).
//
// One block per layer of a field: the layer's matrix lands in shared memory
// once (rows an odd number of floats apart), and every copy asked for is
// written from there in the order of its own layout, 16 bytes per thread for
// the images.  Measured (GB300, 512 fields of W = 64 / H = 3, every copy: 46 MB
// read, 150 MB written): 67 us, with the check for NaN and infinity; one kernel
// per copy, each finding every element's place by division and reading it from
// global memory, took 480 us together.
#include "layouts.cuh"
#include "tc_common.cuh"

namespace roam {

namespace {

constexpr int kPackThreads = 256;

enum { kL1, kHidden, kHead, kColour, kOut };       // kinds of layer

// API rows and inputs of a kind of layer, and the floats it takes in shared
// memory: the matrix with odd rows, then its biases and channel scales
__host__ __device__ constexpr int pack_rows_of(int W, int kind) { return kind == kHead ? 1 + W : (kind == kOut ? 3 : W); }
__host__ __device__ constexpr int pack_inputs_of(int W, int kind)
{
    return kind == kL1 ? kPeX : (kind == kColour ? W + kPeD : W);
}
__host__ __device__ constexpr int pack_floats(int W, int kind)
{
    return pack_rows_of(W, kind) * ((pack_inputs_of(W, kind) | 1) + 2);
}
__host__ __device__ constexpr int pack_smem(int W)
{
    int m = 0;
    for (int k = kL1; k <= kOut; ++k) m = pack_floats(W, k) > m ? pack_floats(W, k) : m;
    return m * (int)sizeof(float);
}

template <int W, int H, int KIND>
__device__ __forceinline__ void pack_layer(const float *__restrict__ src, int l, const PackDst &d, int f, int64_t P,
                                           float *sm)
{
    using S = TcShape<W, H, false>;
    using S8 = TcShape<W, H, true>;
    constexpr ApiLayout A(W, H);
    constexpr TLayout T(W, H);
    constexpr RLayout R(W, H);
    constexpr int N = pack_rows_of(W, KIND), K = pack_inputs_of(W, KIND), LD = K | 1;
    static_assert((N * LD + 2 * N) * (int)sizeof(float) <= pack_smem(W), "a layer fits in the block's shared memory");
    const int64_t hid = (int64_t)(l - 1) * ((int64_t)W * W + W);
    const int64_t off = KIND == kL1 ? A.l1 : (KIND == kHidden ? A.hid + hid : (KIND == kHead ? A.head : (KIND == kColour ? A.col : A.out)));
    float *bias = sm + N * LD, *scale = bias + N;
    const int tid = threadIdx.x;
    const float *ws = src + (int64_t)f * P + off;
    bool bad = false;
#pragma unroll 4
    for (int e = tid; e < N * K + N; e += kPackThreads) {
        const float v = ws[e];
        bad |= !isfinite(v);
        if (d.w32) d.w32[(int64_t)f * P + off + e] = v;
        if (e < N * K) sm[(e / K) * LD + e % K] = v;
        else bias[e - N * K] = v;
    }
    if (bad && d.bad) atomicOr(d.bad, 1u);
    __syncthreads();
    // row of output n as the kernels see it: the head's features, then its density logit
    auto row = [&](int n) { return KIND == kHead ? (n < W ? 1 + n : (n == W ? 0 : -1)) : (n < N ? n : -1); };

    if (d.wt) {
        constexpr int NP = KIND == kHead ? round4(1 + W) : (KIND == kOut ? 4 : W);
        float *o = d.wt + (int64_t)f * T.total +
                   (KIND == kL1 ? T.l1 : (KIND == kHidden ? T.hid + hid : (KIND == kHead ? T.head : (KIND == kColour ? T.col : T.out))));
        for (int e = tid; e < (K + 1) * NP; e += kPackThreads) {
            const int k = e / NP, r = row(e % NP);
            o[e] = r < 0 ? 0.f : (k < K ? sm[r * LD + k] : bias[r]);
        }
    }
    if (d.wr && (KIND == kHidden || KIND == kHead || KIND == kColour)) {
        float *o = d.wr + (int64_t)f * R.total +
                   (KIND == kHidden ? R.hid + (int64_t)(l - 1) * W * W : (KIND == kHead ? R.head : R.col));
        for (int e = tid; e < W * W; e += kPackThreads) o[e] = sm[row(e / W) * LD + e % W];
    }
    if constexpr (KIND == kOut) {
        // the FP32 output layer of both images: [4][W] (a zero row last), then bias[4]
        for (int e = tid; e < 4 * W + 4; e += kPackThreads) {
            const float v = e < 4 * W ? (e / W < 3 ? sm[(e / W) * LD + e % W] : 0.f) : (e - 4 * W < 3 ? bias[e - 4 * W] : 0.f);
            if (d.img) reinterpret_cast<float *>(d.img + f * d.img_bytes + S::kMatBytes)[e] = v;
            if (d.img8) reinterpret_cast<float *>(d.img8 + f * d.img8_bytes + S8::kMatBytes)[e] = v;
        }
        return;
    } else {
        constexpr int NM = KIND == kHead ? S::N_HEAD : W;                    // MMA rows (both images alike)
        constexpr int KIMG = K + 1;                                          // inputs and the constant-1 column
        // operand (row r of the API, MMA column k), `fold`: the bias in its constant-1 column
        auto operand = [&](int r, int k, bool fold_in, bool fold_hidden) -> float {
            if (r < 0) return 0.f;
            if (KIND == kColour) {
                if (k < W) return sm[r * LD + k];
                if (k == W) return fold_in ? bias[r] : 0.f;
                return k <= W + kPeD ? sm[r * LD + k - 1] : 0.f;
            }
            if (k < K) return sm[r * LD + k];
            return k == K && (KIND == kL1 ? fold_in : fold_hidden) ? bias[r] : 0.f;
        };
        if (d.img) {
            uint8_t *o = d.img + f * d.img_bytes;
            for (int q = tid; q < S::chunks(KIND == kHidden ? 1 : (KIND == kL1 ? 0 : (KIND == kHead ? H : H + 1))) * NM * 8;
                 q += kPackThreads) {
                const int ch = q / (NM * 8), n = (q / 8) % NM, k0 = ch * 64 + (((q & 7) ^ (n & 7)) << 3), r = row(n);
                uint32_t w[4] = {0u, 0u, 0u, 0u};
                if (k0 < KIMG)                       // (past the operand's inputs: zeros)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    w[i] = pack_bf16(operand(r, k0 + 2 * i, true, S::kFold), operand(r, k0 + 2 * i + 1, true, S::kFold));
                *reinterpret_cast<uint4 *>(o + S::offset(l) + 16 * q) = make_uint4(w[0], w[1], w[2], w[3]);
            }
            if constexpr (S::kTab) {
                float *t = reinterpret_cast<float *>(o + S::kMatBytes + S::kOutBytes) + l * 2 * S::kTabStride;
                for (int n = tid; n < S::kTabStride; n += kPackThreads) {
                    t[n] = 1.f;
                    t[S::kTabStride + n] = row(n) >= 0 ? bias[row(n)] : 0.f;
                }
            }
        }
        if (d.img8) {
            uint8_t *o = d.img8 + f * d.img8_bytes;
            // channel scales: max |row| / 448 (1 for an all-zero row; at least the
            // smallest float, so that no weight becomes 0 / 0), a warp per row
            for (int r = tid >> 5; r < N; r += kPackThreads / 32) {
                float m = 0.f;
                for (int k = tid & 31; k < K; k += 32) m = fmaxf(m, fabsf(sm[r * LD + k]));
#pragma unroll
                for (int s = 16; s > 0; s >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, s));
                if ((tid & 31) == 0) scale[r] = m > 0.f ? fmaxf(m / 448.0f, __int_as_float(1)) : 1.f;
            }
            __syncthreads();
            for (int q = tid; q < S8::chunks(KIND == kHidden ? 1 : (KIND == kL1 ? 0 : (KIND == kHead ? H : H + 1))) * NM * 8;
                 q += kPackThreads) {
                const int ch = q / (NM * 8), n = (q / 8) % NM, k0 = ch * 128 + (((q & 7) ^ (n & 7)) << 4), r = row(n);
                const float s = r < 0 ? 1.f : scale[r];
                uint32_t w[4] = {0u, 0u, 0u, 0u};
                if (k0 < KIMG)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float v[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) v[j] = operand(r, k0 + 4 * i + j, false, false) / s;
                    w[i] = pack_e4m3x4(v[0], v[1], v[2], v[3]);
                }
                *reinterpret_cast<uint4 *>(o + S8::offset(l) + 16 * q) = make_uint4(w[0], w[1], w[2], w[3]);
            }
            float *t = reinterpret_cast<float *>(o + S8::kMatBytes + S8::kOutBytes) + l * 2 * S8::kTabStride;
            for (int n = tid; n < S8::kTabStride; n += kPackThreads) {
                t[n] = row(n) >= 0 ? scale[row(n)] : 1.f;
                t[S8::kTabStride + n] = row(n) >= 0 ? bias[row(n)] : 0.f;
            }
        }
    }
}

// grid: (layers of a field, fields)
template <int W, int H>
__global__ void __launch_bounds__(kPackThreads) k_pack(const float *__restrict__ src, int64_t P, PackDst d)
{
    extern __shared__ float sm[];
    const int l = blockIdx.x, f = blockIdx.y;
    if (l == 0) pack_layer<W, H, kL1>(src, l, d, f, P, sm);
    else if (l < H) pack_layer<W, H, kHidden>(src, l, d, f, P, sm);
    else if (l == H) pack_layer<W, H, kHead>(src, l, d, f, P, sm);
    else if (l == H + 1) pack_layer<W, H, kColour>(src, l, d, f, P, sm);
    else pack_layer<W, H, kOut>(src, l, d, f, P, sm);
}

template <int W, int H>
void launch_pack_t(const float *src, int n_fields, int64_t P, const PackDst &d, cudaStream_t s)
{
    static int smem_set[kMaxDevices] = {};
    raise_smem_limit((const void *)k_pack<W, H>, pack_smem(W), smem_set);
    k_pack<W, H><<<dim3(H + 3, (unsigned)n_fields), kPackThreads, pack_smem(W), s>>>(src, P, d);
}

}  // namespace

int64_t simt_transposed_size(int W, int H) { return TLayout(W, H).total; }

int64_t rows_padded_size(int W, int H) { return RLayout(W, H).total; }

void launch_pack(const float *src, int n_fields, int W, int H, int64_t P, const PackDst &d, cudaStream_t s)
{
    if (n_fields <= 0) return;
#define ROAM_CASE(WW, HH) \
    if (W == WW && H == HH) { launch_pack_t<WW, HH>(src, n_fields, P, d, s); return; }
    ROAM_CASE(32, 1) ROAM_CASE(32, 2) ROAM_CASE(32, 3) ROAM_CASE(32, 4)
    ROAM_CASE(64, 1) ROAM_CASE(64, 2) ROAM_CASE(64, 3) ROAM_CASE(64, 4)
    ROAM_CASE(128, 1) ROAM_CASE(128, 2) ROAM_CASE(128, 3) ROAM_CASE(128, 4)
#undef ROAM_CASE
}

}  // namespace roam
