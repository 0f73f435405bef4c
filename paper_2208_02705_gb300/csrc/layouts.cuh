// Parameter layouts of one field's MLP (not part of the C ABI).
#pragma once

#include "internal.cuh"

namespace roam {

__host__ __device__ constexpr int round4(int x) { return (x + 3) & ~3; }

// The API layout: per layer the matrix row-major [out][in], then bias[out].
struct ApiLayout {
    int64_t l1, hid, head, col, out, total;
    __host__ __device__ constexpr ApiLayout(int W, int H)
        : l1(0), hid((int64_t)W * kPeX + W), head(hid + (int64_t)(H - 1) * ((int64_t)W * W + W)),
          col(head + (int64_t)(1 + W) * W + (1 + W)), out(col + (int64_t)W * (W + kPeD) + W),
          total(out + 3 * (int64_t)W + 3)
    {
    }
};

// The transposed copy of the FP32 kernels: per layer WT[in][n_pad] then
// bias[n_pad]; the head's row holds the W features, then the density logit
// (column W), then zeros; the output layer's row the 3 colours and a zero.
struct TLayout {
    int64_t l1, hid, head, col, out, total;
    __host__ __device__ constexpr TLayout(int W, int H)
        : l1(0), hid((int64_t)kPeX * W + W), head(hid + (int64_t)(H - 1) * ((int64_t)W * W + W)),
          col(head + (int64_t)W * round4(1 + W) + round4(1 + W)), out(col + (int64_t)(W + kPeD) * W + W),
          total(out + (int64_t)W * 4 + 4)
    {
    }
};

// The dgrad copy of the FP32 adjoint: rows [out][W inputs] of the hidden
// layers, the head's features (its density row is read from the masters) and
// the colour layer (its F(d) inputs need no gradient).
struct RLayout {
    int64_t hid, head, col, total;
    __host__ __device__ constexpr RLayout(int W, int H)
        : hid(0), head((int64_t)(H - 1) * W * W), col(head + (int64_t)W * W), total(col + (int64_t)W * W)
    {
    }
};

}  // namespace roam
