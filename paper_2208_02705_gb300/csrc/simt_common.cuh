// Shared pieces of the FP32 SIMT kernels of the per-field MLPs (forward and
// adjoint): shared-memory rows, the accurate field-local coordinate, and the
// gather of a tile's samples a tile ahead.
#pragma once

#include "layouts.cuh"

namespace roam {

namespace {

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// TN consecutive floats from shared memory
template <int TN>
__device__ __forceinline__ void ld_row(const float *p, float2 (&w)[TN / 2])
{
    if constexpr (TN >= 4) {
#pragma unroll
        for (int q = 0; q < TN / 4; ++q) {
            const float4 v = *reinterpret_cast<const float4 *>(p + 4 * q);
            w[2 * q] = make_float2(v.x, v.y);
            w[2 * q + 1] = make_float2(v.z, v.w);
        }
    } else {
        w[0] = *reinterpret_cast<const float2 *>(p);
    }
}

// Field-local coordinate scale * (o + t d) + offset of sample j, with
// t = (j + 1/2) delta and d = dh + dl carried as unevaluated FP32 pairs
// (error-free products and sums, explicitly rounded operations so that no
// step is contracted): accurate to about one FP32 ulp of the result.
__device__ __forceinline__ float local_coord(float th0, float delta, float o, float dh, float dl, float scale,
                                             float offset)
{
    const float t_hi = __fmul_rn(th0, delta);
    const float t_lo = __fmaf_rn(th0, delta, -t_hi);
    const float ph = __fmul_rn(t_hi, dh);
    const float pl = __fadd_rn(__fmaf_rn(t_hi, dh, -ph), __fadd_rn(__fmul_rn(t_hi, dl), __fmul_rn(t_lo, dh)));
    const float sh = __fadd_rn(o, ph);
    const float bv = __fsub_rn(sh, o);
    const float se = __fadd_rn(__fsub_rn(o, __fsub_rn(sh, bv)), __fsub_rn(ph, bv));
    const float sl = __fadd_rn(se, pl);
    const float qh = __fmul_rn(scale, sh);
    const float ql = __fadd_rn(__fmaf_rn(scale, sh, -qh), __fmul_rn(scale, sl));
    return __fadd_rn(__fadd_rn(qh, offset), ql);
}

// One tile's sample of a thread, gathered in stages a tile ahead so that no
// stage waits for the load before it.
struct SimtPending {
    bool on;
    uint32_t idx, rec, ray;
    float4 o, d, dl;
};

__device__ __forceinline__ void simt_index(SimtPending &q, const BucketBufs &b, const Tile &tl, int s, bool more)
{
    q.on = more && (uint32_t)s < tl.count;
    if (q.on) q.idx = b.sorted[tl.start + s];
}

__device__ __forceinline__ void simt_record(SimtPending &q, const SampleSrc &src)
{
    if (!q.on || src.mode != 0) return;
    const uint32_t i = group_of(q.idx >> 5, (uint32_t)src.R) * 32u + (q.idx & 31u);
    q.rec = src.recs[q.idx];
    q.ray = src.live ? src.live[i] : i;
}

__device__ __forceinline__ void simt_ray(SimtPending &q, const SampleSrc &src)
{
    if (!q.on) return;
    if (src.mode == 0) {
        q.o = src.st.orig[q.ray];
        q.d = src.st.dir[q.ray];
        if (src.accurate) q.dl = src.st.dir_lo[q.ray];
    } else {
        const int64_t k = 3 * (int64_t)q.idx;
        q.o = make_float4(src.p[k], src.p[k + 1], src.p[k + 2], 0.f);
        q.d = make_float4(src.d[k], src.d[k + 1], src.d[k + 2], 0.f);
    }
}

// F(x) of the gathered sample's field-local position and F(d) of its direction
// (F(v) = [v, sin(2^k pi v), cos(2^k pi v)]_k, three sines then three cosines
// per frequency; 2^k x is exact in FP32, sincospif reduces it exactly), as
// column entries XS apart from xp and dp on: the sample's 14 frequencies split
// over its NP threads, this one being `part`.
template <int NP, int XS>
__device__ __forceinline__ void simt_encode(const SimtPending &me, const SampleSrc &src, const float *aff, float *xp,
                                            float *dp, int part)
{
    float xl[3] = {0.f, 0.f, 0.f}, dv[3] = {0.f, 0.f, 1.f};
    if (me.on) {
        const float op[3] = {me.o.x, me.o.y, me.o.z}, dd[3] = {me.d.x, me.d.y, me.d.z}, lp[3] = {me.dl.x, me.dl.y, me.dl.z};
        const float th0 = (float)(me.rec & 0xffffu) + 0.5f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            dv[a] = dd[a];
            if (src.mode == 1) xl[a] = fmaf(aff[a], op[a], aff[3 + a]);
            else if (src.accurate) xl[a] = local_coord(th0, src.delta, op[a], dd[a], lp[a], aff[a], aff[3 + a]);
            else xl[a] = fmaf(aff[a], fmaf(th0 * src.delta, dd[a], op[a]), aff[3 + a]);
        }
    }
    if (part == 0) {
#pragma unroll
        for (int a = 0; a < 3; ++a) xp[a * XS] = xl[a];
    }
    if (part == (NP > 1 ? 1 : 0)) {
#pragma unroll
        for (int a = 0; a < 3; ++a) dp[a * XS] = dv[a];
    }
    for (int k = part; k < 14; k += NP) {
        const bool pos = k < 10;
        const int kk = pos ? k : k - 10;
        float *row = (pos ? xp : dp) + (3 + 6 * kk) * XS;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            float s, c;
            sincospif(ldexpf(pos ? xl[a] : dv[a], kk), &s, &c);
            row[a * XS] = s;
            row[(3 + a) * XS] = c;
        }
    }
}

}  // namespace

}  // namespace roam
