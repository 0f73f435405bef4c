// Progressive probabilistic occupancy (Eq. 6; Alg. 1 stage I): the log-odds
// of every voxel grows by the measurement of each scan (one rendered view:
// depth and the opacity that normalises the weights of Eq. 5), clamped to
// [l_min, l_max], and a voxel is occupied iff its log-odds exceed
// logit(p_occ).  Per scan:
//   k_occ_rays   one thread per pixel with opacity A >= a_min: the ray's end
//                point is o + (D / A) d; every voxel whose interior the
//                segment crosses is marked free (a bit per voxel), the voxel
//                of the end point takes the ray's A as its hit confidence
//                (atomic max)
//   k_occ_apply  every marked voxel: hit -> L += logit(1/2 + (p_hit - 1/2) A),
//                else free -> L += logit(p_miss); clamp; clear the marks;
//                after the last scan the occupancy bits of every voxel
// The traversal walks the segment's voxel-plane crossings in increasing
// order, defined in FP64: the first interval's voxel from its midpoint, then
// one voxel step on every axis that crosses at the next parameter (all at
// once when they tie), marking each interval's voxel unless the interval is
// shorter than 1e-9 voxel; free bits of one 32-voxel word are gathered in
// a register and flushed with one atomic when the word changes.
//
// What bounds it: FP64 runs at 1/64 of the FP32 rate on this GPU, so every
// FP64 instruction of a warp costs its SM 16 cycles.  So the walk steps in
// FP32 while every decision is clear by a bound on the FP32 error of the
// crossing parameters, and takes single steps in FP64 from the same integer
// state (plane indices, voxel) where it is not: the voxels marked are those
// of the FP64 definition.  The bound of axis q at parameter t,
// 2^-23 |origin - o| / |d_q| + 2^-21 t_end, follows the roundings of
// (k vox + (origin - o)) / d_q; a fixed margin of 1e-3 voxel sent ten times
// as many steps to FP64.  What a ray's set-up shares with its view is formed
// once per view (k_occ_views): the FP64 sines and cosines of the pixel columns
// and rows, the first plane index per axis and direction, and the camera's
// voxel.  Beside that, the walk waits for the word bits it checks: looking at
// them one word later, blocks of 128 (which end sooner than 256 where the
// rays' lengths differ): 1318 -> 1071 us.  A step in FP64 takes one reciprocal per
// axis (Newton steps, no division) and forms the end's parameter only where it
// can be the next event: 1045.  Eight blocks per SM at 64 registers, some values
// spilled: 931 (seven at 72: 973; six at 80, none spilled: 1045).  Measured (GB300, four
// 1024x512 scans of a 256^3 floor): rays 3550 -> 931 us, voxel passes
// 225 -> 65 us.
#include "internal.cuh"

namespace roam {

namespace {

// what every ray of a view starts from
struct OccView {
    float k0[2][3];      // first plane with t > 0 per axis: [0] along +, [1] along -
    int cell[3];         // the camera's voxel
    int on_plane;        // the camera lies within 1e-6 voxel of a plane: voxels from midpoints
    uint32_t tab;        // equirectangular: first entry of its table (width columns, then height rows)
};

// One block per view: the table of (sin, cos) of an equirectangular view's
// longitudes and latitudes (as make_ray64 forms them), and its OccView.
__global__ void __launch_bounds__(256) k_occ_views(GridDev g, const DevCamera *cams, OccView *views, double2 *tab)
{
    const DevCamera &c = cams[blockIdx.x];
    uint32_t first = 0;
    for (unsigned v = 0; v < blockIdx.x; ++v)
        if (cams[v].model == ROAM_EQUIRECT) first += (uint32_t)(cams[v].width + cams[v].height);
    if (c.model == ROAM_EQUIRECT)
        for (int i = threadIdx.x; i < c.width + c.height; i += blockDim.x) {
            const double x = i < c.width ? 2.0 * (((double)i + 0.5) / (double)c.width) - 1.0
                                         : 0.5 - ((double)(i - c.width) + 0.5) / (double)c.height;
            double2 sc;
            sincospi(x, &sc.x, &sc.y);
            tab[first + i] = sc;
        }
    if (threadIdx.x < 3) {
        const int a = threadIdx.x;
        const double vox = (double)g.vox, org = (double)g.origin[a], o = (double)c.o[a];
        const double u0 = (o - org) * (1.0 / vox);
        // planes at the start are not crossings (t > 0)
        double kp = floor(u0) + 1.0, kn = ceil(u0) - 1.0;
        while (org + kp * vox - o <= 0.0) kp += 1.0;
        while (org + kn * vox - o >= 0.0) kn -= 1.0;
        OccView &v = views[blockIdx.x];
        v.k0[0][a] = (float)kp;
        v.k0[1][a] = (float)kn;
        v.cell[a] = (int)floor(u0);
        const bool near = fabs(u0 - rint(u0)) < 1e-6;
        const unsigned any = __ballot_sync(7u, near);
        if (a == 0) {
            v.on_plane = any != 0u;
            v.tab = first;
        }
    }
}

__global__ void __launch_bounds__(128, 8) k_occ_rays(GridDev g, const DevCamera *cams, int view, const OccView *views,
                                                  const double2 *tab, const float *depth, const float *opacity,
                                                  float a_min, uint32_t *hit, uint32_t *free_bits, uint32_t *hit_bits)
{
    const DevCamera &c = cams[view];
    const OccView &vw = views[view];
    const uint32_t n_pix = (uint32_t)c.width * (uint32_t)c.height;
    const float vf = g.vox;
    float of[3], gf[3], reach = (float)(g.gx + g.gy + g.gz) * vf;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        of[a] = c.o[a];
        gf[a] = g.origin[a] - of[a];
        reach += fabsf(gf[a]);
    }
    for (uint32_t pix = blockIdx.x * blockDim.x + threadIdx.x; pix < n_pix; pix += gridDim.x * blockDim.x) {
        const uint32_t gp = c.pix_start + pix;
        const float A = opacity[gp];
        if (!(A >= a_min)) continue;
        double3 d;
        if (c.model == ROAM_EQUIRECT) {
            const uint32_t v = pix / (uint32_t)c.width, u = pix - v * (uint32_t)c.width;
            const double2 p = tab[vw.tab + u], t = tab[vw.tab + (uint32_t)c.width + v];
            const double d0 = t.y * p.x, d1 = -t.x, d2 = t.y * p.y;
            d.x = (double)c.R[0] * d0 + (double)c.R[1] * d1 + (double)c.R[2] * d2;
            d.y = (double)c.R[3] * d0 + (double)c.R[4] * d1 + (double)c.R[5] * d2;
            d.z = (double)c.R[6] * d0 + (double)c.R[7] * d1 + (double)c.R[8] * d2;
        } else {
            make_ray64(c, pix, d);
        }
        const double dv[3] = {d.x, d.y, d.z};
        const float D = depth[gp];
        const float te = D / A;
        // per axis: next plane index (exact in FP32), step, crossing parameter
        // and the bound on its FP32 error
        float kf[3], sf[3], inf[3], tf[3], er[3];
        const float d32[3] = {(float)dv[0], (float)dv[1], (float)dv[2]};
        const float dmax = fmaxf(fmaxf(fabsf(d32[0]), fabsf(d32[1])), fabsf(d32[2]));
        // (no crossing inside the grid lies past t_grid)
        const float t_grid = reach / dmax;
        const float e_t = 4.7683716e-7f * fminf(fabsf(te), t_grid);      // 2^-21 t
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float df = d32[a];
            const bool crosses = fabsf(df) >= 1e-20f;            // (else no plane before the end)
            sf[a] = crosses ? copysignf(1.f, df) : 0.f;
            kf[a] = vw.k0[df > 0.f ? 0 : 1][a];
            inf[a] = crosses ? 1.f / df : 0.f;
            er[a] = crosses ? fmaf(1.1920929e-7f, fabsf(gf[a] * inf[a]), e_t) : 0.f;
            tf[a] = crosses ? fmaf(kf[a], vf, gf[a]) * inf[a] : 3.0e38f;
        }
        // 1 / d in FP64, two Newton steps from the FP32 reciprocal (a division is
        // several times as many FP64 operations, each of which takes its turn)
        auto inv64 = [&](int a) {
            double r = (double)inf[a];
            r = fma(fma(-dv[a], r, 1.0), r, r);
            return fma(fma(-dv[a], r, 1.0), r, r);
        };
        auto t64_of = [&](int a, double k, double inv) {
            return ((double)g.origin[a] + k * (double)vf - (double)of[a]) * inv;
        };
        // the first interval's voxel: the camera's, unless it lies on a plane
        int cc[3] = {vw.cell[0], vw.cell[1], vw.cell[2]};
        if (vw.on_plane) {
            double t1 = (double)D / (double)A;
            for (int a = 0; a < 3; ++a)
                if (sf[a] != 0.f) t1 = fmin(t1, t64_of(a, (double)kf[a], inv64(a)));
            for (int a = 0; a < 3; ++a)
                cc[a] = (int)floor(((double)of[a] + 0.5 * t1 * dv[a] - (double)g.origin[a]) * (1.0 / (double)vf));
        }
        // free bits of the current 32-voxel word, flushed when the word changes;
        // every ray of a view starts at the camera, so the words near it are
        // hit by all of them: bits already set (they are only ever set during
        // a scan) skip the atomic.  What a word's bits were is read when it is
        // left and looked at when the next word is left, so the read's latency
        // passes under the walk (an older value only costs an atomic more)
        uint32_t word = 0xffffffffu, mask = 0u;
        uint32_t old_word = 0u, old_mask = 0u, old_bits = 0u;
        auto flush = [&]() {
            if (old_mask & ~old_bits) atomicOr(&free_bits[old_word], old_mask);
            old_mask = mask;
            if (mask) {
                old_word = word;
                old_bits = __ldcg(&free_bits[word]);
            }
        };
        // false once the ray has left the grid for good
        auto mark_if_inside = [&]() -> bool {
            if ((unsigned)cc[0] >= (unsigned)g.gx || (unsigned)cc[1] >= (unsigned)g.gy || (unsigned)cc[2] >= (unsigned)g.gz)
                return !((cc[0] < 0 && sf[0] <= 0.f) || (cc[0] >= g.gx && sf[0] >= 0.f) ||
                         (cc[1] < 0 && sf[1] <= 0.f) || (cc[1] >= g.gy && sf[1] >= 0.f) ||
                         (cc[2] < 0 && sf[2] <= 0.f) || (cc[2] >= g.gz && sf[2] >= 0.f));
            const uint32_t w = ((uint32_t)cc[2] * (uint32_t)g.gy + (uint32_t)cc[1]) * (uint32_t)g.wpr + ((uint32_t)cc[0] >> 5);
            if (w != word) {
                flush();
                word = w;
                mask = 0u;
            }
            mask |= 1u << (cc[0] & 31);
            return true;
        };
        const float len = sqrtf(d32[0] * d32[0] + d32[1] * d32[1] + d32[2] * d32[2]);
        const float t_min = 1e-8f * vf / dmax;                  // (above the 1e-9 voxel rule)
        float cur_hi = 0.f;                                     // the last crossing's parameter and its error bound
        for (int guard = 0; guard < 3 * 65536; ++guard) {
            // the next event (a crossing or the end), the smallest the others can be
            float m1 = te, e1 = e_t, lo2 = 3.0e38f;
            int am = 3;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float x = tf[q];
                if (x < m1) {
                    lo2 = fminf(lo2, m1 - e1);
                    m1 = x;
                    e1 = er[q];
                    am = q;
                } else {
                    lo2 = fminf(lo2, x - er[q]);
                }
            }
            if (m1 + e1 <= lo2 && (m1 - e1) - cur_hi >= t_min) {
                if (!mark_if_inside() || am == 3) break;
                cur_hi = m1 + e1;
#pragma unroll
                for (int q = 0; q < 3; ++q)        // (no dynamic indexing: the arrays stay in registers)
                    if (q == am) {
                        kf[q] += sf[q];
                        cc[q] += (int)sf[q];
                        tf[q] = fmaf(kf[q], vf, gf[q]) * inf[q];
                    }
                continue;
            }
            // FP64: the parameter of the last plane crossed (0 before any)
            // and every axis' next crossing, as the definition computes them
            // (the end only where it may be the next event)
            const double t_end = te - e_t <= m1 + e1 || !(te >= 0.f) ? (double)D / (double)A : 1e300;
            double t_cur = 0.0, t_next = t_end;
            double t64[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                t64[q] = 1e300;
                if (sf[q] == 0.f) continue;
                const double inv = inv64(q), tp = t64_of(q, (double)(kf[q] - sf[q]), inv);
                if (tp > t_cur) t_cur = tp;
                t64[q] = t64_of(q, (double)kf[q], inv);
                t_next = fmin(t_next, t64[q]);
            }
            // the interval's length against 1e-9 voxel: with the FP32 length of d
            // unless that is within 1e-3 of the rule
            const double span = (t_next - t_cur) * (double)len, rule = 1e-9 * (double)vf;
            bool marks = t_next > t_cur && span >= 0.999 * rule;
            if (marks && span <= 1.001 * rule)
                marks = (t_next - t_cur) * sqrt(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]) >= rule;
            if (marks && !mark_if_inside()) break;
            if (t_next >= t_end) break;
            float e = e_t;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (t64[q] == t_next) {
                    kf[q] += sf[q];
                    cc[q] += (int)sf[q];
                    tf[q] = fmaf(kf[q], vf, gf[q]) * inf[q];
                    e = fmaxf(e, er[q]);
                }
            cur_hi = (float)t_next + e;
        }
        flush();
        mask = old_mask & ~old_bits;
        if (mask) atomicOr(&free_bits[old_word], mask);
        // the end point's voxel: in FP32 unless a coordinate is within 1e-2 voxel
        // of a plane.  With the end inside 8192 voxels and the camera within 16,384,
        // its terms stay below 24.6 k voxels: the roundings of te, d, the offset,
        // the sum and the reciprocal come to at most 2^-24 x 90 k = 5.4e-3 voxel
        int ce[3];
        bool clear = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float x = fmaf(te, d32[a], -gf[a]) * g.inv_vox;
            const float fl = floorf(x);
            if (!(x - fl >= 1e-2f && x - fl <= 0.99f && fabsf(x) < 8192.f)) clear = false;
            ce[a] = (int)fl;
        }
        if (!clear) {
            const double t_end = (double)D / (double)A;
            for (int a = 0; a < 3; ++a)
                ce[a] = (int)floor(((double)of[a] + t_end * dv[a] - (double)g.origin[a]) * (1.0 / (double)vf));
        }
        if ((unsigned)ce[0] < (unsigned)g.gx && (unsigned)ce[1] < (unsigned)g.gy && (unsigned)ce[2] < (unsigned)g.gz) {
            const uint32_t w = ((uint32_t)ce[2] * (uint32_t)g.gy + (uint32_t)ce[1]) * (uint32_t)g.wpr + ((uint32_t)ce[0] >> 5);
            const uint32_t bit = 1u << (ce[0] & 31);
            atomicMax(&hit[(int64_t)w * 32 + (ce[0] & 31)], __float_as_uint(A));
            if (!(__ldcg(&hit_bits[w]) & bit)) atomicOr(&hit_bits[w], bit);
        }
    }
}

__device__ __forceinline__ float logit_f(float p) { return logf(p / (1.f - p)); }

// One warp per 32 words of 32 voxels: the words the scan marked, one after the
// other (all of them when the occupancy bits are wanted).  A scan marks a few
// percent of a floor's words: reading only those, the pass over 16.7 M voxels
// takes the time of its 2 x 2 MB of marks; every voxel's hit and log-odds
// (134 MB) took 56 us.
__global__ void __launch_bounds__(256) k_occ_apply(int64_t n_words, roam_occ_params q, uint32_t *hit, uint32_t *free_bits,
                                                   uint32_t *hit_bits, float *logit, uint32_t *bits)
{
    const float l_thr = logit_f(q.p_occ), l_miss = logit_f(q.p_miss);
    const int lane = threadIdx.x & 31;
    for (int64_t w0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; w0 < n_words;
         w0 += (int64_t)gridDim.x * blockDim.x) {
        const bool in = w0 + lane < n_words;
        const uint32_t fw = in ? free_bits[w0 + lane] : 0u, hw = in ? hit_bits[w0 + lane] : 0u;
        const unsigned marked = __ballot_sync(0xffffffffu, (fw | hw) != 0u);
        unsigned todo = bits ? __ballot_sync(0xffffffffu, in) : marked;
        uint32_t my_bits = 0u;
        while (todo) {
            // four words at a time: their loads are in flight together
            int b[4];
            float L[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                b[u] = todo ? __ffs(todo) - 1 : -1;
                todo &= todo - 1u;
                L[u] = b[u] >= 0 ? logit[((w0 + b[u]) << 5) + lane] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (b[u] < 0) break;
                const uint32_t f = __shfl_sync(0xffffffffu, fw, b[u]), h = __shfl_sync(0xffffffffu, hw, b[u]);
                const int64_t v = ((w0 + b[u]) << 5) + lane;
                const bool is_hit = (h >> lane) & 1u, is_free = (f >> lane) & 1u;
                if (is_hit) {
                    const float A = __uint_as_float(hit[v]);
                    L[u] += logit_f(0.5f + (q.p_hit - 0.5f) * A);
                    hit[v] = 0u;
                } else if (is_free) {
                    L[u] += l_miss;
                }
                if (is_hit || is_free) {
                    L[u] = fminf(fmaxf(L[u], q.l_min), q.l_max);
                    logit[v] = L[u];
                }
                if (bits) {
                    const uint32_t occ = __ballot_sync(0xffffffffu, L[u] > l_thr);
                    if (lane == b[u]) my_bits = occ;
                }
            }
        }
        if (fw) free_bits[w0 + lane] = 0u;
        if (hw) hit_bits[w0 + lane] = 0u;
        if (bits && in) bits[w0 + lane] = my_bits;
    }
}

}  // namespace

size_t occupancy_view_bytes(int n_views) { return (size_t)n_views * sizeof(OccView); }

void launch_occupancy_views(const GridDev &g, const DevCamera *cams, int n_views, void *views, double2 *tab,
                            cudaStream_t s)
{
    k_occ_views<<<n_views, 256, 0, s>>>(g, cams, static_cast<OccView *>(views), tab);
}

void launch_occupancy_scan(const GridDev &g, const DevCamera *cams, int view, int n_pix, const void *views,
                           const double2 *tab, const float *depth, const float *opacity, const roam_occ_params &q,
                           uint32_t *hit, uint32_t *free_bits, uint32_t *hit_bits, float *logit, uint32_t *bits, int n_sm,
                           cudaStream_t s)
{
    // one thread per pixel: the traversal lengths differ widely between rays
    int blocks_r = (n_pix + 127) / 128;
    if (blocks_r < 1) blocks_r = 1;
    k_occ_rays<<<blocks_r, 128, 0, s>>>(g, cams, view, static_cast<const OccView *>(views), tab, depth, opacity, q.a_min,
                                        hit, free_bits, hit_bits);
    const int64_t n_words = (int64_t)g.wpr * g.gy * g.gz;
    int64_t blocks_a = (n_words + 255) / 256;
    if (blocks_a > (int64_t)n_sm * 16) blocks_a = (int64_t)n_sm * 16;
    k_occ_apply<<<(unsigned)blocks_a, 256, 0, s>>>(n_words, q, hit, free_bits, hit_bits, logit, bits);
}

}  // namespace roam
