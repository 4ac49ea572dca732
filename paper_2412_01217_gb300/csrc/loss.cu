// loss.cu -- Eq. 10-13 per pyramid level, the Eq. 4-6 image pyramid, and Adam.
//
// RGB term (Eq. 10) and, in semantic-colour mode, the semantic term (Eq. 12):
//   (1 - lambda) mean|I - I_gt| + lambda (1 - SSIM(I, I_gt)),
// SSIM with an 11x11 Gaussian window (sigma 1.5), C1 = 0.01^2, C2 = 0.03^2, zero padding.
// One CTA owns a 32x32 output tile of one view-level and one group of planes.  It stages
// the planes with a 10-pixel halo, forms the five window moments (separable, horizontal
// then vertical) on the tile plus a 5-pixel halo, turns them into the three per-pixel
// partials of SSIM (w.r.t. the window mean, E[x^2] and E[xy]), and convolves those once
// more to get dL/dI for the tile -- one read of I and I_gt and one write of dL/dI per
// pixel, no intermediate maps in HBM.
// Depth term (Eq. 11): mean |D - D_gt| over pixels with D_gt > 0.
// Semantic term, cross-entropy mode: mean CE(softmax(decoder * S), label) over label >= 0.
// Sums are per-CTA partials reduced in a fixed order (deterministic).
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdio>

#include "sg_common.cuh"

namespace sg {

constexpr int kLTW = 32, kLTH = 32;           // loss tile (outputs)
constexpr int kXW = kLTW + 20, kXH = kLTH + 20;  // staged planes (10-px halo)
constexpr int kMW = kLTW + 10, kMH = kLTH + 10;  // moment / partial maps (5-px halo)
constexpr int kXP = kXW + 1, kMP = kMW + 1;      // padded row pitches (odd: no bank conflicts)
constexpr int kLossThreads = 256;

struct LossViews {
    int n;
    int tile_off[SG_MAX_VIEWS + 1];  // loss tiles (32x32) per view, prefix
    int pix_blk_off[SG_MAX_VIEWS + 1];  // 256-pixel blocks per view, prefix
};

__device__ __forceinline__ void gauss_window(float *w) {
    float s = 0.f;
    for (int i = 0; i < 11; ++i) {
        w[i] = expf(-(float)((i - 5) * (i - 5)) / (2.f * 1.5f * 1.5f));
        s += w[i];
    }
    for (int i = 0; i < 11; ++i) w[i] /= s;
}

__device__ __forceinline__ int find_prefix(const int *off, int n, int x) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= x) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ float block_sum(float v, float *s_red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(SG_FULL_MASK, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.f;
    if (threadIdx.x == 0)
        for (int w = 0; w < kLossThreads / 32; ++w) t += s_red[w];
    return t;  // valid in thread 0
}

// One term's images: nch planes per view.
struct SsimPlanes {
    const float *x, *y;  // planar images (rendered, target)
    float *grad;         // dL/dx
    int nch;
    float l1_coef_num;   // (1 - lambda) * weight  (divided by n = nch*W*H per view)
    float ssim_coef_num; // lambda * weight
    float lambda;
};
// The planes are split over kSsimGroups groups of CTAs (blockIdx.y), a group's planes one after
// the other: the first rgb_groups groups take the colour planes, the others the semantic
// ones.  Each plane in a CTA of its own fills the chip three times as well on small image
// sets (320x180 x 3 levels: 80 tiles on 152 SMs); the number of groups is what the workspace's
// four floats per tile hold.
constexpr int kSsimGroups = 4;
struct SsimArgs {
    SsimPlanes rgb, sem;
    int rgb_groups, sem_groups;
    const sg_view *views;
    LossViews lv;
    float *partials;     // per (group, tile): (1 - lambda) sum |x - y| - lambda sum ssim
    // valid-pixel counts (counts[2v]: target depth > 0, counts[2v+1]: label >= 0) gathered
    // on the side by the first group; label may be null
    const float *gt_depth;
    const int *label;
    int *counts;
};

// A pair of floats multiplied and added by one instruction (fma.rn.f32x2; each half rounds as
// fmaf does).
struct F2 {
    uint64_t v;
};
__device__ __forceinline__ F2 f2(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};\n" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack(F2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;\n" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// Sliding-window separable passes: each thread produces a run of consecutive outputs of one
// row (horizontal) or column (vertical), adding each input to every output whose window
// holds it.  The kernel is bound by instruction issue, so the window sums run two quantities
// to an instruction: the planes are staged as (x, y) pairs, the five moments as (x, y), (x^2, y^2)
// and xy, and two of the three partials as pairs, which also makes most shared-memory accesses
// one 8- or 16-byte word.  Every sum keeps its order, so the gradients are bit for bit those of
// one quantity per instruction, with which 1200x680 x 3 levels took 101 us against about 77 (loss
// with a 32-class decoder 233 -> 174 us, colour and four semantic planes at 637x477 x 3 levels
// 112 -> 79, with the loss's other kernels).  One moment of x^2 + y^2 in place of two took 66 us,
// but its rounding put the gradients of flat regions up to 1.46 times as far from 64 bits.
__global__ void __launch_bounds__(kLossThreads, 3) ssim_l1_kernel(SsimArgs a) {
    pdl_begin();
    extern __shared__ __align__(16) float sm[];
    float4 *Hm = reinterpret_cast<float4 *>(sm);                // kXH x kMP moments
    float *Hxy = reinterpret_cast<float *>(Hm + kXH * kMP);      // kXH x kMP: the moment of xy
    float2 *XY = reinterpret_cast<float2 *>(Hxy + kXH * kMP);   // kXH x kXP staged planes
    // the partials reuse the staged planes once the horizontal pass has consumed them, and
    // their horizontal sums the moments
    float2 *PQ = XY;                                            // kMH x kMP
    float *Rp = reinterpret_cast<float *>(PQ + kMH * kMP);      // kMH x kMP
    constexpr int kHP = kLTW + 1;
    float2 *HPQ = reinterpret_cast<float2 *>(Hm);               // kMH x kHP
    float *HR = reinterpret_cast<float *>(HPQ + kMH * kHP);     // kMH x kHP
    static_assert(3 * kMH * kMP <= 2 * kXH * kXP, "partials must fit the staged planes");
    static_assert(3 * kMH * kHP <= 4 * kXH * kMP, "their row sums must fit the moments");
    static_assert(kLossThreads == 256 && kXW <= 64 && kLTH * kLTW == 4 * kLossThreads, "work split");
    __shared__ int s_cnt[2];
    __shared__ float w[11];
    __shared__ float s_red[kLossThreads / 32];
    if (threadIdx.x == 0) gauss_window(w);
    const int item = blockIdx.x, group = blockIdx.y;
    const bool is_rgb = group < a.rgb_groups;
    const SsimPlanes &pl = is_rgb ? a.rgb : a.sem;
    const int sub = is_rgb ? group : group - a.rgb_groups, subs = is_rgb ? a.rgb_groups : a.sem_groups;
    const int nch = pl.nch, ch0 = nch * sub / subs, ch1 = nch * (sub + 1) / subs;
    const int v = find_prefix(a.lv.tile_off, a.lv.n, item);
    const sg_view &vw = a.views[v];
    const int W = vw.W, H = vw.H;
    const int tiles_x = (W + kLTW - 1) / kLTW;
    const int local = item - a.lv.tile_off[v];
    const int bx = local % tiles_x, by = local / tiles_x;
    const int ox = bx * kLTW - 10, oy = by * kLTH - 10;
    const size_t HW = (size_t)W * H;
    const float n = (float)nch * (float)HW;
    const float l1c = pl.l1_coef_num / n, sc = -pl.ssim_coef_num / n;
    const float C1 = 0.01f * 0.01f, C2 = 0.03f * 0.03f;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float l1_sum = 0.f, ssim_sum = 0.f;
    if (threadIdx.x < 2) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    F2 wr[11];  // (weight, weight); the window is symmetric
#pragma unroll
    for (int i = 0; i < 6; ++i) wr[i] = wr[10 - i] = f2(w[i], w[i]);
    auto w1 = [&](int j) { return unpack(wr[j]).x; };
    for (int ch = ch0; ch < ch1; ++ch) {
        const float *xs = pl.x + (size_t)nch * vw.pixel_offset + ch * HW;
        const float *ys = pl.y + (size_t)nch * vw.pixel_offset + ch * HW;
        // stage x, y with a 10-pixel halo (zero outside the image): a warp per row
#pragma unroll
        for (int cs = 0; cs < 2; ++cs) {
            const int c = lane + 32 * cs, gx = ox + c;
            const bool in_x = c < kXW && gx >= 0 && gx < W;
#pragma unroll
            for (int k = 0; k < (kXH + 7) / 8; ++k) {
                const int r = warp + 8 * k, gy = oy + r;
                const bool in = in_x && gy >= 0 && gy < H;
                const size_t q = (size_t)gy * W + gx;
                const float xv = in ? xs[q] : 0.f, yv = in ? ys[q] : 0.f;
                if (c < kXW && r < kXH) XY[r * kXP + c] = make_float2(xv, yv);
            }
        }
        __syncthreads();
        // Run lengths are chosen so that the passes' work items fill whole rounds of the
        // block's 256 threads (728, 252, 168 and 256 items).
        // horizontal window sums of the moments: rows kXH, outputs kMW in runs of 3
        {
            constexpr int RUN = 3, SEGS = kMW / RUN;  // 42 = 14 * 3
            for (int it = threadIdx.x; it < SEGS * kXH; it += kLossThreads) {
                const int seg = it / kXH, r = it - seg * kXH;
                const int c0 = seg * RUN;
                F2 s[RUN][2];
                float sxy[RUN];
#pragma unroll
                for (int o = 0; o < RUN; ++o) {
                    s[o][0] = s[o][1] = f2(0.f, 0.f);
                    sxy[o] = 0.f;
                }
#pragma unroll
                for (int i = 0; i < RUN + 10; ++i) {
                    const float2 q = XY[r * kXP + c0 + i];
                    const F2 xy = f2(q.x, q.y), sq = f2(q.x * q.x, q.y * q.y);
                    const float pr = q.x * q.y;
#pragma unroll
                    for (int o = 0; o < RUN; ++o)
                        if (i - o >= 0 && i - o < 11) {
                            s[o][0] = fma2(wr[i - o], xy, s[o][0]);
                            s[o][1] = fma2(wr[i - o], sq, s[o][1]);
                            sxy[o] = fmaf(w1(i - o), pr, sxy[o]);
                        }
                }
#pragma unroll
                for (int o = 0; o < RUN; ++o) {
                    const float2 p = unpack(s[o][0]), q = unpack(s[o][1]);
                    Hm[r * kMP + c0 + o] = make_float4(p.x, p.y, q.x, q.y);
                    Hxy[r * kMP + c0 + o] = sxy[o];
                }
            }
        }
        __syncthreads();
        // vertical window sums -> SSIM and its partials (zero outside the image): columns
        // kMW, output rows kMH in runs of 7
        {
            constexpr int RUN = 7, SEGS = kMH / RUN;  // 42 = 6 * 7
            for (int it = threadIdx.x; it < SEGS * kMW; it += kLossThreads) {
                const int seg = it / kMW, c = it - seg * kMW;
                const int r0 = seg * RUN;
                F2 m[RUN][2];
                float mxy[RUN];
#pragma unroll
                for (int o = 0; o < RUN; ++o) {
                    m[o][0] = m[o][1] = f2(0.f, 0.f);
                    mxy[o] = 0.f;
                }
#pragma unroll
                for (int i = 0; i < RUN + 10; ++i) {
                    const float4 q = Hm[(r0 + i) * kMP + c];
                    const F2 xy = f2(q.x, q.y), sq = f2(q.z, q.w);
                    const float pr = Hxy[(r0 + i) * kMP + c];
#pragma unroll
                    for (int o = 0; o < RUN; ++o)
                        if (i - o >= 0 && i - o < 11) {
                            m[o][0] = fma2(wr[i - o], xy, m[o][0]);
                            m[o][1] = fma2(wr[i - o], sq, m[o][1]);
                            mxy[o] = fmaf(w1(i - o), pr, mxy[o]);
                        }
                }
#pragma unroll
                for (int o = 0; o < RUN; ++o) {
                    const int r = r0 + o;
                    const int gy = by * kLTH - 5 + r, gx = bx * kLTW - 5 + c;
                    float P = 0.f, Q = 0.f, R = 0.f;
                    if (gx >= 0 && gx < W && gy >= 0 && gy < H) {
                        const float2 mu = unpack(m[o][0]), e2 = unpack(m[o][1]);
                        const float mx = mu.x, my = mu.y;
                        const float sxx = e2.x - mx * mx, syy = e2.y - my * my, sxy = mxy[o] - mx * my;
                        const float A1 = 2.f * mx * my + C1, A2 = 2.f * sxy + C2;
                        const float B1 = mx * mx + my * my + C1, B2 = sxx + syy + C2;
                        const float inv = 1.f / (B1 * B2);
                        const float s = A1 * A2 * inv;
                        if (r >= 5 && r < kLTH + 5 && c >= 5 && c < kLTW + 5) ssim_sum += s;
                        const float d_mx = 2.f * my * A2 * inv - s * 2.f * mx / B1;
                        const float d_sxx = -s / B2;
                        const float d_sxy = 2.f * A1 * inv;
                        P = sc * (d_mx - 2.f * mx * d_sxx - my * d_sxy);
                        Q = sc * d_sxx;
                        R = sc * d_sxy;
                    }
                    PQ[r * kMP + c] = make_float2(P, Q);
                    Rp[r * kMP + c] = R;
                }
            }
        }
        __syncthreads();
        // horizontal sums of the partials: rows kMH, outputs kLTW in runs of 8
        {
            constexpr int RUN = 8, SEGS = kLTW / RUN;
            if (threadIdx.x < SEGS * kMH) {
                const int seg = threadIdx.x / kMH, r = threadIdx.x - seg * kMH;
                const int c0 = seg * RUN;
                F2 s[RUN];
                float t[RUN];
#pragma unroll
                for (int o = 0; o < RUN; ++o) {
                    s[o] = f2(0.f, 0.f);
                    t[o] = 0.f;
                }
#pragma unroll
                for (int i = 0; i < RUN + 10; ++i) {
                    const float2 q = PQ[r * kMP + c0 + i];
                    const F2 pq = f2(q.x, q.y);
                    const float rr = Rp[r * kMP + c0 + i];
#pragma unroll
                    for (int o = 0; o < RUN; ++o)
                        if (i - o >= 0 && i - o < 11) {
                            s[o] = fma2(wr[i - o], pq, s[o]);
                            t[o] = fmaf(w1(i - o), rr, t[o]);
                        }
                }
#pragma unroll
                for (int o = 0; o < RUN; ++o) {
                    HPQ[r * kHP + c0 + o] = unpack(s[o]);
                    HR[r * kHP + c0 + o] = t[o];
                }
            }
        }
        __syncthreads();
        // vertical sums of the partials -> dL/dx on the tile: a column and 4 rows per thread
        float *gs = pl.grad + (size_t)nch * vw.pixel_offset + ch * HW;
        {
            constexpr int RUN = 4;
            const int c = lane, r0 = warp * RUN;
            const int gx = bx * kLTW + c;
            float xv[RUN], yv[RUN];  // (the staged planes now hold partials)
#pragma unroll
            for (int o = 0; o < RUN; ++o) {
                const int gy = by * kLTH + r0 + o;
                const bool in = gx < W && gy < H;
                const size_t gp = (size_t)gy * W + gx;
                xv[o] = in ? xs[gp] : 0.f;
                yv[o] = in ? ys[gp] : 0.f;
            }
            F2 s[RUN];
            float t[RUN];
#pragma unroll
            for (int o = 0; o < RUN; ++o) {
                s[o] = f2(0.f, 0.f);
                t[o] = 0.f;
            }
#pragma unroll
            for (int i = 0; i < RUN + 10; ++i) {
                const float2 q = HPQ[(r0 + i) * kHP + c];
                const F2 pq = f2(q.x, q.y);
                const float rr = HR[(r0 + i) * kHP + c];
#pragma unroll
                for (int o = 0; o < RUN; ++o)
                    if (i - o >= 0 && i - o < 11) {
                        s[o] = fma2(wr[i - o], pq, s[o]);
                        t[o] = fmaf(w1(i - o), rr, t[o]);
                    }
            }
#pragma unroll
            for (int o = 0; o < RUN; ++o) {
                const int gy = by * kLTH + r0 + o;
                if (gx >= W || gy >= H) continue;
                const float2 pq = unpack(s[o]);
                const float d = xv[o] - yv[o];
                l1_sum += fabsf(d);
                const float sg = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
                gs[(size_t)gy * W + gx] = l1c * sg + pq.x + 2.f * xv[o] * pq.y + yv[o] * t[o];
            }
        }
        __syncthreads();
    }
    if (group == 0) {  // the tile's valid pixels
        int n_depth = 0, n_label = 0;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            const int gx = bx * kLTW + lane, gy = by * kLTH + 4 * warp + o;
            if (gx >= W || gy >= H) continue;
            const size_t gp = (size_t)vw.pixel_offset + (size_t)gy * W + gx;
            n_depth += a.gt_depth[gp] > 0.f;
            if (a.label) n_label += a.label[gp] >= 0;
        }
        n_depth = __reduce_add_sync(SG_FULL_MASK, n_depth);
        n_label = __reduce_add_sync(SG_FULL_MASK, n_label);
        if (lane == 0) {
            atomicAdd(&s_cnt[0], n_depth);
            atomicAdd(&s_cnt[1], n_label);
        }
    }
    const float t1 = block_sum(l1_sum, s_red);  // (its barriers also order the counts above)
    const float t2 = block_sum(ssim_sum, s_red);
    if (threadIdx.x == 0) {
        a.partials[(size_t)group * gridDim.x + item] = (1.f - pl.lambda) * t1 - pl.lambda * t2;
        // integer atomics: the totals do not depend on the order
        if (group == 0 && s_cnt[0]) atomicAdd(a.counts + 2 * v, s_cnt[0]);
        if (group == 0 && s_cnt[1]) atomicAdd(a.counts + 2 * v + 1, s_cnt[1]);
    }
}

// ---------------------------------------------------------------------------------------
// depth L1, cross-entropy
// ---------------------------------------------------------------------------------------


struct PixelArgs {
    const float *depth, *gt_depth, *sem;
    const int *label;
    float *g_depth, *g_sem;
    const float *decoder;   // K x C or null
    float *decoder_grad;    // K x C or null
    int C, K, ce;           // ce: cross-entropy mode
    float w_depth, w_sem;
    const int *counts;
    const sg_view *views;
    LossViews lv;
    float *partials;        // per pixel block, kPixSlots slots of (sum |D - D_gt| over valid, sum CE over valid)
    float *dec_partials;    // per CTA: K x C share of the decoder gradient
};

// Loss-sum slots per 256-pixel block: one per warp (the SIMT kernel fills slot 0 with its
// block sum and zeroes the others).
constexpr int kPixSlots = kLossThreads / 32;

// Fixed-order reduction of the per-CTA decoder-gradient shares.  Up to kDecRows rows (what the
// persistent kernel's resident grid writes) are summed by one kernel: a CTA takes 32 outputs, warp
// w rows w, w + 32, ..., the warps in a fixed tree (304 rows of 512: 7.4 us for the two
// kernels below, most of it latency).  More rows go in two levels:
// level 1: chunk c of kDecChunks sums CTAs [c n / kDecChunks, (c+1) n / kDecChunks);
// level 2: decoder_grad[o] += sum over chunks.
constexpr int kDecRows = 1024;
__global__ void __launch_bounds__(1024) decoder_reduce_kernel(const float *__restrict__ part, int rows, int KC,
                                                              float *__restrict__ out) {
    pdl_begin();
    __shared__ float s_sum[32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, o = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (o < KC)
#pragma unroll 8
        for (int b = warp; b < rows; b += 32) s += part[(size_t)b * KC + o];
    s_sum[lane][warp] = s;
    __syncthreads();
    // warp w adds output w's 32 sums
    float t = s_sum[warp][lane];
#pragma unroll
    for (int i = 16; i > 0; i >>= 1) t += __shfl_xor_sync(SG_FULL_MASK, t, i);
    if (lane == 0 && blockIdx.x * 32 + warp < KC) out[blockIdx.x * 32 + warp] += t;
}
constexpr int kDecChunks = 128;
__global__ void decoder_reduce1_kernel(const float *__restrict__ part, int n_blocks, int KC,
                                       float *__restrict__ chunk_sums) {
    pdl_begin();
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    if (o >= KC) return;
    const int b0 = (int)((long long)c * n_blocks / kDecChunks), b1 = (int)((long long)(c + 1) * n_blocks / kDecChunks);
    float s = 0.f;
    for (int b = b0; b < b1; ++b) s += part[(size_t)b * KC + o];
    chunk_sums[(size_t)c * KC + o] = s;
}
__global__ void decoder_reduce2_kernel(const float *__restrict__ chunk_sums, int KC, float *__restrict__ out) {
    pdl_begin();
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= KC) return;
    float s = 0.f;
    for (int c = 0; c < kDecChunks; ++c) s += chunk_sums[(size_t)c * KC + o];
    out[o] += s;
}

// Row pitches of the per-thread stashes of dz (K floats) and S (C floats).  Rows stay
// 16-byte aligned, and the 8 rows written by a quarter-warp's 16-byte stores start in 8
// different 4-bank groups, so neither the stores nor the 16-byte reads of the decoder
// gradient loop have bank conflicts.
template <int K> __host__ __device__ constexpr int stash_pitch() { return K + 4; }

template <int C, int K>
__global__ void __launch_bounds__(kLossThreads) loss_pixel_kernel(PixelArgs a) {
    pdl_begin();
    static_assert(C % 4 == 0 && K % 4 == 0, "float4 stashes");
    constexpr int KP = stash_pitch<K>(), CP = stash_pitch<C>();
    __shared__ __align__(16) float s_dec[K * C];
    __shared__ float s_red[kLossThreads / 32];
    // only used when the decoder gradient is requested
    extern __shared__ __align__(16) float s_dyn[];
    float *s_dz = s_dyn;                          // kLossThreads x KP
    float *s_S = s_dyn + kLossThreads * KP;       // kLossThreads x CP
    float *s_dec_acc = s_S + kLossThreads * CP;   // K x C
    const bool has_dec = a.decoder != nullptr;
    for (int i = threadIdx.x; i < K * C; i += kLossThreads) s_dec[i] = has_dec ? a.decoder[i] : (i / C == i % C ? 1.f : 0.f);
    if (a.decoder_grad)
        for (int o = threadIdx.x; o < K * C; o += kLossThreads) s_dec_acc[o] = 0.f;
    const int blk = blockIdx.x;
    const int v = find_prefix(a.lv.pix_blk_off, a.lv.n, blk);
    const sg_view &vw = a.views[v];
    const int HW = vw.W * vw.H;
    const int p = (blk - a.lv.pix_blk_off[v]) * kLossThreads + threadIdx.x;
    const bool in = p < HW;
    const size_t p0 = (size_t)vw.pixel_offset;
    const int nd = a.counts[2 * v], nl = a.counts[2 * v + 1];
    __syncthreads();
    float l1d = 0.f, ce = 0.f;
    if (in) {
        const float gd = a.gt_depth[p0 + p];
        float gdep = 0.f;
        if (gd > 0.f) {
            const float d = a.depth[p0 + p] - gd;
            l1d = fabsf(d);
            gdep = a.w_depth * (d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f)) / (float)nd;
        }
        a.g_depth[p0 + p] = gdep;
    }
    if (a.ce) {
        float S[C], z[K];
        const int lab = in ? a.label[p0 + p] : -1;
#pragma unroll
        for (int c = 0; c < C; ++c) S[c] = in ? a.sem[(size_t)C * p0 + (size_t)c * HW + p] : 0.f;
        if (has_dec) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                float s = 0.f;
#pragma unroll
                for (int c = 0; c < C; ++c) s = fmaf(s_dec[k * C + c], S[c], s);
                z[k] = s;
            }
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) z[k] = S[k < C ? k : 0];
        }
        float zmax = -INFINITY;
#pragma unroll
        for (int k = 0; k < K; ++k) zmax = fmaxf(zmax, z[k]);
        // z <- exp(z - max); softmax = z / sum
        float se = 0.f, zl = 0.f;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (k == lab) zl = z[k] - zmax;
            z[k] = expf(z[k] - zmax);
            se += z[k];
        }
        const float lse_rel = logf(se);   // log-sum-exp minus zmax
        const bool valid = in && lab >= 0;
        if (valid) ce = lse_rel - zl;
        const float sc = valid ? a.w_sem / (float)nl : 0.f;
        const float inv = 1.f / se;
        float dS[C];
#pragma unroll
        for (int c = 0; c < C; ++c) dS[c] = 0.f;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float dz = sc * (z[k] * inv - (k == lab ? 1.f : 0.f));
            z[k] = dz;
            if (has_dec) {
#pragma unroll
                for (int c = 0; c < C; ++c) dS[c] = fmaf(s_dec[k * C + c], dz, dS[c]);
            } else if (k < C) {
                dS[k] = dz;
            }
        }
        if (in)
#pragma unroll
            for (int c = 0; c < C; ++c) a.g_sem[(size_t)C * p0 + (size_t)c * HW + p] = dS[c];
        if (a.decoder_grad) {
            float4 *dz4 = reinterpret_cast<float4 *>(s_dz + threadIdx.x * KP);
            float4 *S4 = reinterpret_cast<float4 *>(s_S + threadIdx.x * CP);
#pragma unroll
            for (int k = 0; k < K; k += 4) dz4[k / 4] = make_float4(z[k], z[k + 1], z[k + 2], z[k + 3]);
#pragma unroll
            for (int c = 0; c < C; c += 4) S4[c / 4] = make_float4(S[c], S[c + 1], S[c + 2], S[c + 3]);
            __syncwarp();
            // this warp's 32 pixels: each lane accumulates 4 x 4 blocks of dz_p S_p^T in registers
            const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
            constexpr int KB = K / 4, CB = C / 4;
            for (int blk4 = lane; blk4 < KB * CB; blk4 += 32) {
                const int k0 = (blk4 / CB) * 4, c0 = (blk4 % CB) * 4;
                float acc[4][4] = {};
#pragma unroll 4
                for (int t = warp * 32; t < warp * 32 + 32; ++t) {
                    const float4 dz = *reinterpret_cast<const float4 *>(s_dz + t * KP + k0);
                    const float4 sv = *reinterpret_cast<const float4 *>(s_S + t * CP + c0);
                    const float dzv[4] = {dz.x, dz.y, dz.z, dz.w}, svv[4] = {sv.x, sv.y, sv.z, sv.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int jj = 0; jj < 4; ++jj) acc[i][jj] = fmaf(dzv[i], svv[jj], acc[i][jj]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) atomicAdd(s_dec_acc + (k0 + i) * C + c0 + jj, acc[i][jj]);
            }
            __syncthreads();
            // this block's share of dL/ddecoder, reduced later in block order
            for (int o = threadIdx.x; o < K * C; o += kLossThreads)
                a.dec_partials[(size_t)blk * K * C + o] = s_dec_acc[o];
        }
    }
    const float t1 = block_sum(l1d, s_red);
    const float t2 = block_sum(ce, s_red);
    if (threadIdx.x < kPixSlots) {
        a.partials[2 * (kPixSlots * blk + threadIdx.x)] = threadIdx.x == 0 ? t1 : 0.f;
        a.partials[2 * (kPixSlots * blk + threadIdx.x) + 1] = threadIdx.x == 0 ? t2 : 0.f;
    }
}

// Cross-entropy through a linear decoder on the tensor cores.  One warp owns 32 consecutive
// pixels; with S (32 x C) their semantic features and W (K x C) the decoder:
//   Z = S W^T (logits), softmax and CE per pixel row on the accumulator fragments (a row's
//   K logits sit in the 4 lanes of a quad), dZ = scale (softmax - onehot) in place,
//   dS = dZ W with dZ taken from registers as the A operand (the k index of each 8-class
//   step is permuted so that A column tig / tig + 4 is class 2 tig / 2 tig + 1, and the B
//   rows follow the same permutation), and dW = dZ^T S with dZ transposed through shared
//   memory.  All three run as 3xTF32 MMAs (FP32-level accuracy).  Shared-memory operands
//   are read with ldmatrix (a 32-bit 8 x 4 tile is an 8 x 8 tile of 16-bit halves, and
//   ldmatrix hands thread t the word at row t / 4, column t % 4: exactly the (gid, tig)
//   element of an m16n8k8 TF32 fragment), and each decoder fragment serves both 16-pixel
//   tiles.
//
// Persistent: the warps of a resident grid walk the 32-pixel units of the image set, so the
// decoder is split into shared memory once per CTA and each warp keeps its share of dL/dW in
// registers across all of its units; no block barrier inside the loop.  Each warp stages its
// units in shared memory with asynchronous copies: the next unit's features, labels and
// depths are requested as soon as the current unit's last read of them (the dW contraction)
// is done, so they arrive while dS is computed and stored.  Each unit's two loss
// sums go to its own partial slot (kPixSlots per 256-pixel block); the CTA writes one K x C
// row of decoder-gradient partials at the end, its warps summed in a fixed order.
template <int C, int K>
struct CeLayout {
    static constexpr int CP = C + 4;   // W rows (class-major): 16-byte rows, conflict-free ldmatrix
    static constexpr int KT = K + 4;   // W^T rows (feature-major, classes permuted)
    static constexpr int PP = 32 + 4;  // dZ^T rows (class-major over the warp's 32 pixels)
    static constexpr int SP = 32 + 8;  // staged S rows (feature-major): conflict-free A fragments
    static constexpr int W_FLOATS = 2 * K * CP + 2 * C * KT;
    static constexpr int WARP_FLOATS = K * PP > K * C ? K * PP : K * C;
    // per warp: the unit's S (C x SP), labels, depth and GT depth (32 each)
    static constexpr int STAGE_FLOATS = C * SP + 3 * 32;
};

template <int C, int K>
__host__ __device__ constexpr int ce_mma_smem_floats() {
    return CeLayout<C, K>::W_FLOATS + (kLossThreads / 32) * (CeLayout<C, K>::WARP_FLOATS + CeLayout<C, K>::STAGE_FLOATS);
}

// Two CTAs per SM (up to 128 registers): with the per-warp stage, three CTAs at 80 registers
// spilled the warp's fragments and measured slower (loss 0.975 against 0.954 ms on the batched
// workload), and four at 64 slower still.
template <int C, int K>
__global__ void __launch_bounds__(kLossThreads, 2) ce_decoder_mma_kernel(PixelArgs a) {
    pdl_begin();
    static_assert(C % 8 == 0 && K % 16 == 0, "MMA tiles");
    using L = CeLayout<C, K>;
    constexpr int CP = L::CP, KT = L::KT, PP = L::PP, SP = L::SP;
    constexpr int NK = K / 8, NC = C / 8;
    extern __shared__ __align__(16) float s_dyn[];
    float *s_whi = s_dyn, *s_wlo = s_whi + K * CP;     // W [class][feature]
    float *s_thi = s_wlo + K * CP, *s_tlo = s_thi + C * KT;  // W^T [feature][permuted class]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gid = lane >> 2, tig = lane & 3;
    float *s_dz = s_dyn + L::W_FLOATS + warp * L::WARP_FLOATS;  // dZ^T [class][pixel]
    for (int i = threadIdx.x; i < K * C; i += kLossThreads) {
        uint32_t h, l;
        split_tf32(a.decoder[i], h, l);
        const int k = i / C, c = i % C;
        s_whi[k * CP + c] = __uint_as_float(h);
        s_wlo[k * CP + c] = __uint_as_float(l);
        // class k = 8 q + 2 j + e sits at column 8 q + j + 4 e of W^T
        const int kc = (k & ~7) + ((k & 7) >> 1) + 4 * (k & 1);
        s_thi[c * KT + kc] = __uint_as_float(h);
        s_tlo[c * KT + kc] = __uint_as_float(l);
    }
    __syncthreads();
    const bool dec_grad = a.decoder_grad != nullptr;
    // ldmatrix row addresses: lanes 0-7 give rows 0-7 of the first 8 x 4 tile, lanes 8-15 of
    // the second (4 columns further), lanes 16-31 (x4 only) the same 8 rows further down
    const int lr = lane & 7, lc = (lane >> 3) & 1, lh = lane >> 4;
    // this warp's share of dW = dZ^T S over all of its pixels (M = classes, N = features)
    float dw[K / 16][NC][4];
#pragma unroll
    for (int mt = 0; mt < K / 16; ++mt)
#pragma unroll
        for (int nt = 0; nt < NC; ++nt) dw[mt][nt][0] = dw[mt][nt][1] = dw[mt][nt][2] = dw[mt][nt][3] = 0.f;
    // work unit u = 32 pixels: slot u % kPixSlots of 256-pixel block u / kPixSlots; the warps
    // of the grid take units u = w, w + n_warps, ... (w the warp's grid-wide index)
    const int n_units = kPixSlots * a.lv.pix_blk_off[a.lv.n];
    const int n_warps = (int)gridDim.x * kPixSlots;
    float *s_st = s_dyn + L::W_FLOATS + (kLossThreads / 32) * L::WARP_FLOATS + warp * L::STAGE_FLOATS;
    int *s_lab = reinterpret_cast<int *>(s_st + C * SP);
    float *s_dep = s_st + C * SP + 32, *s_gd = s_dep + 32;
    // unit u: view v, its pixel count and offset, the unit's first pixel pw
    struct Unit {
        int v, HW, pw;
        size_t p0;
    };
    auto unit_of = [&](int u) {
        Unit x;
        const int blk = u / kPixSlots, slot = u % kPixSlots;
        x.v = find_prefix(a.lv.pix_blk_off, a.lv.n, blk);
        const sg_view &vw = a.views[x.v];
        x.HW = vw.W * vw.H;
        x.pw = (blk - a.lv.pix_blk_off[x.v]) * kLossThreads + slot * 32;
        x.p0 = (size_t)vw.pixel_offset;
        return x;
    };
    // lane l requests pixel pw + l of every feature plane, its label and both depths
    auto prefetch = [&](const Unit &x) {
        const int p = x.pw + lane;
        const bool ok = p < x.HW;
        const size_t q = x.p0 + (ok ? p : 0);
        const float *src = a.sem + (size_t)C * x.p0 + (ok ? p : 0);
#pragma unroll
        for (int f = 0; f < C; ++f) cp_async4(s_st + f * SP + lane, src + (size_t)f * x.HW, ok);
        cp_async4(s_lab + lane, a.label + q, ok);
        cp_async4(s_dep + lane, a.depth + q, ok);
        cp_async4(s_gd + lane, a.gt_depth + q, ok);
        cp_async_commit_group();
    };
    // (the unit found for the prefetch is the next iteration's: the search and the division of
    // the weight by the view's pixel count once a unit instead of twice and four times a lane:
    // batched workload 402 -> 383 us)
    int u = (int)blockIdx.x * kPixSlots + warp;
    Unit next{};
    if (u < n_units) {
        next = unit_of(u);
        prefetch(next);
    }
    for (; u < n_units; u += n_warps) {
        const Unit x = next;
        const int v = x.v, HW = x.HW, pw = x.pw;
        const size_t p0 = x.p0;
        const int nd = a.counts[2 * v], nl = a.counts[2 * v + 1];
        const float scale = a.w_sem / (float)nl;
        cp_async_wait_groups<0>();
        __syncwarp();
        float l1d = 0.f, ce = 0.f;
        {
            const int p = pw + lane;
            if (p < HW) {
                const float gd = s_gd[lane];
                float gdep = 0.f;
                if (gd > 0.f) {
                    const float d = s_dep[lane] - gd;
                    l1d = fabsf(d);
                    gdep = a.w_depth * (d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f)) / (float)nd;
                }
                a.g_depth[p0 + p] = gdep;
            }
        }
        // staged S (pixels past the view's end read as zero)
        auto S = [&](int px, int f) -> float { return s_st[f * SP + px]; };
        // ---- Z = S W^T: M = pixels (2 x 16), N = classes, K = features ----
        // all of the warp's feature loads are issued before the first MMA (memory-level parallelism)
        float sa[NC][2][4];
#pragma unroll
        for (int ks = 0; ks < NC; ++ks)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const int r0 = 16 * mt + gid, f0 = 8 * ks + tig;
                sa[ks][mt][0] = S(r0, f0);
                sa[ks][mt][1] = S(r0 + 8, f0);
                sa[ks][mt][2] = S(r0, f0 + 4);
                sa[ks][mt][3] = S(r0 + 8, f0 + 4);
            }
        int labs[2][2];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int p = pw + 16 * mt + gid + 8 * h;
                labs[mt][h] = p < HW ? s_lab[16 * mt + gid + 8 * h] : -1;
            }
        float z[2][NK][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int nt = 0; nt < NK; ++nt) z[mt][nt][0] = z[mt][nt][1] = z[mt][nt][2] = z[mt][nt][3] = 0.f;
#pragma unroll
        for (int ks = 0; ks < NC; ++ks) {
            uint32_t ah[2][4], al[2][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int i = 0; i < 4; ++i) split_tf32(sa[ks][mt][i], ah[mt][i], al[mt][i]);
#pragma unroll
            for (int nt = 0; nt < NK; ++nt) {
                // B (8 x 8): b0 (tig, gid) = W[8 nt + gid][8 ks + tig], b1 four features further
                const int w0 = (8 * nt + lr) * CP + 8 * ks + 4 * lc;
                uint32_t bh0, bh1, bl0, bl1;
                ldsm_x2(s_whi + w0, bh0, bh1);
                ldsm_x2(s_wlo + w0, bl0, bl1);
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) mma_tf32x3(z[mt][nt], ah[mt], al[mt], bh0, bh1, bl0, bl1);
            }
        }
        // ---- softmax, CE and dZ per pixel row (row 16 mt + gid + 8 h; classes 8 nt + 2 tig + c) ----
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int lab = labs[mt][h];
                float m = -INFINITY;
#pragma unroll
                for (int nt = 0; nt < NK; ++nt) m = fmaxf(m, fmaxf(z[mt][nt][2 * h], z[mt][nt][2 * h + 1]));
                m = fmaxf(m, __shfl_xor_sync(SG_FULL_MASK, m, 1));
                m = fmaxf(m, __shfl_xor_sync(SG_FULL_MASK, m, 2));
                float se = 0.f, zl = 0.f;
                bool has_lab = false;
#pragma unroll
                for (int nt = 0; nt < NK; ++nt)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int cls = 8 * nt + 2 * tig + c;
                        if (cls == lab) {
                            zl = z[mt][nt][2 * h + c] - m;
                            has_lab = true;
                        }
                        const float e = __expf(z[mt][nt][2 * h + c] - m);
                        z[mt][nt][2 * h + c] = e;
                        se += e;
                    }
                se += __shfl_xor_sync(SG_FULL_MASK, se, 1);
                se += __shfl_xor_sync(SG_FULL_MASK, se, 2);
                const bool valid = lab >= 0;
                if (valid && has_lab) ce += logf(se) - zl;
                const float sc = valid ? scale : 0.f;
                const float inv = 1.f / se;
#pragma unroll
                for (int nt = 0; nt < NK; ++nt)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int cls = 8 * nt + 2 * tig + c;
                        z[mt][nt][2 * h + c] = sc * (z[mt][nt][2 * h + c] * inv - (cls == lab ? 1.f : 0.f));
                    }
            }
        }
        // the two loss sums of this unit
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            l1d += __shfl_xor_sync(SG_FULL_MASK, l1d, o);
            ce += __shfl_xor_sync(SG_FULL_MASK, ce, o);
        }
        if (lane == 0) {
            a.partials[2 * u] = l1d;
            a.partials[2 * u + 1] = ce;
        }
        // ---- dW += dZ^T S: M = classes, N = features, K = pixels ----
        if (dec_grad) {
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int nt = 0; nt < NK; ++nt)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        s_dz[(8 * nt + 2 * tig + (i & 1)) * PP + 16 * mt + gid + 8 * (i >> 1)] = z[mt][nt][i];
            __syncwarp();
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                uint32_t bh[NC][2], bl[NC][2];
#pragma unroll
                for (int nt = 0; nt < NC; ++nt) {
                    split_tf32(S(8 * ks + tig, 8 * nt + gid), bh[nt][0], bl[nt][0]);
                    split_tf32(S(8 * ks + tig + 4, 8 * nt + gid), bh[nt][1], bl[nt][1]);
                }
#pragma unroll
                for (int mt = 0; mt < K / 16; ++mt) {
                    // A (16 x 8): rows = classes 16 mt .., columns = pixels 8 ks ..
                    uint32_t ar[4], ah[4], al[4];
                    ldsm_x4(s_dz + (16 * mt + lr + 8 * lc) * PP + 8 * ks + 4 * lh, ar);
#pragma unroll
                    for (int i = 0; i < 4; ++i) split_tf32(__uint_as_float(ar[i]), ah[i], al[i]);
#pragma unroll
                    for (int nt = 0; nt < NC; ++nt)
                        mma_tf32x3(dw[mt][nt], ah, al, bh[nt][0], bh[nt][1], bl[nt][0], bl[nt][1]);
                }
            }
            __syncwarp();  // the stash is rewritten by the next unit
        }
        // the stage's last read is done: request the next unit (it arrives during dS)
        __syncwarp();
        if (u + n_warps < n_units) {
            next = unit_of(u + n_warps);
            prefetch(next);
        }
        // ---- dS = dZ W: M = pixels, N = features, K = classes (permuted within each 8-class step) ----
        {
            float ds[2][NC][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int nt = 0; nt < NC; ++nt) ds[mt][nt][0] = ds[mt][nt][1] = ds[mt][nt][2] = ds[mt][nt][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < NK; ++ks) {
                uint32_t ah[2][4], al[2][4];
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    // A column tig = class 8 ks + 2 tig (d0 / d2), column tig + 4 = class 8 ks + 2 tig + 1 (d1 / d3)
                    split_tf32(z[mt][ks][0], ah[mt][0], al[mt][0]);
                    split_tf32(z[mt][ks][2], ah[mt][1], al[mt][1]);
                    split_tf32(z[mt][ks][1], ah[mt][2], al[mt][2]);
                    split_tf32(z[mt][ks][3], ah[mt][3], al[mt][3]);
                }
#pragma unroll
                for (int nt = 0; nt < NC; ++nt) {
                    // B (8 x 8): b0 (tig, gid) = W[8 ks + 2 tig][8 nt + gid], b1 = W[8 ks + 2 tig + 1][..]:
                    // rows 8 nt + gid, columns 8 ks + tig (+ 4) of the permuted W^T
                    const int t0 = (8 * nt + lr) * KT + 8 * ks + 4 * lc;
                    uint32_t bh0, bh1, bl0, bl1;
                    ldsm_x2(s_thi + t0, bh0, bh1);
                    ldsm_x2(s_tlo + t0, bl0, bl1);
#pragma unroll
                    for (int mt = 0; mt < 2; ++mt) mma_tf32x3(ds[mt][nt], ah[mt], al[mt], bh0, bh1, bl0, bl1);
                }
            }
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int nt = 0; nt < NC; ++nt)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int p = pw + 16 * mt + gid + 8 * (i >> 1);
                        const int f = 8 * nt + 2 * tig + (i & 1);
                        if (p < HW) a.g_sem[(size_t)C * p0 + (size_t)f * HW + p] = ds[mt][nt][i];
                    }
        }
    }
    if (!dec_grad) return;
    // this CTA's share of dL/dW: every warp's fragments into its own stash, then summed over
    // the warps in order (deterministic), one K x C row per CTA
#pragma unroll
    for (int mt = 0; mt < K / 16; ++mt)
#pragma unroll
        for (int nt = 0; nt < NC; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                s_dz[(16 * mt + gid + 8 * (i >> 1)) * C + 8 * nt + 2 * tig + (i & 1)] = dw[mt][nt][i];
    __syncthreads();
    const float *s_all = s_dyn + L::W_FLOATS;
    for (int o = threadIdx.x; o < K * C; o += kLossThreads) {
        float s = 0.f;
        for (int w = 0; w < kLossThreads / 32; ++w) s += s_all[w * L::WARP_FLOATS + o];
        a.dec_partials[(size_t)blockIdx.x * K * C + o] = s;
    }
}

// Resident grid of the persistent decoder kernel (at most one CTA per pixel block); returns
// the number of CTAs, i.e. of decoder-gradient partial rows.
template <int C, int K>
static int launch_ce_mma(PixelArgs &pa, int blocks, cudaStream_t st) {
    const size_t smem = sizeof(float) * ce_mma_smem_floats<C, K>();
    static int resident = 0;
    if (!resident) {
        cudaFuncSetAttribute(ce_decoder_mma_kernel<C, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int dev = 0, sms = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ce_decoder_mma_kernel<C, K>, kLossThreads, smem);
        resident = (per_sm > 0 ? per_sm : 1) * (sms > 0 ? sms : 1);
    }
    const int grid = blocks < resident ? blocks : resident;
    launch_pdl(ce_decoder_mma_kernel<C, K>, grid, kLossThreads, smem, st, pa);
    return grid;
}

struct FinalArgs {
    const float *ssim, *pix;  // partial arrays
    int rgb_groups, sem_groups, n_tiles;
    const int *counts;
    const sg_view *views;
    LossViews lv;
    int C, sem_mode;
    float lambda_r, lambda_s, w_depth, w_sem;
    float *terms;
    uint32_t *status;  // non-NULL: flag non-finite loss terms (SG_STATUS_NUMERIC)
};

// A sum of floats with the rounding errors kept beside it (about 48 bits).
struct PairSum {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float x) {
        const DF s = two_sum(hi, x);
        hi = s.hi;
        lo += s.lo;
    }
    __device__ __forceinline__ void add(float h, float l) {
        add(h);
        lo += l;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// A view's partial sums and its loss terms by a cluster of kFinalCtas CTAs, their shares added
// in rank order through distributed shared memory.  Bound by the latency of the partials'
// loads; the sums over a CTA are pairs of floats, because an SM does only a few double additions
// per clock (12.7 us with doubles, 637x477 x 3 levels 9.7 -> 7.2): 1200x680 x 3 levels with
// one CTA per view took 38 us (25 us less of the loss with a 32-class decoder).  A warp whose pairs
// leave the range of a float (sums beyond it, or a partial that is not finite) sums again in
// double.
constexpr int kFinalCtas = 8;
__global__ void __cluster_dims__(kFinalCtas, 1, 1) __launch_bounds__(kLossThreads) loss_finalize_kernel(FinalArgs a) {
    pdl_begin();
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const int v = blockIdx.x / kFinalCtas, rank = blockIdx.x % kFinalCtas;
    const int first = rank * kLossThreads + (int)threadIdx.x;
    constexpr int kStride = kFinalCtas * kLossThreads;
    const sg_view &vw = a.views[v];
    const double HW = (double)vw.W * vw.H;
    __shared__ double s_w[kLossThreads / 32][4];
    __shared__ double s_part[kFinalCtas][4];  // (rank 0's holds the shares)
    // add(k, x) for the thread's partials: colour, semantics, depth L1, CE
    auto gather = [&](auto add) {
        for (int i = a.lv.tile_off[v] + first; i < a.lv.tile_off[v + 1]; i += kStride)
#pragma unroll
            for (int g = 0; g < kSsimGroups; ++g)
                if (g < a.rgb_groups + a.sem_groups) {
                    const float t = a.ssim[(size_t)g * a.n_tiles + i];
                    if (g < a.rgb_groups) add(0, t); else add(1, t);
                }
        // the per-unit (depth L1, CE) sums: two units per 16-byte load, four loads in flight per
        // thread, summed in a fixed order
        const float4 *p4 = reinterpret_cast<const float4 *>(a.pix);
        const int s1 = kPixSlots * a.lv.pix_blk_off[v + 1] / 2;
        for (int i = kPixSlots * a.lv.pix_blk_off[v] / 2 + first; i < s1; i += 4 * kStride) {
            float4 q[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                q[k] = i + k * kStride < s1 ? p4[i + k * kStride] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                add(2, q[k].x);
                add(2, q[k].z);
                add(3, q[k].y);
                add(3, q[k].w);
            }
        }
    };
    // the four sums side by side: warp trees, then one thread each over the warps and the CTAs, in
    // order and in double
    PairSum part[4];
    gather([&](int k, float x) { part[k].add(x); });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < 4; ++k)
            part[k].add(__shfl_down_sync(SG_FULL_MASK, part[k].hi, o), __shfl_down_sync(SG_FULL_MASK, part[k].lo, o));
    double sum[4];
    bool finite = true;  // (lane 0's sums take in every lane's: one that is not finite stays so)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        sum[k] = part[k].value();
        finite = finite && isfinite(part[k].hi);
    }
    if (!__shfl_sync(SG_FULL_MASK, (int)finite, 0)) {
#pragma unroll
        for (int k = 0; k < 4; ++k) sum[k] = 0.0;
        gather([&](int k, float x) { sum[k] += x; });
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < 4; ++k) sum[k] += __shfl_down_sync(SG_FULL_MASK, sum[k], o);
    }
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int k = 0; k < 4; ++k) s_w[threadIdx.x >> 5][k] = sum[k];
    cluster.sync();  // (rank 0 runs: its shared memory can be written)
    const int k = threadIdx.x;
    if (k < 4) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < kLossThreads / 32; ++w) t += s_w[w][k];
        *cluster.map_shared_rank(&s_part[rank][k], 0) = t;
    }
    cluster.sync();
    if (rank != 0 || threadIdx.x >= 32) return;
    double t = 0.0;
    if (k < 4)
#pragma unroll
        for (int r = 0; r < kFinalCtas; ++r) t += s_part[r][k];
    // thread k's term: colour, semantic images, depth, cross-entropy
    const int nd = a.counts[2 * v], nl = a.counts[2 * v + 1];
    const double n = k == 0 ? 3.0 * HW : k == 1 ? (double)a.C * HW : (double)(k == 2 ? nd : nl);
    double L = n > 0.0 ? t / n : 0.0;
    // (1 - lambda) L1 + lambda (1 - SSIM)
    if (k == 0) L += a.lambda_r;
    if (k == 1) L = a.w_sem * (L + a.lambda_s);
    if (k == 2) L *= a.w_depth;
    if (k == 3) L *= a.w_sem;
    const double L_r = __shfl_sync(SG_FULL_MASK, L, 0), L_d = __shfl_sync(SG_FULL_MASK, L, 2);
    const double L_s = __shfl_sync(SG_FULL_MASK, L, a.sem_mode == 0 ? 3 : 1);
    if (k == 0) {
        a.terms[4 * v + 0] = (float)L_r;
        a.terms[4 * v + 1] = (float)L_d;
        a.terms[4 * v + 2] = (float)L_s;
        a.terms[4 * v + 3] = (float)(L_r + L_d + L_s);
        if (a.status && !isfinite(L_r + L_d + L_s)) atomicOr(a.status, SG_STATUS_NUMERIC);
    }
}

// ---------------------------------------------------------------------------------------

static size_t ssim_smem() { return sizeof(float) * (2 * kXH * kXP + 5 * kXH * kMP); }

static void make_loss_views(const sg_view *vh, int n_views, LossViews &lv) {
    lv.n = n_views;
    lv.tile_off[0] = 0;
    lv.pix_blk_off[0] = 0;
    for (int v = 0; v < n_views; ++v) {
        const int tx = (vh[v].W + kLTW - 1) / kLTW, ty = (vh[v].H + kLTH - 1) / kLTH;
        lv.tile_off[v + 1] = lv.tile_off[v] + tx * ty;
        lv.pix_blk_off[v + 1] = lv.pix_blk_off[v] + (vh[v].W * vh[v].H + kLossThreads - 1) / kLossThreads;
    }
}

static size_t loss_ws_bytes(int n_views, int n_tiles, int n_blocks, int KC) {
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    return al(sizeof(int) * 2 * n_views) + 2 * al(sizeof(float) * (kSsimGroups / 2) * n_tiles) +
           al(sizeof(float) * 2 * kPixSlots * n_blocks) + al(sizeof(float) * (size_t)n_blocks * KC) +
           al(sizeof(float) * (size_t)kDecChunks * KC);
}

// Decoder-gradient floats the loss keeps per pixel block: K x C partials in cross-entropy
// mode when a decoder gradient is requested, none otherwise (paper mode has no decoder).
int loss_decoder_partials(const sg_loss_config *lc, int C) {
    return (lc->sem_mode == 0 && lc->decoder_grad) ? lc->n_classes * C : 0;
}

// Exact scratch bytes when KC decoder-gradient floats per block are needed (0 = none).
size_t loss_workspace_size_kc(const sg_view *vh, int n_views, int KC) {
    LossViews lv;
    make_loss_views(vh, n_views, lv);
    return loss_ws_bytes(n_views, lv.tile_off[n_views], lv.pix_blk_off[n_views], KC);
}

size_t loss_workspace_size(const sg_view *vh, int n_views, int C, int n_classes) {
    LossViews lv;
    make_loss_views(vh, n_views, lv);
    const int K = n_classes > C ? n_classes : C;
    return loss_ws_bytes(n_views, lv.tile_off[n_views], lv.pix_blk_off[n_views], K * C);
}

template <int C, int K>
static void launch_pixel_t(PixelArgs &pa, int blocks, cudaStream_t st) {
    const size_t full = sizeof(float) * (kLossThreads * (stash_pitch<K>() + stash_pitch<C>()) + K * C);
    const size_t dyn = pa.decoder_grad ? full : 0;
    static bool attr = false;
    if (!attr) {
        cudaFuncSetAttribute(loss_pixel_kernel<C, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)full);
        attr = true;
    }
    launch_pdl(loss_pixel_kernel<C, K>, blocks, kLossThreads, dyn, st, pa);
}

// Launches the per-pixel loss kernel; returns the number of decoder-gradient partial rows it
// writes (its CTAs), or 0 for an unsupported (C, K).
static int launch_pixel(PixelArgs &pa, int blocks, cudaStream_t st) {
    const int C = pa.C, K = pa.K;
    if (pa.ce && pa.decoder) {
#define SG_CE(c, k) if (C == c && K == k) return launch_ce_mma<c, k>(pa, blocks, st);
        SG_CE(16, 16) SG_CE(16, 32) SG_CE(32, 32)
#undef SG_CE
    }
#define SG_PIX(c, k) if (C == c && K == k) { launch_pixel_t<c, k>(pa, blocks, st); return blocks; }
    SG_PIX(4, 4) SG_PIX(8, 8) SG_PIX(16, 16) SG_PIX(16, 32) SG_PIX(32, 32) SG_PIX(40, 40)
#undef SG_PIX
    return 0;
}

sg_status launch_loss(const sg_images *r, const sg_targets *gt, const sg_view *views,
                      const sg_view *vh, int n_views, int C, const sg_loss_config *lc,
                      float *terms, sg_images *dL, void *ws, size_t ws_bytes, uint32_t *status,
                      cudaStream_t st) {
    LossViews lv;
    make_loss_views(vh, n_views, lv);
    const int n_tiles = lv.tile_off[n_views], n_blocks = lv.pix_blk_off[n_views];
    char *base = (char *)ws;
    size_t off = 0;
    auto take = [&](size_t bytes) { char *p = base + off; off += (bytes + 255) & ~(size_t)255; return p; };
    int *counts = (int *)take(sizeof(int) * 2 * n_views);
    float *p_ssim = (float *)take(sizeof(float) * (kSsimGroups / 2) * n_tiles);
    take(sizeof(float) * (kSsimGroups / 2) * n_tiles);  // (its second half)
    float *p_pix = (float *)take(sizeof(float) * 2 * kPixSlots * n_blocks);
    const int ce = lc->sem_mode == 0;
    const int K = ce ? lc->n_classes : C;
    const int KC = loss_decoder_partials(lc, C);
    float *p_dec = (float *)take(sizeof(float) * (size_t)n_blocks * KC);
    float *p_dec2 = (float *)take(sizeof(float) * (size_t)kDecChunks * KC);
    if (loss_ws_bytes(n_views, n_tiles, n_blocks, KC) > ws_bytes) {
        set_error("pyramid_loss: workspace %zu bytes < %zu needed", ws_bytes,
                  loss_ws_bytes(n_views, n_tiles, n_blocks, KC));
        return SG_ERR_CAPACITY;
    }
    cudaMemsetAsync(counts, 0, sizeof(int) * 2 * n_views, st);
    static bool attr = false;
    if (!attr) {
        cudaFuncSetAttribute(ssim_l1_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssim_smem());
        attr = true;
    }
    // cross-entropy: a group per colour plane; otherwise one for the colour planes and three for
    // the semantic ones
    const int rgb_groups = ce ? 3 : 1, sem_groups = ce ? 0 : std::min(C, kSsimGroups - rgb_groups);
    const SsimArgs sa{{r->rgb, gt->rgb, dL->rgb, 3, 1.f - lc->lambda_r, lc->lambda_r, lc->lambda_r},
                      {r->sem, gt->sem, dL->sem, C, lc->w_sem * (1.f - lc->lambda_s), lc->w_sem * lc->lambda_s,
                       lc->lambda_s},
                      rgb_groups, sem_groups, views, lv, p_ssim, gt->depth, ce ? gt->label : nullptr, counts};
    launch_pdl(ssim_l1_kernel, dim3(n_tiles, rgb_groups + sem_groups), kLossThreads, ssim_smem(), st, sa);
    PixelArgs pa{r->depth, gt->depth, r->sem, gt->label, dL->depth, dL->sem, lc->decoder,
                 KC ? lc->decoder_grad : nullptr, C, K, ce, lc->w_depth, lc->w_sem, counts, views, lv, p_pix, p_dec};
    const int dec_rows = launch_pixel(pa, n_blocks, st);
    if (!dec_rows) {
        set_error("pyramid_loss: unsupported (C=%d, classes=%d)", C, K);
        return SG_ERR_INVALID_ARG;
    }
    if (ce && lc->decoder_grad) {
        if (dec_rows <= kDecRows) {
            launch_pdl(decoder_reduce_kernel, (KC + 31) / 32, 1024, 0, st, p_dec, dec_rows, KC, lc->decoder_grad);
            count_launches(1);
        } else {
            launch_pdl(decoder_reduce1_kernel, dim3((KC + 127) / 128, kDecChunks), 128, 0, st, p_dec, dec_rows, KC, p_dec2);
            launch_pdl(decoder_reduce2_kernel, (KC + 127) / 128, 128, 0, st, p_dec2, KC, lc->decoder_grad);
            count_launches(2);
        }
    }
    FinalArgs fa{p_ssim, p_pix, rgb_groups, sem_groups, n_tiles, counts, views, lv, C, lc->sem_mode,
                 lc->lambda_r, lc->lambda_s, lc->w_depth, lc->w_sem, terms, status};
    launch_pdl(loss_finalize_kernel, n_views * kFinalCtas, kLossThreads, 0, st, fa);
    count_launches(3);
    return check_launch("pyramid_loss");
}

// ---------------------------------------------------------------------------------------
// Eq. 4-6 pyramid: level l+1 from level l of the same camera
// ---------------------------------------------------------------------------------------

__global__ void pyramid_down_kernel(float *rgb, float *depth, int *label, float *sem, int n_sem,
                                    sg_view src, sg_view dst) {
    pdl_begin();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= dst.W || y >= dst.H) return;
    const size_t sHW = (size_t)src.W * src.H, dHW = (size_t)dst.W * dst.H;
    const size_t s00 = (size_t)(2 * y) * src.W + 2 * x;
    const size_t idx[4] = {s00, s00 + 1, s00 + src.W, s00 + src.W + 1};
    const size_t o = (size_t)y * dst.W + x;
    for (int c = 0; c < 3; ++c) {
        const float *s = rgb + 3 * (size_t)src.pixel_offset + c * sHW;
        rgb[3 * (size_t)dst.pixel_offset + c * dHW + o] = 0.25f * ((s[idx[0]] + s[idx[1]]) + (s[idx[2]] + s[idx[3]]));
    }
    for (int c = 0; c < n_sem; ++c) {
        const float *s = sem + (size_t)n_sem * src.pixel_offset + c * sHW;
        sem[(size_t)n_sem * dst.pixel_offset + c * dHW + o] = 0.25f * ((s[idx[0]] + s[idx[1]]) + (s[idx[2]] + s[idx[3]]));
    }
    float ds = 0.f;
    int dn = 0;
    for (int k = 0; k < 4; ++k) {
        const float d = depth[src.pixel_offset + idx[k]];
        if (d > 0.f) { ds += d; ++dn; }
    }
    depth[dst.pixel_offset + o] = dn ? ds / (float)dn : 0.f;
    if (label) {
        int l[4];
        for (int k = 0; k < 4; ++k) l[k] = label[src.pixel_offset + idx[k]];
        int best = -1, bc = 0;
        for (int k = 0; k < 4; ++k) {
            if (l[k] < 0) continue;
            int c = 0;
            for (int j = 0; j < 4; ++j) c += l[j] == l[k];
            if (c > bc || (c == bc && l[k] < best)) { best = l[k]; bc = c; }
        }
        label[dst.pixel_offset + o] = best;
    }
}

sg_status launch_pyramid(float *rgb, float *depth, int *label, float *sem, int n_sem,
                         const sg_view *vh, int n_views, cudaStream_t st) {
    int max_level = 0;
    for (int v = 0; v < n_views; ++v) max_level = vh[v].level > max_level ? vh[v].level : max_level;
    for (int l = 1; l <= max_level; ++l)
        for (int v = 0; v < n_views; ++v) {
            if (vh[v].level != l) continue;
            int s = -1;
            for (int u = 0; u < n_views; ++u)
                if (vh[u].camera == vh[v].camera && vh[u].level == l - 1) s = u;
            if (s < 0) {
                set_error("build_pyramid: view %d (camera %d, level %d) has no parent level", v, vh[v].camera, l);
                return SG_ERR_INVALID_ARG;
            }
            const dim3 blk(32, 8), grd((vh[v].W + 31) / 32, (vh[v].H + 7) / 8);
            launch_pdl(pyramid_down_kernel, grd, blk, 0, st, rgb, depth, label, sem, n_sem, vh[s], vh[v]);
            count_launches(1);
        }
    return check_launch("build_pyramid");
}

// ---------------------------------------------------------------------------------------
// Adam
// ---------------------------------------------------------------------------------------

__global__ void adam_kernel(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                            float bc1, float bc2) {
    pdl_begin();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    }
}

// All parameter groups in one launch; the gradient is zeroed after it is read, ready for
// the next iteration's accumulation.
struct AdamGroups {
    sg_adam_group g[SG_ADAM_MAX_GROUPS];
    int64_t start[SG_ADAM_MAX_GROUPS + 1];  // prefix of element counts
    int n;
    uint32_t *status;  // non-NULL: flag non-finite gradients (SG_STATUS_NUMERIC)
};

__global__ void adam_multi_kernel(AdamGroups G, float b1, float b2, float eps, float bc1, float bc2,
                                  int zero_grad) {
    pdl_begin();
    const int64_t total = G.start[G.n];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        int k = 0;
        while (k + 1 < G.n && i >= G.start[k + 1]) ++k;
        const sg_adam_group &q = G.g[k];
        const int64_t j = i - G.start[k];
        const float gi = q.grad[j];
        if (G.status) flag_status(!isfinite(gi), G.status, SG_STATUS_NUMERIC);
        const float mi = b1 * q.m[j] + (1.f - b1) * gi;
        const float vi = b2 * q.v[j] + (1.f - b2) * gi * gi;
        q.m[j] = mi;
        q.v[j] = vi;
        q.param[j] -= q.lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
        if (zero_grad) q.grad[j] = 0.f;
    }
}

// The same update, four elements per thread with 16-byte loads and stores: start[] counts
// quads (every group holds a multiple of 4 elements, all arrays 16-byte aligned).
// ibc1, ibc2: reciprocals of the bias corrections.  sqrt and the division use the fast
// hardware approximations (a few ulp; the update is a step size, not a value the path
// returns); sqrt(0) is taken as 0 so that a parameter with no gradient history stays put.
__device__ __forceinline__ float adam_one(float &m, float &v, float p, float g, float lr, float b1, float b2,
                                          float eps, float ibc1, float ibc2) {
    m = b1 * m + (1.f - b1) * g;
    v = b2 * v + (1.f - b2) * g * g;
    const float vh = v * ibc2;
    const float s = vh > 0.f ? vh * rsqrtf(vh) : 0.f;
    return p - lr * __fdividef(m * ibc1, s + eps);
}

__global__ void adam_multi4_kernel(AdamGroups G, float b1, float b2, float eps, float ibc1, float ibc2,
                                   int zero_grad) {
    pdl_begin();
    const int64_t total = G.start[G.n];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        int k = 0;
        while (k + 1 < G.n && i >= G.start[k + 1]) ++k;
        const sg_adam_group &q = G.g[k];
        const int64_t j = i - G.start[k];
        float4 *gp = reinterpret_cast<float4 *>(q.grad) + j;
        float4 *mp = reinterpret_cast<float4 *>(q.m) + j;
        float4 *vp = reinterpret_cast<float4 *>(q.v) + j;
        float4 *pp = reinterpret_cast<float4 *>(q.param) + j;
        const float4 g = *gp;
        if (G.status)
            flag_status(!isfinite(g.x) || !isfinite(g.y) || !isfinite(g.z) || !isfinite(g.w), G.status,
                        SG_STATUS_NUMERIC);
        float4 m = *mp, v = *vp, p = *pp;
        p.x = adam_one(m.x, v.x, p.x, g.x, q.lr, b1, b2, eps, ibc1, ibc2);
        p.y = adam_one(m.y, v.y, p.y, g.y, q.lr, b1, b2, eps, ibc1, ibc2);
        p.z = adam_one(m.z, v.z, p.z, g.z, q.lr, b1, b2, eps, ibc1, ibc2);
        p.w = adam_one(m.w, v.w, p.w, g.w, q.lr, b1, b2, eps, ibc1, ibc2);
        *mp = m;
        *vp = v;
        *pp = p;
        if (zero_grad) *gp = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

sg_status launch_adam_multi(const sg_adam_group *groups, int n, float b1, float b2, float eps, int step,
                            int zero_grad, uint32_t *status, cudaStream_t st) {
    AdamGroups G{};
    G.n = n;
    G.status = status;
    G.start[0] = 0;
    for (int k = 0; k < n; ++k) {
        G.g[k] = groups[k];
        G.start[k + 1] = G.start[k] + groups[k].n;
    }
    const float bc1 = 1.f - powf(b1, (float)step), bc2 = 1.f - powf(b2, (float)step);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    bool quads = true;
    for (int k = 0; k < n; ++k) {
        const sg_adam_group &q = groups[k];
        quads = quads && q.n % 4 == 0 && ((uintptr_t)q.param | (uintptr_t)q.grad | (uintptr_t)q.m |
                                          (uintptr_t)q.v) % 16 == 0;
    }
    if (quads)
        for (int k = 0; k <= n; ++k) G.start[k] /= 4;
    int64_t blocks = (G.start[n] + 255) / 256;
    if (blocks > 8 * (int64_t)sms) blocks = 8 * (int64_t)sms;
    if (blocks > 0) {
        if (quads)
            launch_pdl(adam_multi4_kernel, (int)blocks, 256, 0, st, G, b1, b2, eps, 1.f / bc1, 1.f / bc2, zero_grad);
        else
            launch_pdl(adam_multi_kernel, (int)blocks, 256, 0, st, G, b1, b2, eps, bc1, bc2, zero_grad);
        count_launches(1);
    }
    return check_launch("adam_multi");
}

sg_status launch_adam(float *p, const float *g, float *m, float *v, int64_t n, float lr, float b1,
                      float b2, float eps, int step, cudaStream_t st) {
    const float bc1 = 1.f - powf(b1, (float)step), bc2 = 1.f - powf(b2, (float)step);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t blocks = (n + 255) / 256;
    if (blocks > 8 * (int64_t)sms) blocks = 8 * (int64_t)sms;
    if (blocks > 0) {
        launch_pdl(adam_kernel, (int)blocks, 256, 0, st, p, g, m, v, n, lr, b1, b2, eps, bc1, bc2);
        count_launches(1);
    }
    return check_launch("adam");
}

}  // namespace sg
