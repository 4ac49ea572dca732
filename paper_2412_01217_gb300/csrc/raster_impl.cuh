// raster_impl.cuh -- tile compositing of RGB, depth and C semantic channels (Eq. 7-9) and its
// adjoint (Sec. III-D backpropagation), templated on the semantic width C and, in the
// forward, on the number of pixels each thread owns (PPT = 1, 2 or 4; the adjoint has one).
//
// One CTA owns one screen tile of one view-level.  Every view-level of every keyframe is
// addressed through one global tile id, so a single launch renders the whole pyramid of
// all keyframes; with `persistent` set, a grid of resident CTAs pulls tile ids from an
// atomic work counter.  Each warp owns an 8 x (4 PPT) pixel sub-tile: lane l has the PPT
// pixels (l mod 8, l div 8 + 4k), k < PPT.  A whole warp skips a Gaussian whose footprint
// misses its sub-tile (one uniform test), and with PPT > 1 every per-Gaussian cost
// (shared-memory loads) is shared by PPT pixels.
//
// Forward: the tile's depth-sorted list is walked in batches the CTA stages into shared
// memory; each pixel composites front to back and stops when T would fall below T_min;
// the CTA leaves the tile when all pixels are done.  Saved per pixel: T_final, last (list
// entries examined up to and including the last contributor), contributor count.
//
// Backward: back to front from the tile's largest `last`.  Each pixel rebuilds T by
// dividing by (1 - alpha) and tracks only the scalar a = g . A of the background-weighted
// suffix colour A.  Per chunk of 16 list entries every lane writes, for each entry, its
// weight w = alpha T and s = dL/dsigma into two chunk buffers; the three sums over the
// warp's pixels -- g . f, the 4 + C feature gradients dF = W^T G (colour, depth, semantics)
// and the six pixel moments of s, which give the 2D-mean, conic and opacity gradients --
// then run on the tensor cores (mma.m16n8k8, TF32 split into hi + lo parts for FP32-level
// accuracy); no shuffles in the per-entry loop.
#pragma once

#include "raster.cuh"

namespace sg {

// Stages entries [b0, b0 + cnt) of a tile's list.  Per entry:
//   s_geo0 = (ui - px0, vi - py0, uf, vf): integer part of the 2D mean relative to the tile
//            origin (exact in float) and its float fraction,
//   s_geo1 = (m00, m10, m11, opacity),
//   s_geo2 = (u, v, ex, ey): approximate tile-relative mean and the projection's conservative
//            half extents of the alpha >= alpha_min region (warp-level skip test only),
// the 4 + C features, and (backward) the Gaussian index.
template <int NF>
__device__ __forceinline__ void load_batch(const RasterArgs &a, int C, int list_start, int b0, int cnt,
                                           int px0, int py0, uint32_t rec_base, float4 *s_geo0,
                                           float4 *s_geo1, float4 *s_geo2, float *s_feat, uint32_t *s_rec,
                                           int nthreads) {
    for (int j = threadIdx.x; j < cnt; j += nthreads) {
        const uint32_t rec = a.record[list_start + b0 + j] & a.rec_mask;
        const float4 g0 = a.geo[2 * (size_t)rec];
        const float4 g1 = a.geo[2 * (size_t)rec + 1];
        const uint32_t packed = __float_as_uint(g1.w);
        const float uI = (float)((int)(short)(packed & 0xffffu) - px0);
        const float vI = (float)((int)(short)(packed >> 16) - py0);
        const float2 ex = a.ext[rec];
        s_geo0[j] = make_float4(uI, vI, g0.x, g0.y);
        s_geo1[j] = make_float4(g1.x, g1.y, g1.z, g0.w);
        s_geo2[j] = make_float4(uI + g0.x, vI + g0.y, ex.x, ex.y);
        const uint32_t gi = rec - rec_base;  // every record of a tile belongs to its view-level
        const size_t ci = a.col_rec ? rec : gi;
        float *f = s_feat + (size_t)j * NF;
        f[0] = a.rgb[3 * ci];
        f[1] = a.rgb[3 * ci + 1];
        f[2] = a.rgb[3 * ci + 2];
        f[3] = g0.z;  // depth (camera z of the mean, Eq. 8)
        const float4 *s4 = reinterpret_cast<const float4 *>(a.sem + (size_t)(a.sem_rec ? rec : gi) * C);
        float4 *f4 = reinterpret_cast<float4 *>(f + 4);
#pragma unroll
        for (int k = 0; k < (NF - 4) / 4; ++k) f4[k] = s4[k];
        if (s_rec) s_rec[j] = rec;
    }
}

// Features of a warp's 16 chunk rows into s_feat by asynchronous copies: colour into f[0..2],
// semantics into f[4..]; f[3] (the depth) is left to the caller.  Lanes r and r + 16 copy row r
// (record rec), half of its words each.
template <int NF>
__device__ __forceinline__ void stage_features_async(const RasterArgs &a, uint32_t rec, uint32_t rec_base,
                                                     float *s_feat) {
    constexpr int C = NF - 4, NS = C / 4;
    const int lane = threadIdx.x & 31, h = lane >> 4;
    float *f = s_feat + (lane & 15) * NF;
    const float *sem = a.sem + (size_t)(a.sem_rec ? rec : rec - rec_base) * C;
    const float *rgb = a.rgb + 3 * (size_t)(a.col_rec ? rec : rec - rec_base);
#pragma unroll
    for (int q = 0; q < (NS + 1) / 2; ++q)
        if (2 * q + h < NS) cp_async16(f + 4 + 4 * (2 * q + h), sem + 4 * (2 * q + h));
    cp_async4(f + h, rgb + h, true);
    if (h) cp_async4(f + 2, rgb + 2, true);
}

// One list entry's geometry, relative to the tile: integer part (exact in float) and float
// fraction of the 2D mean, the conic form and the opacity.
struct EntryGeo {
    float ui, vi, uf, vf, m00, m10, m11, o;
};
__device__ __forceinline__ EntryGeo entry_geo(const float4 &g0, const float4 &g1) {  // staged rows
    return {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
}
__device__ __forceinline__ EntryGeo record_geo(const float4 &g0, const float4 &g1, int px0, int py0) {
    const uint32_t packed = __float_as_uint(g1.w);
    return {(float)((int)(short)(packed & 0xffffu) - px0), (float)((int)(short)(packed >> 16) - py0), g0.x, g0.y,
            g1.x, g1.y, g1.z, g0.w};
}

// Alphas of a chunk of 16 entries at the warp's 32 PPT pixels.  Lane l evaluates entry l % 16
// at the four columns x0 .. x0 + 3 (x0 = lx0, the left or the right half of the sub-tile by
// l / 16) of every row ly0 .. ly0 + 4 PPT - 1, so that dx and its square terms are formed once
// per column and dy once per row, and writes alpha (0 below alpha_min) to
// s_A[pixel * kAPitch + entry]; pixel 32 k + lane then reads its 16 alphas back as float4s.
// With a lane per pixel instead, every entry's eight geometry floats would be broadcast to all
// lanes through shared memory (8 data-pipe cycles per entry and warp), which bound both
// kernels (l1tex data pipe 80 % busy).  kAPitch: rows of 16 plus 4, conflict-free both ways.
// Returns whether the entry contributes to any of the lane's pixels.
constexpr int kAPitch = 20;
template <int PPT>
__device__ __forceinline__ bool chunk_alphas(const EntryGeo &g, float lx0, float ly0, float alpha_max, float alpha_min,
                                             float *s_A) {
    const int lane = threadIdx.x & 31;
    float *out = s_A + 4 * (lane >> 4) * kAPitch + (lane & 15);
    float dx[4], p1[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        dx[c] = __fsub_rn(__fsub_rn(lx0 + (float)c, g.ui), g.uf);
        const float p = __fmul_rn(g.m00, dx[c]);
        p1[c] = __fmul_rn(p, p);
    }
    float top = 0.f;
#pragma unroll
    for (int r = 0; r < 4 * PPT; ++r) {
        const float q = __fmul_rn(g.m11, __fsub_rn(__fsub_rn(ly0 + (float)r, g.vi), g.vf));
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float al = entry_alpha(g.m10, dx[c], q, p1[c], g.o, alpha_max, alpha_min);
            out[(8 * r + c) * kAPitch] = al;
            top = fmaxf(top, al);
        }
    }
    return top > 0.f;
}

// Persistent work queue: work_counter[0] hands out slots, work_counter[1] counts the CTAs
// that have drawn their terminating slot; the last of them zeroes both, so the queue is
// ready for the next launch without a memset.
__device__ __forceinline__ int next_item(const RasterArgs &a, int n_items, int &s_item) {
    if (!a.persistent) return blockIdx.x;
    if (threadIdx.x == 0) {
        const int slot = atomicAdd(a.work_counter, 1);
        if (slot >= n_items && atomicAdd(a.work_counter + 1, 1) == (int)gridDim.x - 1) {
            a.work_counter[0] = 0;
            a.work_counter[1] = 0;
        }
        s_item = slot;
    }
    __syncthreads();
    return s_item;
}

template <int PPT>
struct WarpTile {
    int lx, ly;      // first pixel of the thread, relative to the tile origin (others: ly + 4k)
    float cxw, cyw;  // centre of the warp's 8 x (4 PPT) sub-tile
    __device__ WarpTile(int tile_w) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const int warps_x = tile_w >> 3;
        const int wx = (warp % warps_x) * 8, wy = (warp / warps_x) * (4 * PPT);
        lx = wx + (lane & 7);
        ly = wy + (lane >> 3);
        cxw = wx + 3.5f;
        cyw = wy + 2.f * PPT - 0.5f;
    }
    // true if no pixel of the warp's sub-tile can reach alpha_min (g2 = u, v, ex, ey)
    __device__ __forceinline__ bool misses(const float4 &g2) const {
        return fabsf(g2.x - cxw) > g2.z + 3.5f || fabsf(g2.y - cyw) > g2.w + (2.f * PPT - 0.5f);
    }
    // The same, exactly for the ellipse: besides the box test, true if the minimum of
    // sigma = (m00 dx)^2 + (m10 dx + m11 dy)^2 over the rectangle spanned by the sub-tile's
    // pixel centres exceeds ln(o / alpha_min), so alpha < alpha_min at every pixel of the warp
    // (g1 = m00, m10, m11, o).  Conservative: the continuous rectangle contains every pixel
    // centre, and the 1e-3 margin on sigma covers rounding and the fast exponential.
    __device__ __forceinline__ bool misses(const float4 &g2, const float4 &g1, float ln_alpha_min) const {
        if (misses(g2)) return true;
        const float hx = 3.5f, hy = 2.f * PPT - 0.5f;
        // pixel offsets from the mean: dx in [x0, x1], dy in [y0, y1]
        const float x0 = cxw - g2.x - hx, x1 = cxw - g2.x + hx;
        const float y0 = cyw - g2.y - hy, y1 = cyw - g2.y + hy;
        if (x0 <= 0.f && x1 >= 0.f && y0 <= 0.f && y1 >= 0.f) return false;  // the mean is inside
        // sigma = A dx^2 + 2 B dx dy + Cq dy^2, a convex quadratic: with the mean outside, its
        // minimum over the rectangle lies on an edge, where it is a clamped 1D minimum
        const float A = g1.x * g1.x + g1.y * g1.y, B = g1.y * g1.z, Cq = g1.z * g1.z;
        const float iA = 1.f / A, iC = 1.f / Cq;
        auto on_x = [&](float dx) {
            const float dy = fminf(y1, fmaxf(y0, -B * dx * iC));
            return fmaf(A * dx, dx, fmaf(2.f * B * dx, dy, Cq * dy * dy));
        };
        auto on_y = [&](float dy) {
            const float dx = fminf(x1, fmaxf(x0, -B * dy * iA));
            return fmaf(A * dx, dx, fmaf(2.f * B * dx, dy, Cq * dy * dy));
        };
        const float smin = fminf(fminf(on_x(x0), on_x(x1)), fminf(on_y(y0), on_y(y1)));
        const float tau = __logf(g1.w) - ln_alpha_min;  // alpha >= alpha_min needs sigma <= tau
        return smin > tau * 1.0001f + 1e-3f;
    }
};

struct TileInfo {
    int v, px0, py0;
    const sg_view *vw;
};

__device__ __forceinline__ TileInfo tile_info(const RasterArgs &a, int item) {
    TileInfo t;
    t.v = find_view(a.views, a.n_views, item);
    t.vw = &a.views[t.v];
    const int local = item - t.vw->tile_offset;
    t.px0 = (local % t.vw->tiles_x) * a.tile_w;
    t.py0 = (local / t.vw->tiles_x) * a.tile_h;
    return t;
}

// Both kernels work on chunks of 16 consecutive entries of a warp's list.
constexpr int kChunk = 16;
// Ring of pending entries of a warp (< 16 pending + one 32-entry scan).
constexpr int kRing = 64;

// Half mode of the forward (8 x 8 tiles, one pixel per thread, lists with half masks): a
// CTA is one warp that owns one half (8 x 4 pixels) of a tile; it walks the tile's list front
// to back, queues (position, record) of the entries whose mask holds its half, and composites
// them 16 at a time with no block barrier, stopping as soon as its own 32 pixels are
// saturated; the next chunk's geometry (registers) and features (asynchronous copies into the
// other of two buffers) are requested before the current one is composited.  The per-pixel
// sequence of contributing entries, and so the output, is the same as with shared batches.

// acc[i] += w f[i] where w != 0 (a pixel without a contribution takes nothing from a
// non-finite feature)
template <int N>
__device__ __forceinline__ void fma_if(float *acc, float w, const float *f) {
    if constexpr (N >= 5) {
        asm("{\n\t.reg .pred p;\n\tsetp.ne.f32 p, %5, 0f00000000;\n\t"
            "@p fma.rn.f32 %0, %5, %6, %0;\n\t@p fma.rn.f32 %1, %5, %7, %1;\n\t@p fma.rn.f32 %2, %5, %8, %2;\n\t"
            "@p fma.rn.f32 %3, %5, %9, %3;\n\t@p fma.rn.f32 %4, %5, %10, %4;\n}\n"
            : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2]), "+f"(acc[3]), "+f"(acc[4])
            : "f"(w), "f"(f[0]), "f"(f[1]), "f"(f[2]), "f"(f[3]), "f"(f[4]));
        fma_if<N - 5>(acc + 5, w, f + 5);
    } else if constexpr (N == 4) {
        asm("{\n\t.reg .pred p;\n\tsetp.ne.f32 p, %4, 0f00000000;\n\t"
            "@p fma.rn.f32 %0, %4, %5, %0;\n\t@p fma.rn.f32 %1, %4, %6, %1;\n\t@p fma.rn.f32 %2, %4, %7, %2;\n\t"
            "@p fma.rn.f32 %3, %4, %8, %3;\n}\n"
            : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2]), "+f"(acc[3])
            : "f"(w), "f"(f[0]), "f"(f[1]), "f"(f[2]), "f"(f[3]));
    } else if constexpr (N >= 1) {
        asm("{\n\t.reg .pred p;\n\tsetp.ne.f32 p, %1, 0f00000000;\n\t@p fma.rn.f32 %0, %1, %2, %0;\n}\n"
            : "+f"(acc[0])
            : "f"(w), "f"(f[0]));
        fma_if<N - 1>(acc + 1, w, f + 1);
    }
}

// The four lanes of a quad share the feature sums of their pixels: lane s of the quad sums a
// quarter of the channels (one of r, g, b, depth; sem[16 q + 4 s ..], then sem[16 (C / 16) +
// (C % 16) / 4 s ..]) at all four pixels, whose weights it takes by shuffles.  Every feature is
// then loaded by one lane in four, a quarter of the shared-memory traffic of a lane that sums
// every channel of its own pixel; each pixel and channel still sums its entries in list order.
template <int C>
struct QuadChannels {
    static constexpr int NQ = C / 16, REM = C % 16 / 4, N = 1 + 4 * NQ + REM;
    static __device__ __forceinline__ void load(const float *row, int s, float (&f)[N]) {
        f[0] = row[s];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float4 t = *reinterpret_cast<const float4 *>(row + 4 + 16 * q + 4 * s);
            f[1 + 4 * q] = t.x; f[2 + 4 * q] = t.y; f[3 + 4 * q] = t.z; f[4 + 4 * q] = t.w;
        }
        if constexpr (REM == 2) {
            const float2 t = *reinterpret_cast<const float2 *>(row + 4 + 16 * NQ + 2 * s);
            f[1 + 4 * NQ] = t.x; f[2 + 4 * NQ] = t.y;
        } else if constexpr (REM == 1) {
            f[1 + 4 * NQ] = row[4 + 16 * NQ + s];
        }
    }
    // semantic channel of f[1 + i]
    static __device__ __forceinline__ int sem(int i, int s) {
        return i < 4 * NQ ? 16 * (i / 4) + 4 * s + i % 4 : 16 * NQ + REM * s + i - 4 * NQ;
    }
};

// v[0 .. 3] to the pixels x .. x + 3 of a row (p points at x; those from n_in on are outside)
__device__ __forceinline__ void store_quad(float *p, const float (&v)[4], int n_in) {
    if (n_in >= 4 && ((uintptr_t)p & 15) == 0) {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < n_in) p[j] = v[j];
    }
}

// shared memory of one forward warp (4-byte words): the ring (rows, or positions and records),
// the chunk's rows (or positions), the alphas, and in half mode two feature buffers
template <int C, int PPT, bool HALF>
__host__ __device__ constexpr int fwd_warp_words() {
    return (HALF ? 2 : 1) * kRing + kChunk + 32 * PPT * kAPitch + (HALF ? 2 * kChunk * (4 + C) : 0);
}

// One pixel per thread, C <= 16: 80 registers, i.e. 25 one-warp CTAs per SM in half mode (batched
// workload, C = 16, against 80: 6 % longer at 72, 12 % at 64 with spills, 7 % at the compiler's 99).
template <int C, int PPT>
__host__ __device__ constexpr int fwd_max_regs() { return PPT == 1 ? (C <= 16 ? 80 : 128) : PPT == 2 ? 168 : 255; }

template <int C, int PPT, bool HALF = false>
__global__ void __launch_bounds__(kMaxTileThreads) __maxnreg__((fwd_max_regs<C, PPT>())) raster_fwd_kernel(RasterArgs a) {
    pdl_begin();
    constexpr int NF = 4 + C;
    using QC = QuadChannels<C>;
    constexpr bool hm = HALF;
    static_assert(!HALF || PPT == 1, "half mode runs one pixel per thread");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_item;
    const int batch = hm ? 0 : a.batch;
    float4 *s_geo0 = reinterpret_cast<float4 *>(smem_raw);
    float4 *s_geo1 = s_geo0 + batch;
    float4 *s_geo2 = s_geo1 + batch;
    float *s_feat = reinterpret_cast<float *>(s_geo2 + batch);
    const int nthreads = hm ? 32 : a.tile_w * a.tile_h / PPT;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane & 3;
    int *s_q = reinterpret_cast<int *>(s_feat + (size_t)batch * NF) + (size_t)warp * fwd_warp_words<C, PPT, HALF>();
    uint32_t *s_qr = reinterpret_cast<uint32_t *>(s_q + kRing);  // (half mode)
    int *s_row = s_q + (hm ? 2 : 1) * kRing;
    float *s_A = reinterpret_cast<float *>(s_row + kChunk);
    float *s_hf = s_A + 32 * PPT * kAPitch;  // half mode: 2 x 16 feature rows
    const WarpTile<PPT> wt(a.tile_w);
    const float ln_amin = __logf(a.alpha_min);
    const float ax = (float)(wt.lx - (lane & 7) + 4 * (lane >> 4)), ay = (float)(wt.ly - (lane >> 3));
    const uint32_t lt = (1u << lane) - 1u;
    const int n_items = hm ? 2 * a.n_tiles : a.n_tiles;
    for (int iter = 0;; ++iter) {
        if (!a.persistent && iter > 0) break;
        const int slot = next_item(a, n_items, s_item);
        if (slot >= n_items) break;
        const int tslot = hm ? slot >> 1 : slot, hf = hm ? slot & 1 : 0;
        const int item = a.order ? a.order[tslot] : tslot;  // tile id
        TileInfo ti = tile_info(a, item);
        ti.py0 += hf * (a.tile_h / 2);  // half mode: this warp's half
        const sg_view &vw = *ti.vw;
        const int px = ti.px0 + wt.lx;
        const int2 range = a.ranges[item];
        const int n = range.y - range.x;
        const uint32_t rec_base = (uint32_t)ti.v * (uint32_t)a.N;
        float acc[PPT][4][QC::N];  // [k][x]: the lane's channels at the pixel of lane ^ x
        float T[PPT], Tl[PPT];  // transmittance; the same while the pixel is live, then -1
        int last[PPT], nc[PPT];
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int c = 0; c < QC::N; ++c) acc[k][x][c] = 0.f;
            T[k] = 1.f;
            last[k] = 0;
            nc[k] = 0;
            Tl[k] = px < vw.W && ti.py0 + wt.ly + 4 * k < vw.H ? 1.f : -1.f;
        }
        // The chunk whose alphas are in s_A: hits has a bit for each entry that contributes to
        // some pixel of the warp; entry e has its features at feat_of(e) and list position
        // pos_of(e).  The recurrence in T, then the feature sums.
        auto composite = [&](const uint32_t hits, auto feat_of, auto pos_of) {
            uint32_t hit[PPT];  // the entries that contribute to the pixel
#pragma unroll
            for (int k = 0; k < PPT; ++k) hit[k] = 0;
#pragma unroll 1
            for (int e0 = 0; e0 < kChunk; e0 += 4) {
                const uint32_t h4 = (hits >> e0) & 15u;
                if (!h4) continue;
                float tl = -1.f;
#pragma unroll
                for (int k = 0; k < PPT; ++k) tl = fmaxf(tl, Tl[k]);
                if (!__any_sync(SG_FULL_MASK, tl >= 0.f)) break;
                float al[PPT][4];
#pragma unroll
                for (int k = 0; k < PPT; ++k) {
                    const float4 t = *reinterpret_cast<const float4 *>(s_A + (32 * k + lane) * kAPitch + e0);
                    al[k][0] = t.x; al[k][1] = t.y; al[k][2] = t.z; al[k][3] = t.w;
                }
                uint32_t hb[PPT];
#pragma unroll
                for (int k = 0; k < PPT; ++k) hb[k] = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (!((h4 >> i) & 1u)) continue;  // (warp-uniform)
                    float f[QC::N];
                    QC::load(feat_of(e0 + i), sub, f);
#pragma unroll
                    for (int k = 0; k < PPT; ++k) {
                        const float A = al[k][i];
                        const float Tn = __fmul_rn(Tl[k], __fsub_rn(1.f, A));
                        const bool stop = Tn < a.T_min;  // (and again for a stopped pixel: Tl = -1)
                        const float w = stop ? 0.f : A * Tl[k];
                        if (!stop && A > 0.f) hb[k] |= 1u << i;
                        T[k] = stop ? T[k] : Tn;
                        Tl[k] = stop ? -1.f : Tn;
#pragma unroll
                        for (int x = 0; x < 4; ++x)
                            fma_if<QC::N>(acc[k][x], x ? __shfl_xor_sync(SG_FULL_MASK, w, x) : w, f);
                    }
                }
#pragma unroll
                for (int k = 0; k < PPT; ++k) hit[k] |= hb[k] << e0;
            }
#pragma unroll
            for (int k = 0; k < PPT; ++k) {
                nc[k] += __popc(hit[k]);
                if (hit[k]) last[k] = pos_of(31 - __clz(hit[k])) + 1;
            }
        };
        auto any_live = [&]() {
            bool r = false;
#pragma unroll
            for (int k = 0; k < PPT; ++k) r |= Tl[k] >= 0.f;
            return r;
        };
        if (!hm) {
            for (int b0 = 0; b0 < n; b0 += batch) {
                if (__syncthreads_count(!any_live()) == nthreads) break;
                const int cnt = min(batch, n - b0);
                load_batch<NF>(a, C, range.x, b0, cnt, ti.px0, ti.py0, rec_base, s_geo0, s_geo1, s_geo2, s_feat,
                               nullptr, nthreads);
                __syncthreads();
                // rows whose footprint can reach the warp's sub-tile (32 tested at once), queued
                // front to back and composited 16 at a time
                int top = 0, head = 0, qn = 0;
                while (__any_sync(SG_FULL_MASK, any_live())) {
                    while (qn < kChunk && top < cnt) {
                        const int j = top + lane;
                        const bool sel = j < cnt && !wt.misses(s_geo2[j], s_geo1[j], ln_amin);
                        const uint32_t bal = __ballot_sync(SG_FULL_MASK, sel);
                        if (sel) s_q[(head + qn + __popc(bal & lt)) & (kRing - 1)] = j;
                        qn += __popc(bal);
                        top += 32;
                    }
                    if (qn == 0) break;
                    __syncwarp();
                    const int c = min(kChunk, qn), e = lane & 15;
                    const int j = s_q[(head + min(e, c - 1)) & (kRing - 1)];
                    EntryGeo g = entry_geo(s_geo0[j], s_geo1[j]);
                    if (e >= c) g.o = 0.f;
                    if (lane < kChunk) s_row[lane] = j;
                    const uint32_t bal = __ballot_sync(
                        SG_FULL_MASK, chunk_alphas<PPT>(g, ax, ay, a.alpha_max, a.alpha_min, s_A));
                    __syncwarp();
                    composite((bal | (bal >> 16)) & 0xffffu, [&](int r) { return s_feat + (size_t)s_row[r] * NF; },
                              [&](int r) { return b0 + s_row[r]; });
                    __syncwarp();
                    head += c;
                    qn -= c;
                }
            }
        } else {
            // list positions whose half mask holds this half, ascending: (s_q, s_qr) is a ring
            // of (position, record), top the next position scanned, word its list word (loaded
            // one scan ahead)
            int top = 0, head = 0, qn = 0;
            uint32_t word = lane < n ? a.record[range.x + lane] : 0u;  // record | half mask << 30
            auto fill = [&]() {
                while (qn < kChunk && top < n) {
                    const uint32_t w = word;
                    const int pos = top + lane;
                    top += 32;
                    word = top + lane < n ? a.record[range.x + top + lane] : 0u;
                    const bool sel = (w >> (30 + hf)) & 1u;  // (0 past the list's end)
                    const uint32_t bal = __ballot_sync(SG_FULL_MASK, sel);
                    if (sel) {
                        const int q = (head + qn + __popc(bal & lt)) & (kRing - 1);
                        s_q[q] = pos;
                        s_qr[q] = w & 0x3fffffffu;
                    }
                    qn += __popc(bal);
                }
                __syncwarp();
            };
            // requests the next chunk of the ring: geometry of entry lane % 16 and its position
            // into registers, features into buffer buf
            float4 g0, g1;
            int pos = 0;
            auto request = [&](int buf) {
                fill();
                const int c = min(kChunk, qn), e = lane & 15;
                if (c > 0) {
                    const int q = (head + min(e, c - 1)) & (kRing - 1);
                    const uint32_t rec = s_qr[q];
                    pos = s_q[q];
                    g0 = a.geo[2 * (size_t)rec];
                    g1 = a.geo[2 * (size_t)rec + 1];
                    stage_features_async<NF>(a, rec, rec_base, s_hf + buf * kChunk * NF);
                }
                cp_async_commit_group();
                head += c;
                qn -= c;
                return c;
            };
            int buf = 0;
            int c = request(0);
            while (c > 0 && __any_sync(SG_FULL_MASK, any_live())) {
                const int e = lane & 15;
                float *feat = s_hf + buf * kChunk * NF;
                EntryGeo g = record_geo(g0, g1, ti.px0, ti.py0);
                if (e >= c) g.o = 0.f;
                if (lane < kChunk) {
                    s_row[lane] = pos;
                    feat[lane * NF + 3] = g0.z;  // depth (camera z of the mean, Eq. 8)
                }
                __syncwarp();
                c = request(buf ^ 1);
                const uint32_t bal = __ballot_sync(
                    SG_FULL_MASK, chunk_alphas<PPT>(g, ax, ay, a.alpha_max, a.alpha_min, s_A));
                cp_async_wait_groups<1>();
                __syncwarp();
                composite((bal | (bal >> 16)) & 0xffffu, [&](int r) { return feat + r * NF; },
                          [&](int r) { return s_row[r]; });
                __syncwarp();
                buf ^= 1;
            }
            cp_async_wait_groups<0>();
        }
        // the quad's pixels in order: v[j] is the pixel of lane (lane & ~3) + j
        const size_t HW = (size_t)vw.W * vw.H;
        const size_t p0 = (size_t)vw.pixel_offset;
        const int qx = px - sub;  // first pixel column of the quad
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
            const int py = ti.py0 + wt.ly + 4 * k;
            float Tq[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) Tq[j] = __shfl_sync(SG_FULL_MASK, T[k], (lane & ~3) | j);
            if (py >= vw.H) continue;
            const size_t p = (size_t)py * vw.W + qx;
#pragma unroll
            for (int i = 0; i < QC::N; ++i) {
                float v[4] = {acc[k][0][i], acc[k][1][i], acc[k][2][i], acc[k][3][i]};
                if (sub & 1) {
                    float t = v[0]; v[0] = v[1]; v[1] = t;
                    t = v[2]; v[2] = v[3]; v[3] = t;
                }
                if (sub & 2) {
                    float t = v[0]; v[0] = v[2]; v[2] = t;
                    t = v[1]; v[1] = v[3]; v[3] = t;
                }
                if (i == 0) {
                    if (sub < 3) {
                        const float bg = sub == 0 ? a.bg0 : sub == 1 ? a.bg1 : a.bg2;
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[j] = v[j] + Tq[j] * bg;
                    }
                    store_quad(sub < 3 ? a.img_rgb + 3 * p0 + sub * HW + p : a.img_depth + p0 + p, v, vw.W - qx);
                } else {
                    store_quad(a.img_sem + (size_t)C * p0 + QC::sem(i - 1, sub) * HW + p, v, vw.W - qx);
                }
            }
            if (px >= vw.W) continue;
            a.T_final[p0 + p + sub] = T[k];
            a.last[p0 + p + sub] = last[k];
            a.n_contrib[p0 + p + sub] = nc[k];
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------
// Backward helpers
// ---------------------------------------------------------------------------------------

// The backward works on chunks of 16 consecutive list entries.  Three of its sums are
// contractions over the warp's pixels and run on the tensor cores (mma.m16n8k8, TF32
// operands split as x = hi + lo, hi = x with its 13 low mantissa bits cleared, lo = x - hi
// exactly; hi*hi + hi*lo + lo*hi keeps about 22 mantissa bits of every product, i.e.
// FP32-level accuracy):
//   gf[p][r] = sum_f g[p][f] F[r][f]          (pixel gradient . Gaussian features)
//   dF[r][f] = sum_p w[p][r] g[p][f]          (colour / depth / semantic gradients)
//   M[r][m]  = sum_p s[p][r] P_m(X_p, Y_p)    (moments of s = dL/dsigma)
// with w = alpha T and P = (1, X, Y, X^2, XY, Y^2) the pixel offsets from the warp centre.
// The 2D-mean, conic and opacity gradients are linear in the moments (see moment_grads).
constexpr int kHalfQueue = kChunk + 32;  // entries pending (< 16 + one 32-entry scan)

constexpr int kChunkPitch = 32 + 4;  // 4 mod 32: conflict-free fragments

template <int NF>
__host__ __device__ constexpr int padded_features() { return (NF + 7) / 8 * 8; }

// Row pitch of the per-warp copy G of dL/dimage (a row per pixel).  It is read by ldmatrix (8
// rows of 16 bytes) and by words, lane (gid, tig) row tig and column gid of a tile.  Where the
// features padded to 8 are 8 mod 16 (C = 4, 16, 32) that is the pitch, with the 4-column groups of
// rows 4 .. 7 of every 8 swapped (g_swap): both reads are then free of bank conflicts (at the
// least odd multiple of 4 the word reads took two passes, 24 of some 330 shared-memory passes of
// a chunk; batched workload 2030 -> 2006 us, 1200x680 x 3 levels 276 -> 272).  Otherwise the least odd multiple of 4 that holds the features: padding to 8 mod 16
// would cost a CTA per SM.  Features NF .. padded_features - 1 are not stored: their fragment
// loads are predicated to zero.
template <int NF>
__host__ __device__ constexpr bool g_swapped() { return padded_features<NF>() % 16 == 8; }
template <int NF>
__host__ __device__ constexpr int g_pitch() {
    return g_swapped<NF>() ? padded_features<NF>() : (NF / 4) % 2 == 1 ? NF : NF + 4;
}
// what to exclusive-or a 4-column group's index with in G's row p
template <int NF>
__device__ __forceinline__ int g_swap(int p) { return g_swapped<NF>() ? (p >> 2) & 1 : 0; }

// The adjoint gives every thread one pixel, whatever the forward's number.  With two or four, the
// per-chunk costs are shared by more pixels, but half or a quarter of the warps are left, each
// with a longer serial recurrence, and shared memory holds fewer of them: at 16 x 16, 32 x 8,
// 16 x 8 and 8 x 8 tiles, C = 4 to 40 and 100 to 4270 tiles a whole iteration took 0 to 12 %
// longer with two (320x180 x 3 levels, C = 16: 293 against 261 us; 640x480 x 2 levels with 1M
// Gaussians, C = 40: 1647 against 1474) and up to 58 % with four.
//
// shared memory of one warp (4-byte words): the chunk's rows and the queue (with records in
// half mode), their list positions, G (32 x g_pitch), the first chunk buffer (16 x kChunkPitch)
// and the chunk's alphas; a multiple of 16 bytes.  The second chunk buffer reuses the alphas'
// (read into registers first): 20 instead of 17 one-warp CTAs per SM in half mode (batched
// workload 2072 -> 2009 us).
template <int C, bool HALF>
__host__ __device__ constexpr int bwd_warp_words() {
    static_assert(kChunk * kChunkPitch <= 32 * kAPitch, "the second chunk buffer reuses the alphas'");
    return 2 * kChunk + (HALF ? 2 : 1) * kHalfQueue + 32 * g_pitch<4 + C>() + kChunk * kChunkPitch + 32 * kAPitch;
}

// Gradients of the 2D mean (u, v), the conic (a, b, c) and the opacity from the moments
// M = (sum s, sum s X, sum s Y, sum s X^2, sum s XY, sum s Y^2) of s = dL/dsigma over the
// pixels (X, Y offsets from the warp centre; U, V the mean's offset from it, so that
// dx = X - U, dy = Y - V).  With sigma = p1^2 + p2^2, p1 = m00 dx, p2 = m10 dx + m11 dy:
//   dL/du = -2 ((m00^2 + m10^2) S_x + m10 m11 S_y),  dL/dv = -2 (m10 m11 S_x + m11^2 S_y),
//   dL/d(a, b, c) = (S_xx / 2, S_xy, S_yy / 2),       dL/do = -S_1 / o,
// S_x = sum s dx, S_xx = sum s dx^2, ...; the last because s = -dL/dalpha alpha and
// dalpha/do = alpha / o wherever s is non-zero (alpha not clamped).  `part` (0..2) picks
// the pair this lane writes.
__device__ __forceinline__ void moment_grads(const float (&M)[6], float U, float V, const float4 &g1, int part,
                                             float &r0, float &r1) {
    const float M0 = M[0], Mx = M[1], My = M[2], Mxx = M[3], Mxy = M[4], Myy = M[5];
    if (part == 0) {
        const float Sx = fmaf(-U, M0, Mx), Sy = fmaf(-V, M0, My);
        const float m00 = g1.x, m10 = g1.y, m11 = g1.z;
        r0 = -2.f * ((m00 * m00 + m10 * m10) * Sx + m10 * m11 * Sy);
        r1 = -2.f * (m10 * m11 * Sx + m11 * m11 * Sy);
    } else if (part == 1) {
        r0 = 0.5f * (Mxx - 2.f * U * Mx + U * U * M0);
        r1 = Mxy - V * Mx - U * My + U * V * M0;
    } else {
        r0 = 0.5f * (Myy - 2.f * V * My + V * V * M0);
        r1 = -M0 / g1.w;
    }
}

template <int C>
__host__ __device__ constexpr int bwd_max_regs() { return C <= 16 ? 96 : 128; }

template <int C, bool HALF>
__global__ void __maxnreg__((bwd_max_regs<C>())) raster_bwd_kernel(RasterArgs a) {
    pdl_begin();
    constexpr int NF = 4 + C;                     // rgb(3) depth | sem(C)
    constexpr int NFP = padded_features<NF>();    // features padded to 8
    constexpr int NT = NFP / 8;                   // 8-feature tiles
    constexpr int NPX = 32;                       // pixels of one warp (pixel = lane)
    constexpr int KS = NPX / 8;                   // 8-pixel steps
    constexpr int WQ = kChunkPitch;
    constexpr int GP = g_pitch<NF>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_item, s_max_last;
    // Half mode (8 x 8 tiles, half masks given): a CTA is one warp that
    // works on one half (8 x 4 pixels) of a tile at a time; it walks the tile's list back to
    // front, keeps the entries whose half mask holds its half in a queue, and stages and
    // processes them 16 at a time, so its chunks hold only its own entries; no block barrier.
    // Otherwise the CTA's warps share each batch of the list, staged between two block
    // barriers.
    constexpr bool hm = HALF;
    const int batch = hm ? kChunk : a.batch;
    float4 *s_geo0 = reinterpret_cast<float4 *>(smem_raw);
    float4 *s_geo1 = s_geo0 + batch;
    // (half mode stages no (u, v, ex, ey) rows: its entries passed the half's culling rule,
    // which rejects what the warp's ellipse test would)
    float4 *s_geo2 = hm ? nullptr : s_geo1 + batch;
    float *s_feat = reinterpret_cast<float *>(s_geo1 + (hm ? batch : 2 * batch));
    uint32_t *s_rec = reinterpret_cast<uint32_t *>(s_feat + (size_t)batch * NF);
    // per warp: the staged row of each chunk row (shared batches), its list position, and the
    // queue of pending entries: (list position, record), or staged rows
    const int nthreads = hm ? 32 : a.tile_w * a.tile_h;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int *s_pos = reinterpret_cast<int *>(s_rec + batch) + (size_t)warp * bwd_warp_words<C, HALF>();
    int *s_lp = s_pos + kChunk;  // list position of each chunk row (the largest int past its end)
    int *s_q = s_lp + kChunk;
    uint32_t *s_qr = reinterpret_cast<uint32_t *>(s_q + kHalfQueue);
    float *s_G = reinterpret_cast<float *>(s_qr + (hm ? kHalfQueue : 0));
    float *s_gw = s_G + NPX * GP;     // per chunk row: gf, then overwritten with w = alpha T
    float *s_A = s_gw + kChunk * WQ;  // alphas (chunk_alphas)
    float *s_sg = s_A;                // per chunk row: s = dL/dsigma
    const int gid = lane >> 2, tig = lane & 3;
    const WarpTile<1> wt(a.tile_w);
    const float ax = (float)(wt.lx - (lane & 7) + 4 * (lane >> 4)), ay = (float)(wt.ly - (lane >> 3));
    const float ln_amin = __logf(a.alpha_min);
    // moment polynomials at the B-fragment pixels: pixel 8 ks + tig (+ 4) has X = tig - 3.5
    // (tig + 0.5), Y = ks - 1.5; P_gid = P0 + Y (P1 + Y P2)
    // (all values small multiples of 1/4: exact in TF32, so B needs no split)
    const float X0 = tig - 3.5f, X1 = tig + 0.5f;
    const float P0a = gid == 0 ? 1.f : gid == 1 ? X0 : gid == 3 ? X0 * X0 : 0.f;
    const float P0b = gid == 0 ? 1.f : gid == 1 ? X1 : gid == 3 ? X1 * X1 : 0.f;
    const float P1a = gid == 2 ? 1.f : gid == 4 ? X0 : 0.f;
    const float P1b = gid == 2 ? 1.f : gid == 4 ? X1 : 0.f;
    const float P2 = gid == 5 ? 1.f : 0.f;
    // half mode: a work item is one half tile, or (half_pairs) a whole tile whose halves the
    // warp takes in turn, so that the second half's staging loads can hit L1
    const bool pairs = hm && a.half_pairs;
    const uint32_t lt = (1u << lane) - 1u;
    const int n_items = hm && !pairs ? 2 * a.n_tiles : a.n_tiles;
    for (int iter = 0;; ++iter) {
        if (!a.persistent && iter > 0) break;
        const int slot = next_item(a, n_items, s_item);
        if (slot >= n_items) break;
        const int tslot = hm && !pairs ? slot >> 1 : slot;
        const int item = a.order ? a.order[tslot] : tslot;  // tile id
        const int hf0 = hm && !pairs ? slot & 1 : 0, hf1 = pairs ? 2 : hf0 + 1;
        for (int hf = hf0; hf < hf1; ++hf) {
        TileInfo ti = tile_info(a, item);
        ti.py0 += hf * (a.tile_h / 2);  // half mode: this warp's half
        const sg_view &vw = *ti.vw;
        const int px = ti.px0 + wt.lx;
        const int2 range = a.ranges[item];
        const size_t HW = (size_t)vw.W * vw.H;
        const size_t p0 = (size_t)vw.pixel_offset;
        const uint32_t rec_base = (uint32_t)ti.v * (uint32_t)a.N;
        float T = 1.f, acc_a;
        int my_last = 0;
        {
            const int py = ti.py0 + wt.ly;
            const bool inside = px < vw.W && py < vw.H;
            const size_t p = (size_t)py * vw.W + px;
            float g[NFP];
#pragma unroll
            for (int f = 0; f < NFP; ++f) g[f] = 0.f;
            if (inside) {
                g[0] = a.dL_rgb[3 * p0 + p];
                g[1] = a.dL_rgb[3 * p0 + HW + p];
                g[2] = a.dL_rgb[3 * p0 + 2 * HW + p];
                g[3] = a.dL_depth[p0 + p];
#pragma unroll
                for (int c = 0; c < C; ++c) g[4 + c] = a.dL_sem[(size_t)C * p0 + c * HW + p];
                T = a.T_final[p0 + p];
                my_last = a.last[p0 + p];
            }
            acc_a = g[0] * a.bg0 + g[1] * a.bg1 + g[2] * a.bg2;
            float4 *row = reinterpret_cast<float4 *>(s_G + lane * GP);
#pragma unroll
            for (int f = 0; f < NF; f += 4) row[(f / 4) ^ g_swap<NF>(lane)] = make_float4(g[f], g[f + 1], g[f + 2], g[f + 3]);
        }
        const int warp_last = __reduce_max_sync(SG_FULL_MASK, my_last);
        __syncwarp();
        // One chunk of c <= 16 list entries, back to front: chunk row r (ascending list position)
        // is staged row row_of(r) at list position s_lp[r] (>= warp_last for r >= c), and lane l
        // holds the geometry g of row l % 16 (rows >= c: opacity 0).
        auto chunk = [&](const int c, const EntryGeo &g, auto row_of) {
                chunk_alphas<1>(g, ax, ay, a.alpha_max, a.alpha_min, s_A);
                // ---- gf = F G^T for the chunk (M = entries, N = pixels, K = features) ----
                // ldmatrix row addresses: lanes 0-15 rows 0-15 of the first four columns, lanes
                // 16-31 the same rows four columns further (A); lanes 8 m + i row i of matrix m (B)
                {
                    const float *fa = s_feat + (size_t)row_of(lane & 15) * NF + 4 * (lane >> 4);
                    const float *ga =
                        s_G + ((lane & 7) + 8 * (lane >> 4)) * GP + 4 * (((lane >> 3) & 1) ^ g_swap<NF>(lane & 7));
                    float d[KS][4];
#pragma unroll
                    for (int nt = 0; nt < KS; ++nt) d[nt][0] = d[nt][1] = d[nt][2] = d[nt][3] = 0.f;
#pragma unroll
                    for (int kk = 0; kk < NF / 8; ++kk) {
                        uint32_t ar[4], ah[4], al[4];
                        ldsm_x4(fa + 8 * kk, ar);
#pragma unroll
                        for (int i = 0; i < 4; ++i) split_tf32(__uint_as_float(ar[i]), ah[i], al[i]);
#pragma unroll
                        for (int n2 = 0; n2 < KS / 2; ++n2) {
                            uint32_t br[4], bh[4], bl[4];
                            ldsm_x4(ga + 16 * n2 * GP + 8 * kk, br);
#pragma unroll
                            for (int i = 0; i < 4; ++i) split_tf32(__uint_as_float(br[i]), bh[i], bl[i]);
                            mma_tf32x3(d[2 * n2], ah, al, bh[0], bh[1], bl[0], bl[1]);
                            mma_tf32x3(d[2 * n2 + 1], ah, al, bh[2], bh[3], bl[2], bl[3]);
                        }
                    }
                    if constexpr (NF % 8 != 0) {
                        // the last four features: K = 4 products
                        const float *f4 = s_feat + (size_t)row_of(lane & 15) * NF + 8 * (NF / 8);
                        uint32_t ar[2], ah[2], al[2];
                        ldsm_x2(f4, ar[0], ar[1]);
#pragma unroll
                        for (int i = 0; i < 2; ++i) split_tf32(__uint_as_float(ar[i]), ah[i], al[i]);
#pragma unroll
                        for (int n4 = 0; n4 < KS / 4; ++n4) {
                            uint32_t br[4];
                            ldsm_x4(s_G + (32 * n4 + lane) * GP + 8 * (NF / 8) + 4 * g_swap<NF>(lane), br);
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                uint32_t bh, bl;
                                split_tf32(__uint_as_float(br[i]), bh, bl);
                                mma_tf32x3_k4(d[4 * n4 + i], ah, al, bh, bl);
                            }
                        }
                    }
                    // D (16 x 8): d0, d1 (gid, 2 tig + 0 / 1), d2, d3 (gid + 8, ..)
#pragma unroll
                    for (int nt = 0; nt < KS; ++nt) {
                        *reinterpret_cast<float2 *>(s_gw + gid * WQ + 8 * nt + 2 * tig) = make_float2(d[nt][0], d[nt][1]);
                        *reinterpret_cast<float2 *>(s_gw + (gid + 8) * WQ + 8 * nt + 2 * tig) =
                            make_float2(d[nt][2], d[nt][3]);
                    }
                }
                __syncwarp();
                // ---- back to front: the recurrence in T and a ----
                uint32_t hits = 0;  // rows that contribute to the lane's pixel
                float4 al[kChunk / 4];
#pragma unroll
                for (int q = 0; q < kChunk / 4; ++q)
                    al[q] = *reinterpret_cast<const float4 *>(s_A + lane * kAPitch + 4 * q);
                __syncwarp();  // (s_sg reuses s_A)
#pragma unroll
                for (int q = kChunk / 4 - 1; q >= 0; --q) {  // rows 4 q .. 4 q + 3
                    if (4 * q >= c) continue;  // (warp-uniform)
                    const int4 lp = *reinterpret_cast<const int4 *>(s_lp + 4 * q);
                    const int pos[4] = {lp.x, lp.y, lp.z, lp.w};
                    const float a4[4] = {al[q].x, al[q].y, al[q].z, al[q].w};
                    uint32_t hb = 0;
#pragma unroll
                    for (int i = 3; i >= 0; --i) {
                        float *gw = s_gw + (4 * q + i) * WQ + lane;
                        const float A = pos[i] < my_last ? a4[i] : 0.f, om = 1.f - A;
                        // (a pixel without a contribution keeps T and a: A = 0, gf taken as 0;
                        // w and s are 0 there even if T or a is not finite, which would reach every
                        // row's sums over the warp's pixels)
                        const bool on = A > 0.f;
                        const float gf = on ? *gw : 0.f;
                        if (on) hb |= 1u << i;
                        // transmittance before this Gaussian (only gradients depend on it)
                        T *= rcp_fast(om);
                        const float dalpha = T * (gf - acc_a);
                        acc_a = fmaf(om, acc_a, A * gf);
                        *gw = on ? A * T : 0.f;
                        // (alpha = alpha_max: clamped, no gradient; else alpha = o G)
                        s_sg[(4 * q + i) * WQ + lane] = on && A < a.alpha_max ? -dalpha * A : 0.f;
                    }
                    hits |= hb << (4 * q);
                }
                const uint32_t mask = __reduce_or_sync(SG_FULL_MASK, hits);
                __syncwarp();
                if (!mask) return;  // (warp-uniform)
                // ---- dF = W G (M = entries, N = features, K = pixels), moments M = S P ----
                // (rows without a contribution may hold stale values: they are not written out)
                const bool keep0 = (mask >> gid) & 1u, keep1 = (mask >> (gid + 8)) & 1u;
                const float *wa = s_gw + (lane & 15) * WQ + 4 * (lane >> 4);
                const float *sa = s_sg + (lane & 15) * WQ + 4 * (lane >> 4);
                float df[NT][4], mom[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) df[nt][0] = df[nt][1] = df[nt][2] = df[nt][3] = 0.f;
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) {
                    uint32_t ar[4], ah[4], al[4];
                    ldsm_x4(wa + 8 * ks, ar);
#pragma unroll
                    for (int i = 0; i < 4; ++i) split_tf32(__uint_as_float(ar[i]), ah[i], al[i]);
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        // B (8 x 8): b0 (tig, gid), b1 (tig + 4, gid) = G[pixel][feature]
                        const float *gp = s_G + (8 * ks + tig) * GP + 8 * nt;
                        const bool stored = 8 * nt + 8 <= NF || 8 * nt + gid < NF;
                        uint32_t bh0, bl0, bh1, bl1;
                        split_tf32(stored ? gp[gid] : 0.f, bh0, bl0);
                        split_tf32(stored ? gp[4 * GP + (gid ^ (g_swapped<NF>() ? 4 : 0))] : 0.f, bh1, bl1);
                        mma_tf32x3(df[nt], ah, al, bh0, bh1, bl0, bl1);
                    }
                    ldsm_x4(sa + 8 * ks, ar);
#pragma unroll
                    for (int i = 0; i < 4; ++i) split_tf32(__uint_as_float(ar[i]), ah[i], al[i]);
                    const float Y = (float)ks - 1.5f;
                    const uint32_t pb0 = __float_as_uint(fmaf(Y, fmaf(Y, P2, P1a), P0a));
                    const uint32_t pb1 = __float_as_uint(fmaf(Y, fmaf(Y, P2, P1b), P0b));
                    mma_tf32(mom, al, pb0, pb1);
                    mma_tf32(mom, ah, pb0, pb1);
                }
                // feature gradients: D rows gid, gid + 8 (entries), columns 2 tig, 2 tig + 1 (features)
#pragma unroll
                for (int hr = 0; hr < 2; ++hr) {
                    if (!(hr ? keep1 : keep0)) continue;
                    const uint32_t rec = s_rec[row_of(gid + 8 * hr)];
                    const uint32_t gi = rec - rec_base;
                    float *gs = a.g_sem + (size_t)C * (a.sem_rec ? rec : gi);
                    // features 0-7: colour and depth in lanes 0, 1 of the quad, semantics in 2, 3
                    float *p0 = a.g_col + (size_t)a.col_stride * (a.col_rec ? rec : gi) + 2 * tig;
                    float *p1 = tig == 1 ? a.g2d + 8 * (size_t)rec + 6 : p0 + 1;
                    if (tig >= 2) {
                        p0 = gs + 2 * tig - 4;
                        p1 = p0 + 1;
                    }
                    atomicAdd(p0, df[0][2 * hr]);
                    atomicAdd(p1, df[0][2 * hr + 1]);
#pragma unroll
                    for (int nt = 1; nt < NT; ++nt) {
                        // features 2 tig, 2 tig + 1 of this n-tile: one 8-byte vector reduction when
                        // the buffer allows it
                        const int f0 = 8 * nt + 2 * tig;
                        if (f0 >= NF) continue;
                        if (a.sem_v2) {
                            red_add_v2(gs + (f0 - 4), df[nt][2 * hr], df[nt][2 * hr + 1]);
                        } else {
                            atomicAdd(gs + (f0 - 4), df[nt][2 * hr]);
                            atomicAdd(gs + (f0 - 3), df[nt][2 * hr + 1]);
                        }
                    }
                }
                // geometric gradients: lane tig of a quad holds moments (2 tig, 2 tig + 1) of its rows
                float Mr[2][6];
#pragma unroll
                for (int t = 0; t < 3; ++t) {
                    const int src = (lane & ~3) | t;
                    Mr[0][2 * t] = __shfl_sync(SG_FULL_MASK, mom[0], src);
                    Mr[0][2 * t + 1] = __shfl_sync(SG_FULL_MASK, mom[1], src);
                    Mr[1][2 * t] = __shfl_sync(SG_FULL_MASK, mom[2], src);
                    Mr[1][2 * t + 1] = __shfl_sync(SG_FULL_MASK, mom[3], src);
                }
                if (tig < 3) {
#pragma unroll
                    for (int hr = 0; hr < 2; ++hr) {
                        if (!(hr ? keep1 : keep0)) continue;
                        const int j = row_of(gid + 8 * hr);
                        const float4 g0 = s_geo0[j];
                        const float4 g1 = s_geo1[j];
                        const float U = (g0.x - wt.cxw) + g0.z, V = (g0.y - wt.cyw) + g0.w;
                        float r0, r1;
                        moment_grads(Mr[hr], U, V, g1, tig, r0, r1);
                        // (records are 32 bytes of the 16-byte aligned workspace)
                        red_add_v2(a.g2d + 8 * (size_t)s_rec[j] + 2 * tig, r0, r1);
                    }
                }
                __syncwarp();  // the chunk buffers are rewritten next
        };
        if (!hm) {
            if (threadIdx.x == 0) s_max_last = 0;
            __syncthreads();
            if (lane == 0 && warp_last > 0) atomicMax(&s_max_last, warp_last);
            __syncthreads();
            const int max_last = s_max_last;
            const int n_batches = (max_last + batch - 1) / batch;
            for (int b = n_batches - 1; b >= 0; --b) {
                const int b0 = b * batch;
                const int cnt = min(batch, max_last - b0);
                __syncthreads();
                load_batch<NF>(a, C, range.x, b0, cnt, ti.px0, ti.py0, rec_base, s_geo0, s_geo1, s_geo2, s_feat,
                               s_rec, nthreads);
                __syncthreads();
                // rows of the batch whose footprint reaches the warp's pixels, back to front: (the
                // exact ellipse test, 32 rows at a time), processed 16 at a time
                const int jmax = min(cnt, warp_last - b0);  // warp-uniform
                int qn = 0;
                for (int top = jmax; top > 0 || qn > 0;) {
                    while (qn < kChunk && top > 0) {
                        const int j = top - 1 - lane;
                        const bool sel = j >= 0 && !wt.misses(s_geo2[j], s_geo1[j], ln_amin);
                        const uint32_t bal = __ballot_sync(SG_FULL_MASK, sel);
                        if (sel) s_q[qn + __popc(bal & lt)] = j;
                        qn += __popc(bal);
                        top -= 32;
                    }
                    if (qn == 0) break;
                    __syncwarp();
                    const int c = min(kChunk, qn);
                    // chunk row r is queue entry c - 1 - r; rows past c stay out of reach
                    if (lane < kChunk) {
                        s_pos[lane] = lane < c ? s_q[c - 1 - lane] : 0;
                        s_lp[lane] = lane < c ? b0 + s_q[c - 1 - lane] : 0x7fffffff;
                    }
                    const int rest = qn - c;  // (< 32)
                    const int keep = lane < rest ? s_q[c + lane] : 0;
                    __syncwarp();
                    if (lane < rest) s_q[lane] = keep;
                    qn = rest;
                    const int j = s_pos[lane & 15];
                    EntryGeo g = entry_geo(s_geo0[j], s_geo1[j]);
                    if ((lane & 15) >= c) g.o = 0.f;
                    chunk(c, g, [s_pos](int r) { return s_pos[r]; });
                }
            }
            __syncthreads();
        } else {
            // list positions < warp_last whose half mask holds this half, in descending order:
            // (s_q, s_qr)[0 .. qn) is the queue of (position, record), top the next position
            // scanned (exclusive)
            int top = warp_last, qn = 0;
            for (;;) {
                while (qn < kChunk && top > 0) {
                    const int pos = top - 1 - lane;
                    uint32_t rec = 0u;
                    bool sel = false;
                    if (pos >= 0) {
                        const uint32_t word = a.record[range.x + pos];  // record | half mask << 30
                        rec = word & 0x3fffffffu;
                        sel = (word >> (30 + hf)) & 1u;
                    }
                    const uint32_t bal = __ballot_sync(SG_FULL_MASK, sel);
                    if (sel) {
                        s_q[qn + __popc(bal & lt)] = pos;
                        s_qr[qn + __popc(bal & lt)] = rec;
                    }
                    qn += __popc(bal);
                    top = max(top - 32, 0);
                    __syncwarp();
                }
                if (qn == 0) break;
                const int c = min(kChunk, qn);
                // rows 0 .. c-1 in ascending list position: row r is queue entry c - 1 - r; lane l
                // loads the geometry of row l % 16 (lanes 0-15 also stage it)
                const int q = max(c - 1 - (lane & 15), 0);
                const uint32_t rec = s_qr[q];
                const float4 r0 = a.geo[2 * (size_t)rec], r1 = a.geo[2 * (size_t)rec + 1];
                stage_features_async<NF>(a, rec, rec_base, s_feat);
                cp_async_commit_group();
                EntryGeo g = record_geo(r0, r1, ti.px0, ti.py0);
                if ((lane & 15) >= c) g.o = 0.f;
                if (lane < kChunk) {
                    s_geo0[lane] = make_float4(g.ui, g.vi, g.uf, g.vf);
                    s_geo1[lane] = make_float4(g.m00, g.m10, g.m11, g.o);
                    s_rec[lane] = rec;
                    s_feat[lane * NF + 3] = r0.z;  // depth (camera z of the mean, Eq. 8)
                    s_lp[lane] = lane < c ? s_q[q] : 0x7fffffff;
                }
                const int rest = qn - c;  // (< 32)
                const int keep = lane < rest ? s_q[c + lane] : 0;
                const uint32_t keep_rec = lane < rest ? s_qr[c + lane] : 0u;
                __syncwarp();
                if (lane < rest) {
                    s_q[lane] = keep;
                    s_qr[lane] = keep_rec;
                }
                qn = rest;
                cp_async_wait_groups<0>();
                __syncwarp();
                chunk(c, g, [](int r) { return r; });
            }
            __syncwarp();
        }
        }
    }
}

// ---------------------------------------------------------------------------------------

template <int C>
inline size_t batch_smem(int batch) {
    return (size_t)batch * (3 * 16 + 4 * (4 + C));
}
template <int C, int PPT>
inline size_t fwd_smem(int batch, int threads) {
    return batch_smem<C>(batch) + sizeof(float) * (threads / 32) * fwd_warp_words<C, PPT, false>();
}
template <int C>
inline size_t fwd_half_smem() {
    return sizeof(float) * fwd_warp_words<C, 1, true>();
}
template <int C>
inline size_t bwd_smem(int batch, int threads) {
    return batch_smem<C>(batch) + (size_t)batch * 4 + sizeof(float) * (threads / 32) * bwd_warp_words<C, false>();
}
// half mode: one 16-entry chunk staged without its (u, v, ex, ey) rows, one warp
template <int C>
inline size_t bwd_half_smem() {
    return batch_smem<C>(kChunk) - (size_t)kChunk * 16 + (size_t)kChunk * 4 + sizeof(float) * bwd_warp_words<C, true>();
}

inline int resident_grid(const void *fn, int threads, size_t smem) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
    if (per_sm < 1) per_sm = 1;
    return sms * per_sm;
}

// One launch of kernel fn (one of the instantiations below).  configured: the dynamic shared
// memory that fn has been opted in to.
inline sg_status launch_raster_fn(void (*fn)(RasterArgs), RasterArgs &a, bool half, bool backward, int threads, size_t smem,
                                  size_t &configured, cudaStream_t st) {
    // opt in to the dynamic size whenever it grows: at 48 KB and just below, the kernel's
    // static shared variables alone take the total past the default limit
    if (configured < smem) {
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            return check_launch("raster smem attribute");
        configured = smem;
    }
    // the half-tile adjoint takes whole tiles as work items when there are at least 16 tiles
    // per resident CTA (measured: batched workload, 29 per CTA, -1.4 %); with fewer, twice as
    // long items leave the persistent grid's tail unbalanced
    const int resident = a.persistent ? resident_grid((const void *)fn, threads, smem) : 0;
    a.half_pairs = backward && half && a.persistent && (int64_t)a.n_tiles >= 16 * (int64_t)resident;
    const int n_items = half && !a.half_pairs ? 2 * a.n_tiles : a.n_tiles;
    int grid = n_items;
    if (a.persistent) {
        grid = resident;
        if (grid > n_items) grid = n_items;
    }
    if (grid <= 0) return SG_OK;
    launch_pdl(fn, grid, threads, smem, st, a);
    count_launches(1);
    return check_launch(backward ? "raster_bwd" : "raster_fwd");
}

// Lists with half masks (8 x 8 tiles): the adjoint runs one warp per half tile, and so does the
// forward at one pixel per thread when the config asks for it.
template <int C, int PPT>
sg_status launch_raster_fwd(RasterArgs &a, cudaStream_t st) {
    static size_t configured[2] = {0, 0};
    const bool half = a.half && PPT == 1 && a.tile_w == 8 && a.tile_h == 8 && a.half_fwd;
    const int threads = half ? 32 : a.tile_w * a.tile_h / PPT;
    return half ? launch_raster_fn(raster_fwd_kernel<C, PPT, PPT == 1>, a, true, false, threads, fwd_half_smem<C>(),
                                   configured[1], st)
                : launch_raster_fn(raster_fwd_kernel<C, PPT>, a, false, false, threads, fwd_smem<C, PPT>(a.batch, threads),
                                   configured[0], st);
}

template <int C>
sg_status launch_raster_bwd(RasterArgs &a, cudaStream_t st) {
    static size_t configured[2] = {0, 0};
    const bool half = a.half && a.tile_w == 8 && a.tile_h == 8;
    const int threads = half ? 32 : a.tile_w * a.tile_h;
    return half ? launch_raster_fn(raster_bwd_kernel<C, true>, a, true, true, threads, bwd_half_smem<C>(), configured[1], st)
                : launch_raster_fn(raster_bwd_kernel<C, false>, a, false, true, threads, bwd_smem<C>(a.batch, threads),
                                   configured[0], st);
}

template <int C>
sg_status launch_raster_c(RasterArgs &a, bool backward, cudaStream_t st) {
    if (backward) return launch_raster_bwd<C>(a, st);
    switch (a.ppt) {
        case 1: return launch_raster_fwd<C, 1>(a, st);
        case 2: return launch_raster_fwd<C, 2>(a, st);
        default: return launch_raster_fwd<C, 4>(a, st);
    }
}

}  // namespace sg
