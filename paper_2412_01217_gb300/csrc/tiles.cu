// tiles.cu -- per-tile depth-sorted instance lists (the sorted set N of Eq. 7-9).
//
// Pipeline (all counts stay on the device, so the whole sequence can be captured in a
// CUDA graph with a fixed launch shape):
//   1. compact:  visible records r (non-empty tile rectangle) -> (depth bits, r), in r order,
//                and the digit histograms of the depth keys
//   2. sort:     stable LSD radix sort by the 32 float32 depth bits (depths are > z_near > 0
//                so their bit patterns order like the values); ties keep record order
//   3. emit:     the slots are the tile rows of each record's rectangle, record after
//                record in depth order (a prefix of the row counts numbers them); for each
//                slot the span of the record's alpha >= alpha_min region within the row (a
//                float32 computation) gives the contiguous run of tiles it reaches, and the
//                kept tiles are written as (global tile id, r), row-major, with the digit
//                histograms of the tile ids
//   4. sort:     stable LSD radix sort of the instances by global tile id (only the bits
//                n_tiles needs), which keeps the (depth, record) order inside each tile
//   5. ranges:   [start, end) of every tile
//   6. order:    (when requested) the tile ids by descending half-octave bucket of their list
//                length, one stable counting pass: the compositing kernels' work order
// The result equals sorting all kept instances by (tile, depth bits, record id).
//
// Every step that needs a prefix over the whole input (compaction, slot numbering, emission,
// each radix pass, the work order) is one kernel with a chained scan: a block draws its part's
// number from a counter, publishes the part's aggregate, sums its predecessors' published
// words back to the nearest one that already holds an inclusive prefix, and publishes its own.
// Parts are drawn in order, so the predecessors of a part are held by blocks that already run;
// every wait is bounded all the same (SG_STATUS_TIMEOUT), and a step whose predecessor gave up
// takes its input as empty: what the failed step left behind (places never written) is not read,
// and the lists come out empty.  The steps were three kernels each before (count, scan of the
// counts, apply): 33 launches per list build, now 10 to 12 (by the width of the tile ids) and one
// memset, and the keys and footprints are read once instead of twice.  What that gives is the
// launches and their latencies (320x180 x 3 levels with 30k Gaussians: 110 -> 70 us of kernels
// and 21 launch gaps); on the batched workload (2.1M visible records, 19M instances) the kernels
// take the same time as before (1.0 ms).
#include <cstdio>

#include <algorithm>

#include "sg_common.cuh"

namespace sg {

constexpr int kScanThreads = 256;
// Widest digit of the tile sort.  Each pass scatters a part's instances over 2^digit runs
// of the output; with 9-bit digits (512 runs per part) the partly written output lines no
// longer stay in L2 and the pass reads and writes twice its bytes in DRAM (measured), so 17 or
// 18 bits of tile id sort in three passes of 6 bits rather than two of 9 and 8.
constexpr int kTileDigitBits = 8;

// Exclusive block scan of one value per thread (blockDim == NT).
template <int NT = kScanThreads>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t &total) {
    __shared__ uint32_t s_warp[NT / 32 + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(SG_FULL_MASK, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int nw = NT / 32;
        uint32_t w = lane < nw ? s_warp[lane] : 0u;
        uint32_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(SG_FULL_MASK, wi, o);
            if (lane >= o) wi += t;
        }
        if (lane < nw) s_warp[lane] = wi - w;
        if (lane == nw - 1) s_warp[nw] = wi;
    }
    __syncthreads();
    const uint32_t res = incl - v + s_warp[warp];
    total = s_warp[NT / 32];
    __syncthreads();
    return res;
}

// ---------------------------------------------------------------------------------------
// Chained scan over parts.  A part's word is 0 until published, then flag | value.
// ---------------------------------------------------------------------------------------

constexpr uint64_t kAggregate = 1ull << 32;  // value: the part's own sum
constexpr uint64_t kPrefix = 1ull << 33;     // value: inclusive prefix through the part
constexpr uint32_t kSpinLimit = 1u << 22;

// A step's bounded waits.  polls: limit of each; before, own: flags of the step before (null for
// the first) and of this one, set once a wait has given up.  withhold (self-test): part 0
// publishes nothing, so that every wait for it runs out.
struct StepWaits {
    uint32_t *status;
    const int *before;
    int *own;
    uint32_t polls;
    int withhold;
    __device__ __forceinline__ void gave_up() const {
        atomicOr(status, SG_STATUS_TIMEOUT);
        *own = 1;
    }
    // n, or 0 if an earlier step gave up (uniform over the grid: their kernels are done; the flag
    // and n, which the caller has read, are in flight together).
    __device__ __forceinline__ int input(int n) const {
        if (!before || !*before) return n;
        *own = 1;
        return 0;
    }
};

__device__ __forceinline__ uint64_t load_word(const uint64_t *p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];\n" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void store_word(uint64_t *p, uint64_t v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;\n" ::"l"(p), "l"(v) : "memory");
}

// The word of an earlier part, once published; on a timeout an empty prefix.
__device__ __forceinline__ uint64_t wait_word(const uint64_t *p, uint64_t w, const StepWaits &sw) {
    for (uint32_t polls = 0; !(w >> 32); ++polls) {
        if (polls >= sw.polls) {
            sw.gave_up();
            return kPrefix;
        }
        w = load_word(p);
    }
    return w;
}

// Exclusive prefix of the part whose sum is `own`, for a whole block (every thread gets it);
// publishes the part's words.  256 predecessors are examined at a time: with several hundred
// parts in flight most of them hold only their own sum yet.
__device__ __forceinline__ uint32_t block_look_back(uint64_t *words, int part, uint32_t own, const StepWaits &sw) {
    __shared__ uint32_t s_sum[kScanThreads / 32];
    __shared__ bool s_has[kScanThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0 && !(sw.withhold && part == 0)) store_word(words + part, (part == 0 ? kPrefix : kAggregate) | own);
    uint32_t sum = 0;
    bool found = part == 0;
    for (int p = part - 1; !found; p -= kScanThreads) {  // (block-uniform)
        const int q = p - (int)threadIdx.x;
        uint64_t w = kPrefix;  // before the first part: an empty prefix
        if (q >= 0) w = wait_word(words + q, load_word(words + q), sw);
        const uint32_t pre = __ballot_sync(SG_FULL_MASK, (w & kPrefix) != 0);
        // lanes past the nearest prefix do not count
        const int stop = pre ? __ffs(pre) - 1 : 31;
        const uint32_t ws = __reduce_add_sync(SG_FULL_MASK, lane <= stop ? (uint32_t)w : 0u);
        if (lane == 0) {
            s_sum[warp] = ws;
            s_has[warp] = pre != 0;
        }
        __syncthreads();
        for (int i = 0; i < kScanThreads / 32 && !found; ++i) {
            sum += s_sum[i];
            found = s_has[i];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0 && part > 0) store_word(words + part, kPrefix | (uint64_t)(sum + own));
    return sum;
}

// The same for the threads of a warp, each with its own words (digits of a radix pass): a
// thread's sum has been published in words[part * stride]; four predecessors' words are
// requested at a time.  Called by whole warps, and the warp stays together: the waits and the
// loop end for all lanes at once (inactive lanes sum nothing), so that no lane runs ahead to the
// caller's block barrier while others still look back.  late: set when a wait gave up (for all
// lanes of the warp).
__device__ __forceinline__ uint32_t look_back(const uint64_t *words, int stride, int part, bool active,
                                              const StepWaits &sw, bool &late) {
    uint32_t sum = 0;
    bool done = !active;
    for (int p = part - 1; p >= 0 && !__all_sync(SG_FULL_MASK, done); p -= 4) {
        uint64_t w[4];  // (before the first part: an empty prefix)
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = !done && p - i >= 0 ? load_word(words + (size_t)(p - i) * stride) : kPrefix;
        for (uint32_t polls = 0;; ++polls) {
            bool missing = false;
#pragma unroll
            for (int i = 0; i < 4; ++i) missing |= !(w[i] >> 32);
            if (!__any_sync(SG_FULL_MASK, missing)) break;
            if (polls >= sw.polls) {  // (warp-uniform)
                if (missing) sw.gave_up();
                late = true;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (!(w[i] >> 32)) w[i] = kPrefix;
                break;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (!(w[i] >> 32)) w[i] = load_word(words + (size_t)(p - i) * stride);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (!done) {
                sum += (uint32_t)w[i];
                done = (w[i] & kPrefix) != 0;
            }
    }
    __syncwarp();
    return sum;
}

// The next part of a kernel's input (block-uniform).
__device__ __forceinline__ int next_part(int *counter) {
    __shared__ int s_part;
    __syncthreads();
    if (threadIdx.x == 0) s_part = atomicAdd(counter, 1);
    __syncthreads();
    return s_part;
}

// Adds a block's digit counts in shared memory (n words) to the global histogram.
__device__ __forceinline__ void flush_hist(const uint32_t *s_h, int n, uint32_t *hist) {
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kScanThreads)
        if (s_h[i]) atomicAdd(hist + i, s_h[i]);
}

__device__ __forceinline__ uint32_t rect_tiles(uint2 r) {
    const uint32_t tx0 = r.x & 0xffffu, ty0 = r.x >> 16, tx1 = r.y & 0xffffu, ty1 = r.y >> 16;
    return (tx1 > tx0 && ty1 > ty0) ? (tx1 - tx0) * (ty1 - ty0) : 0u;
}

__device__ __forceinline__ uint32_t rect_rows(uint2 r) {
    const uint32_t ty0 = r.x >> 16, ty1 = r.y >> 16;
    return rect_tiles(r) ? ty1 - ty0 : 0u;
}

// Compaction: (depth bits, record) of every visible record, in record order, and the four
// 8-bit digit histograms of the depth bits.  Each thread takes 8 consecutive records (two
// 16-byte loads of their rectangles when the array is 16-byte aligned), so a part is 2048
// records with one block scan and all of its loads in flight together.
constexpr int kCompactPerThread = 8;
constexpr int kCompactPart = kScanThreads * kCompactPerThread;
__global__ void __launch_bounds__(kScanThreads) compact_kernel(const uint2 *__restrict__ rect,
                                                               const float4 *__restrict__ geo, int n,
                                                               uint64_t *__restrict__ words, int *__restrict__ counter,
                                                               uint32_t *__restrict__ key, uint32_t *__restrict__ val,
                                                               int *__restrict__ total, uint32_t *__restrict__ hist,
                                                               int *__restrict__ instances, StepWaits sw) {
    pdl_begin();
    constexpr int E = kCompactPerThread;
    __shared__ uint32_t s_h[4 * 256];
    __shared__ uint32_t s_key[kCompactPart], s_val[kCompactPart];
    // (written by the last part of the emission, which has none without slots)
    if (blockIdx.x == 0 && threadIdx.x == 0) *instances = 0;
    for (int i = threadIdx.x; i < 4 * 256; i += kScanThreads) s_h[i] = 0;
    const bool vec = (reinterpret_cast<uintptr_t>(rect) & 15u) == 0;
    const int parts = (n + kCompactPart - 1) / kCompactPart;
    for (int part; (part = next_part(counter)) < parts;) {
        const int i0 = part * kCompactPart + (int)threadIdx.x * E;
        uint2 r[E];
        if (vec && i0 + E <= n) {
            const uint4 *p4 = reinterpret_cast<const uint4 *>(rect + i0);
#pragma unroll
            for (int q = 0; q < E / 2; ++q) {
                const uint4 w = p4[q];
                r[2 * q] = make_uint2(w.x, w.y);
                r[2 * q + 1] = make_uint2(w.z, w.w);
            }
        } else {
#pragma unroll
            for (int q = 0; q < E; ++q) r[q] = i0 + q < n ? rect[i0 + q] : make_uint2(0, 0);
        }
        uint32_t f = 0, bits = 0;
#pragma unroll
        for (int q = 0; q < E; ++q)
            if (r[q].x != r[q].y) {
                bits |= 1u << q;
                ++f;
            }
        uint32_t dep[E];
#pragma unroll
        for (int q = 0; q < E; ++q)
            dep[q] = ((bits >> q) & 1u) ? __float_as_uint(geo[2 * (size_t)(i0 + q)].z) : 0u;
        uint32_t tot;
        uint32_t o = block_exclusive_scan(f, tot);
#pragma unroll
        for (int q = 0; q < E; ++q)
            if ((bits >> q) & 1u) {
                s_key[o] = dep[q];
                s_val[o] = (uint32_t)(i0 + q);
                ++o;
            }
        const uint32_t off = block_look_back(words, part, tot, sw);
        if (part == parts - 1 && threadIdx.x == 0) *total = (int)(off + tot);
        __syncthreads();
        for (uint32_t j = threadIdx.x; j < ((tot + 31) & ~31u); j += kScanThreads) {
            const bool in = j < tot;
            const uint32_t d = in ? s_key[j] : 0u;
            if (in) {
                key[off + j] = d;
                val[off + j] = s_val[j];
#pragma unroll
                for (int q = 0; q < 3; ++q) atomicAdd(&s_h[256 * q + ((d >> (8 * q)) & 255u)], 1u);
            }
            // the top digit (sign and exponent) takes a handful of values: one add per value and warp
            const uint32_t top = in ? d >> 24 : 256u;
            const uint32_t peers = __match_any_sync(SG_FULL_MASK, top);
            if (in && (threadIdx.x & 31) == (uint32_t)(__ffs(peers) - 1))
                atomicAdd(&s_h[256 * 3 + top], (uint32_t)__popc(peers));
        }
        // (next_part's barriers order these reads before the next part's writes)
    }
    flush_hist(s_h, 4 * 256, hist);
}

// The columns of a tile row that the record's alpha >= alpha_min region reaches.  The
// projection wrote the half extent ex = sqrt(2 thr s00) 1.002 + 0.01 with
// thr = ln(o / alpha_min) + 1e-3 and m00 = 1 / sqrt(2 s00), so
// thr' = ((ex - 0.01) (1 / 1.002) m00)^2 recovers the threshold from the record (to float
// rounding, far inside its 1e-3 margin).  Within the band dy in [y0, y1] of the row's pixel
// centres, the ellipse sigma = (m00 dx)^2 + (m10 dx + m11 dy)^2 <= thr' spans dx in
// [xl, xr]: with A = m00^2 + m10^2, B = m10 m11, C = m11^2 and p = m00 m11 (A C - B^2 = p^2),
// the band is cut to |dy| <= sqrt(A thr') / p, the right edge (s - B dy) / A with
// s = sqrt(A thr' - (p dy)^2) is largest at dy = -B (sqrt(thr' C) / p) / C and the left edge
// (-B dy - s) / A smallest at the opposite dy, each clamped to the band.  A tile is kept when
// its pixel-centre columns [X0, X1] meet [xl, xr]; the kept tiles of a row are contiguous.
// Every step is one correctly rounded float32 operation (square roots and divisions
// included) in a fixed order with no contraction, so the decision is reproducible bit for
// bit.  Returns false when the band misses the ellipse.
struct RowSpan {
    float xl, xr;  // extent of the footprint in the band, relative to the mean
    float uf;      // fraction of the mean
    int ui;        // integer part of the mean
};
// The band-independent part of the rule: the mean and the ellipse's constants.
struct Footprint {
    float uf, vf;            // fractions of the mean
    int ui, vi;              // integer parts of the mean
    float A, B, Cq, p, At;   // A thr' = At
    float dymax, dyr;        // |dy| bound; dy of the right edge's maximum
};
__device__ __forceinline__ Footprint footprint(const float4 g0, const float4 g1, float ex) {
    Footprint f;
    const uint32_t packed = __float_as_uint(g1.w);
    f.ui = (int)(short)(packed & 0xffffu);
    f.vi = (int)(short)(packed >> 16);
    f.uf = g0.x;
    f.vf = g0.y;
    const float m00 = g1.x, m10 = g1.y, m11 = g1.z;
    const float t = __fmul_rn(__fmul_rn(__fsub_rn(ex, 0x1.47ae14p-7f /* float(0.01) */), 0x1.fefa62p-1f /* float(1/1.002) */),
                              m00);
    const float thr = __fmul_rn(t, t);
    f.A = __fadd_rn(__fmul_rn(m00, m00), __fmul_rn(m10, m10));
    f.B = __fmul_rn(m10, m11);
    f.Cq = __fmul_rn(m11, m11);
    f.p = __fmul_rn(m00, m11);
    f.dymax = __fdiv_rn(__fsqrt_rn(__fmul_rn(f.A, thr)), f.p);
    const float dxmax = __fdiv_rn(__fsqrt_rn(__fmul_rn(thr, f.Cq)), f.p);
    f.dyr = -__fdiv_rn(__fmul_rn(f.B, dxmax), f.Cq);
    f.At = __fmul_rn(f.A, thr);
    return f;
}
// The span of the footprint within the band of pixel-centre rows [Y0, Y1].
__device__ __forceinline__ bool band_span(const Footprint &f, int Y0, int Y1, RowSpan &rs) {
    rs.ui = f.ui;
    rs.uf = f.uf;
    const float y0 = __fsub_rn((float)(Y0 - f.vi), f.vf), y1 = __fsub_rn((float)(Y1 - f.vi), f.vf);
    const float yb0 = fmaxf(y0, -f.dymax), yb1 = fminf(y1, f.dymax);
    if (!(yb0 <= yb1)) return false;
    auto s_of = [&](float dy) {
        const float q = __fmul_rn(f.p, dy);
        return __fsqrt_rn(fmaxf(__fsub_rn(f.At, __fmul_rn(q, q)), 0.f));
    };
    const float dr = fminf(yb1, fmaxf(yb0, f.dyr));
    const float dl = fminf(yb1, fmaxf(yb0, -f.dyr));
    rs.xr = __fdiv_rn(__fsub_rn(s_of(dr), __fmul_rn(f.B, dr)), f.A);
    rs.xl = __fdiv_rn(__fsub_rn(-__fmul_rn(f.B, dl), s_of(dl)), f.A);
    return true;
}
// The same rule in one pass (the band-independent constants after the early exit), for the
// lists without half masks; identical operations, so identical results.
__device__ __forceinline__ bool row_span(const float4 g0, const float4 g1, float ex, int Y0, int Y1, RowSpan &rs) {
    const uint32_t packed = __float_as_uint(g1.w);
    rs.ui = (int)(short)(packed & 0xffffu);
    rs.uf = g0.x;
    const int vi = (int)(short)(packed >> 16);
    const float m00 = g1.x, m10 = g1.y, m11 = g1.z;
    const float t = __fmul_rn(__fmul_rn(__fsub_rn(ex, 0x1.47ae14p-7f /* float(0.01) */), 0x1.fefa62p-1f /* float(1/1.002) */),
                              m00);
    const float thr = __fmul_rn(t, t);
    const float A = __fadd_rn(__fmul_rn(m00, m00), __fmul_rn(m10, m10));
    const float B = __fmul_rn(m10, m11);
    const float Cq = __fmul_rn(m11, m11);
    const float p = __fmul_rn(m00, m11);
    const float y0 = __fsub_rn((float)(Y0 - vi), g0.y), y1 = __fsub_rn((float)(Y1 - vi), g0.y);
    const float dymax = __fdiv_rn(__fsqrt_rn(__fmul_rn(A, thr)), p);
    const float yb0 = fmaxf(y0, -dymax), yb1 = fminf(y1, dymax);
    if (!(yb0 <= yb1)) return false;
    const float dxmax = __fdiv_rn(__fsqrt_rn(__fmul_rn(thr, Cq)), p);
    const float dyr = -__fdiv_rn(__fmul_rn(B, dxmax), Cq);
    const float At = __fmul_rn(A, thr);
    auto s_of = [&](float dy) {
        const float q = __fmul_rn(p, dy);
        return __fsqrt_rn(fmaxf(__fsub_rn(At, __fmul_rn(q, q)), 0.f));
    };
    const float dr = fminf(yb1, fmaxf(yb0, dyr));
    const float dl = fminf(yb1, fmaxf(yb0, -dyr));
    rs.xr = __fdiv_rn(__fsub_rn(s_of(dr), __fmul_rn(B, dr)), A);
    rs.xl = __fdiv_rn(__fsub_rn(-__fmul_rn(B, dl), s_of(dl)), A);
    return true;
}
// does the row's footprint [xl, xr] meet the pixel-centre columns [X0, X1]?
__device__ __forceinline__ bool span_meets(const RowSpan &rs, int X0, int X1) {
    return __fsub_rn((float)(X1 - rs.ui), rs.uf) >= rs.xl && __fsub_rn((float)(X0 - rs.ui), rs.uf) <= rs.xr;
}

// The kept tile columns [a, b) of a row within [tx0, tx1): the tiles whose pixel-centre
// columns meet the span.  Both halves of span_meets are monotone in the column (the left test
// turns true once, the right test turns false once; each is a correctly rounded subtraction
// of an increasing integer), so a is the first column passing the left test and b the first
// failing the right one.  Each is estimated from the span and then moved to the exact
// boundary by the tests themselves (a step or two), so the result equals a walk over every
// column of the rectangle.
__device__ __forceinline__ void span_run(const RowSpan &rs, int tx0, int tx1, int tile_w, int W, int &a, int &b) {
    auto left = [&](int tx) {  // the tile's last pixel-centre column reaches xl
        return __fsub_rn((float)(min(tx * tile_w + tile_w - 1, W - 1) - rs.ui), rs.uf) >= rs.xl;
    };
    auto right = [&](int tx) {  // the tile's first pixel-centre column is within xr
        return __fsub_rn((float)(tx * tile_w - rs.ui), rs.uf) <= rs.xr;
    };
    const float ca = ((float)rs.ui + rs.uf + rs.xl - (float)(tile_w - 1)) / (float)tile_w;
    a = !(ca > (float)tx0) ? tx0 : (!(ca < (float)tx1) ? tx1 : (int)ceilf(ca));  // (NaN: tx0)
    while (a > tx0 && left(a - 1)) --a;
    while (a < tx1 && !left(a)) ++a;
    const float cb = ((float)rs.ui + rs.uf + rs.xr) / (float)tile_w + 1.f;
    b = !(cb > (float)a) ? a : (!(cb < (float)tx1) ? tx1 : (int)floorf(cb));
    while (b > a && !right(b - 1)) --b;
    while (b < tx1 && right(b)) ++b;
    if (b < a) b = a;
}

// With half masks, the kept tiles [a, a + cnt) of a (record, tile row) slot and which halves
// of each tile they may reach (without them the rule above runs once on the tile row's band
// of pixel-centre rows [Y0, Y1]).  The band splits into a top half [Y0, Y0 + tile_h / 2)
// and a bottom half (clamped to the image), the rule runs on each, and a tile is kept when
// its columns meet either half's span.  The two runs [a0, b0), [a1, b1) of one convex
// footprint overlap (their spans cover the whole band's span), so the kept tiles are the
// contiguous run [a, b) = their hull.  half packs the runs relative to a, one byte each
// (a0 - a, b0 - a, a1 - a, b1 - a), or is kHalfAll when the run is longer than 255 tiles
// (every tile then marked as reaching both halves, a conservative superset).
constexpr uint32_t kHalfAll = 0xffffffffu;
struct SlotRun {
    int a, cnt;
    uint32_t half;
};
__device__ __forceinline__ SlotRun slot_run(const float4 g0, const float4 g1, float ex, int Y0, int Y1, int tile_h,
                                            int tx0, int tx1, int tile_w, int W) {
    RowSpan rs;
    const Footprint f = footprint(g0, g1, ex);
    const int Yh = Y0 + tile_h / 2;
    int a0 = tx1, b0 = tx1, a1 = tx1, b1 = tx1;
    if (band_span(f, Y0, min(Yh - 1, Y1), rs)) span_run(rs, tx0, tx1, tile_w, W, a0, b0);
    if (Yh <= Y1 && band_span(f, Yh, Y1, rs)) span_run(rs, tx0, tx1, tile_w, W, a1, b1);
    const bool e0 = b0 <= a0, e1 = b1 <= a1;
    SlotRun r;
    if (e0 && e1) {
        r.a = tx1;
        r.cnt = 0;
        r.half = 0u;
        return r;
    }
    if (e0) a0 = b0 = a1;
    if (e1) a1 = b1 = a0;
    r.a = min(a0, a1);
    r.cnt = max(b0, b1) - r.a;
    r.half = r.cnt > 255 ? kHalfAll
                         : (uint32_t)(a0 - r.a) | ((uint32_t)(b0 - r.a) << 8) | ((uint32_t)(a1 - r.a) << 16) |
                               ((uint32_t)(b1 - r.a) << 24);
    return r;
}
// Half mask (bit 0 top, bit 1 bottom) of the q-th tile of a slot's run.
__device__ __forceinline__ uint32_t half_mask(uint32_t half, uint32_t q) {
    if (half == kHalfAll) return 3u;
    const uint32_t top = q >= (half & 0xffu) && q < ((half >> 8) & 0xffu);
    const uint32_t bot = q >= ((half >> 16) & 0xffu) && q < (half >> 24);
    return top | (bot << 1);
}

// The (record, tile row) slots: the tile rows of every depth-sorted record's rectangle,
// record after record; P[i] is the first slot of sorted record i and first_rec[b] the record
// that owns slot 256 b (for the first kMaxChunks chunks of 256 slots).
constexpr int kMaxChunks = 1 << 16;
__global__ void __launch_bounds__(kScanThreads) slot_prefix_kernel(const uint2 *__restrict__ rect,
                                                                   const uint32_t *__restrict__ rec,
                                                                   const int *__restrict__ m_ptr,
                                                                   uint64_t *__restrict__ words, int *__restrict__ counter,
                                                                   uint32_t *__restrict__ P,
                                                                   uint32_t *__restrict__ first_rec,
                                                                   int *__restrict__ total, StepWaits sw) {
    pdl_begin();
    constexpr int E = kCompactPerThread;
    const int n = sw.input(*m_ptr);
    const int parts = (n + kCompactPart - 1) / kCompactPart;
    for (int part; (part = next_part(counter)) < parts;) {
        // thread t takes records base + 32 (8 warp + q) + lane: coalesced loads, and the scan runs
        // over warps' blocks of 256 records
        const int lane = threadIdx.x & 31, base = part * kCompactPart + (int)(threadIdx.x >> 5) * (32 * E);
        uint32_t c[E], incl[E], sum = 0;
#pragma unroll
        for (int q = 0; q < E; ++q) {
            const int i = base + 32 * q + lane;
            c[q] = i < n ? rect_rows(rect[rec[i]]) : 0u;
        }
#pragma unroll
        for (int q = 0; q < E; ++q) {
            uint32_t v = c[q];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(SG_FULL_MASK, v, o);
                if (lane >= o) v += t;
            }
            incl[q] = sum + v;
            sum += __shfl_sync(SG_FULL_MASK, v, 31);
        }
        uint32_t tot;
        const uint32_t ex = block_exclusive_scan(lane == 0 ? sum : 0u, tot);
        const uint32_t off = block_look_back(words, part, tot, sw) + __shfl_sync(SG_FULL_MASK, ex, 0);
        if (part == parts - 1 && threadIdx.x == 0) *total = (int)(off + tot);
#pragma unroll
        for (int q = 0; q < E; ++q) {
            const int i = base + 32 * q + lane;
            if (i >= n) continue;
            const uint64_t p = off + incl[q] - c[q];
            P[i] = (uint32_t)p;
            for (uint64_t b = (p + 255) / 256; b * 256 < p + c[q] && b < (uint64_t)kMaxChunks; ++b)
                first_rec[b] = (uint32_t)i;
        }
    }
}

// The sorted record that owns slot s: the last i with P[i] <= s among records that have slots
// (all records in the lists have at least one row).
__device__ __forceinline__ int slot_owner(const uint32_t *__restrict__ P, int n, uint32_t s) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = lo + (hi - lo + 1) / 2;
        if (P[mid] <= s) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Digits of the tile sort's passes.
struct Digits {
    int n;
    int shift[4];
    uint32_t mask[4];
};

// Culling and emission over the slots, in chunks of 256 (a thread's slot each).  A part is one
// chunk for small inputs; for larger ones it is several, at most two parts per block (one chunk
// at a time measured 490 against 360 us on the batched workload), counted before the part's
// place is known and emitted afterwards from the slot cache (the tile sort's idle ping-pong
// buffers and the output tile ids, when they hold every slot).  A slot's record is found by a binary search
// over the prefixes of the (at most 256) records that can own the chunk, staged in shared
// memory; the row's footprint span gives the contiguous run of kept tile columns.  The part's
// kept counts give its instances' place by the chained scan, and consecutive threads write
// consecutive instances (global tile id, record), each finding its slot by a binary search
// over the slots' offsets: (record, row, column) order.  The few near records with huge
// rectangles are spread over many parts.  Also counted here: the tile ids' digit histograms;
// and the words of the tile sort's first pass are cleared for the parts that start among the
// emitted instances (sweep_part each).
// HALVES: the rule runs per half tile row (slot_run) and the emitted records carry each
// tile's half mask in bits 30-31.
template <bool HALVES>
__global__ void __launch_bounds__(kScanThreads, 6) cull_kernel(
    const uint2 *__restrict__ rect, const float4 *__restrict__ geo, const float2 *__restrict__ ext,
    const uint32_t *__restrict__ rec, const int *__restrict__ m_ptr, const int *__restrict__ s_ptr,
    const uint32_t *__restrict__ P, const uint32_t *__restrict__ first_rec, uint64_t *__restrict__ words,
    int *__restrict__ counter, int N, const sg_view *__restrict__ views, int n_views, int tile_w, int tile_h,
    uint32_t *__restrict__ tkey, uint32_t *__restrict__ tval, int capacity, int *__restrict__ total, Digits dg,
    uint32_t *__restrict__ hist, uint64_t *__restrict__ sweep_words, int sweep_part, uint32_t *__restrict__ slot_tf,
    uint32_t *__restrict__ slot_cnt, uint32_t *__restrict__ slot_half, StepWaits sw) {
    pdl_begin();
    __shared__ uint32_t s_P[kScanThreads], s_ex[kScanThreads], s_tf[kScanThreads], s_or[kScanThreads],
        s_hf[HALVES ? kScanThreads : 1];
    __shared__ uint32_t s_h[4 * 256];
    __shared__ int s_next;
    __shared__ int4 s_vw[SG_MAX_VIEWS];  // (W, H, tile_offset, tiles_x) of each view-level
    for (int v = threadIdx.x; v < n_views; v += kScanThreads)
        s_vw[v] = make_int4(views[v].W, views[v].H, views[v].tile_offset, views[v].tiles_x);
    for (int i = threadIdx.x; i < 4 * 256; i += kScanThreads) s_h[i] = 0;
    const int n = *m_ptr;
    const uint32_t S = (uint32_t)sw.input(*s_ptr);  // (without slots no record is read)
    const int chunks = (int)(((uint64_t)S + 255) / 256);
    // chunks of a part: at most two parts per block, one chunk for small inputs
    const int per = max(1, max((chunks + kMaxChunks - 1) / kMaxChunks, (chunks + 2 * (int)gridDim.x - 1) / (2 * (int)gridDim.x)));
    const bool cached = S <= (uint32_t)capacity;  // the slot cache holds every slot
    const int parts = (chunks + per - 1) / per;
    bool overflow = false;
    // the slot c0 + threadIdx.x, c0 in sorted record ic: its kept tiles [tfirst, tfirst + count),
    // from the slot cache when an earlier pass over the part stored them (use), or stored there
    auto slot = [&](uint64_t c0, int ic, int &k, uint32_t &orec, uint32_t &tfirst, uint32_t &half, bool use,
                    bool store) {
        const int j = ic + (int)threadIdx.x;
        s_P[threadIdx.x] = j < n ? P[j] : 0xffffffffu;
        __syncthreads();
        k = 0;
        orec = tfirst = half = 0;
        uint32_t cnt = 0;
        const uint32_t s = (uint32_t)(c0 + threadIdx.x);
        if (c0 + threadIdx.x < S) {
            int lo = 0, hi = kScanThreads - 1;  // the last k with s_P[k] <= s (s_P[0] <= c0)
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (s_P[mid] <= s) lo = mid; else hi = mid - 1;
            }
            k = lo;
            orec = rec[ic + k];
            if (use) {
                tfirst = slot_tf[s];
                cnt = slot_cnt[s];
                if (HALVES) half = slot_half[s];
            } else {
                const uint2 rc = rect[orec];
                const int tx0 = (int)(rc.x & 0xffffu), tx1 = (int)(rc.y & 0xffffu);
                const int ty = (int)(rc.x >> 16) + (int)(s - s_P[k]);
                const int4 vw = s_vw[orec / (uint32_t)N];
                const int Y0 = ty * tile_h;
                const int Y1 = min(Y0 + tile_h - 1, vw.y - 1);
                int tx_a = tx1;
                if constexpr (HALVES) {
                    const SlotRun sr = slot_run(geo[2 * (size_t)orec], geo[2 * (size_t)orec + 1], ext[orec].x, Y0, Y1,
                                                tile_h, tx0, tx1, tile_w, vw.x);
                    cnt = (uint32_t)sr.cnt;
                    half = sr.half;
                    tx_a = sr.a;
                } else {
                    RowSpan rs;
                    if (row_span(geo[2 * (size_t)orec], geo[2 * (size_t)orec + 1], ext[orec].x, Y0, Y1, rs)) {
                        // the kept columns are contiguous
                        int tb;
                        span_run(rs, tx0, tx1, tile_w, vw.x, tx_a, tb);
                        cnt = (uint32_t)(tb - tx_a);
                        if (!cnt) tx_a = tx1;
                    }
                }
                tfirst = (uint32_t)vw.z + (uint32_t)ty * (uint32_t)vw.w + (uint32_t)tx_a;
                if (store) {
                    slot_tf[s] = tfirst;
                    slot_cnt[s] = cnt;
                    if (HALVES) slot_half[s] = half;
                }
            }
        }
        // the next chunk starts in the record that owns this chunk's last slot, or in the one after
        // if that ends here (its prefix is not staged when the 256 slots have 256 owners)
        if (threadIdx.x == kScanThreads - 1) {
            const int e = ic + k + 1;
            const uint32_t after = k + 1 < kScanThreads ? s_P[k + 1] : e < n ? P[e] : 0xffffffffu;
            s_next = after <= c0 + kScanThreads ? e : e - 1;
        }
        return cnt;
    };
    // the chunk's instances [run, run + tot)
    auto emit = [&](uint32_t run, uint32_t ex, uint32_t cnt, uint32_t tot, uint32_t orec, uint32_t tfirst,
                    uint32_t half) {
        // the upper digits are the same over most of a run: counted per slot, the lowest per
        // instance below (per instance they would serialise on a few shared words)
        const uint64_t at = (uint64_t)run + ex;
        const uint32_t kept = at < (uint64_t)capacity ? (uint32_t)min((uint64_t)cnt, (uint64_t)capacity - at) : 0u;
#pragma unroll
        for (int d = 1; d < 4; ++d) {
            if (d >= dg.n) break;
            for (uint32_t t = tfirst, left = kept; left > 0;) {
                const uint32_t m = min(left, (((t >> dg.shift[d]) + 1u) << dg.shift[d]) - t);
                atomicAdd(&s_h[256 * d + ((t >> dg.shift[d]) & dg.mask[d])], m);
                t += m;
                left -= m;
            }
        }
        s_ex[threadIdx.x] = ex;
        s_tf[threadIdx.x] = tfirst;
        s_or[threadIdx.x] = orec;
        if (HALVES) s_hf[threadIdx.x] = half;
        __syncthreads();
        for (uint32_t o = threadIdx.x; o < tot; o += kScanThreads) {
            int lo = 0, hi = kScanThreads - 1;  // the last slot t with s_ex[t] <= o
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (s_ex[mid] <= o) lo = mid; else hi = mid - 1;
            }
            const uint32_t g = run + o;
            if (g < (uint32_t)capacity) {
                const uint32_t q = o - s_ex[lo], t = s_tf[lo] + q;
                tkey[g] = t;
                // (with halves, records are below 2^30: checked by the caller)
                tval[g] = HALVES ? s_or[lo] | (half_mask(s_hf[lo], q) << 30) : s_or[lo];
                atomicAdd(&s_h[t & dg.mask[0]], 1u);
            } else {
                overflow = true;
            }
        }
        __syncthreads();
    };
    for (int part; (part = next_part(counter)) < parts;) {
        const int b0 = part * per, b1 = min(chunks, b0 + per);
        const int i0 = b0 < kMaxChunks ? (int)first_rec[b0] : slot_owner(P, n, (uint32_t)b0 * 256u);
        int k;
        uint32_t orec, tfirst, half, run, sum = 0, tot;
        if (per == 1) {
            const uint32_t cnt = slot((uint64_t)b0 * 256, i0, k, orec, tfirst, half, false, false);
            const uint32_t ex = block_exclusive_scan(cnt, tot);
            run = block_look_back(words, part, tot, sw);
            sum = tot;
            emit(run, ex, cnt, tot, orec, tfirst, half);
        } else {
            int ic = i0;
            uint32_t kept = 0;
            for (int b = b0; b < b1; ++b) {
                kept += slot((uint64_t)b * 256, ic, k, orec, tfirst, half, false, cached);
                __syncthreads();
                ic = s_next;
            }
            block_exclusive_scan(kept, sum);
            run = block_look_back(words, part, sum, sw);
            ic = i0;
            uint32_t at = run;
            for (int b = b0; b < b1; ++b) {
                const uint32_t cnt = slot((uint64_t)b * 256, ic, k, orec, tfirst, half, cached, false);
                const uint32_t ex = block_exclusive_scan(cnt, tot);
                ic = s_next;
                emit(at, ex, cnt, tot, orec, tfirst, half);
                at += tot;
            }
        }
        if (part == parts - 1 && threadIdx.x == 0) *total = (int)(run + sum);
        const uint64_t end = min((uint64_t)run + sum, (uint64_t)capacity);
        for (uint64_t q = ((uint64_t)run + sweep_part - 1) / sweep_part; q * sweep_part < end; ++q)
            sweep_words[q * 256 + threadIdx.x] = 0;
    }
    flush_hist(s_h, 256 * dg.n, hist);
    if (overflow) atomicOr(sw.status, SG_STATUS_CAPACITY);
}

// ---------------------------------------------------------------------------------------
// Stable LSD radix sort of (uint32 key, uint32 value) pairs, 8-bit digits (or fewer).
// ---------------------------------------------------------------------------------------

// One digit pass (digits of at most 8 bits, histogram given).  A part is 256 IPT elements; warp
// w owns the part's elements [32 IPT w, 32 IPT (w + 1)), lane l element 32 it + l of them.
// Ranking needs no block barrier per element row: every warp ranks its own elements against a
// warp-private digit count (warp match_any + the lanes below), one block pass turns the
// per-warp counts into per-digit offsets, thread d publishes digit d's count and looks back for
// its prefix while the part is reordered by digit in shared memory, and consecutive threads
// store consecutive elements of one digit run (coalesced stores instead of one scattered sector
// per element).  clear: the next pass's words, cleared for the parts this pass handles.
constexpr int kSweepIpt = 12;
constexpr int kSweepPart = kScanThreads * kSweepIpt;
__global__ void __launch_bounds__(kScanThreads, 4) sweep_kernel(
    const uint32_t *__restrict__ kin, const uint32_t *__restrict__ vin, uint32_t *__restrict__ kout,
    uint32_t *__restrict__ vout, const int *__restrict__ n_ptr, int cap, int shift, uint32_t mask,
    const uint32_t *__restrict__ hist, uint64_t *__restrict__ words, uint64_t *__restrict__ clear,
    int *__restrict__ counter, StepWaits sw) {
    pdl_begin();
    constexpr int kWarps = kScanThreads / 32, IPT = kSweepIpt, CH = kSweepPart;
    __shared__ uint32_t to[256];            // output position of the part's slot 0 if it had digit d
    __shared__ uint32_t loc[256];           // first slot of each digit in the reordered part
    __shared__ uint32_t wcnt[kWarps][256];  // per-warp digit counts, then per-warp offsets
    __shared__ uint32_t skey[CH], sval[CH];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = sw.input(min(*n_ptr, cap));
    const int parts = (int)(((int64_t)n + CH - 1) / CH);
    uint32_t unused;
    const uint32_t first = block_exclusive_scan(hist[tid], unused);  // digit tid's first output position
    const uint32_t lt_mask = (1u << lane) - 1u;
    uint32_t *wc = wcnt[warp];
    for (int part; (part = next_part(counter)) < parts;) {
        const int cbase = part * CH, cn = min(CH, n - cbase);
#pragma unroll
        for (int q = 0; q < 8; ++q) wc[32 * q + lane] = 0;
        const int wbase = 32 * IPT * warp;
        uint32_t key[IPT], val[IPT], rank[IPT];
        // all of the warp's loads first (their latencies overlap), then the ranking; each pair is
        // read once: evict-first loads, which leave L2 to the partly written output lines
#pragma unroll
        for (int it = 0; it < IPT; ++it) {
            const int i = wbase + 32 * it + lane;
            key[it] = i < cn ? __ldcs(kin + cbase + i) : 0u;
            val[it] = i < cn ? __ldcs(vin + cbase + i) : 0u;
        }
        __syncwarp();
#pragma unroll
        for (int it = 0; it < IPT; ++it) {
            const bool valid = wbase + 32 * it + lane < cn;
            const uint32_t d = valid ? ((key[it] >> shift) & mask) : 256u;
            const uint32_t peers = __match_any_sync(SG_FULL_MASK, d);
            const uint32_t below = __popc(peers & lt_mask);
            rank[it] = valid ? wc[d] + below : 0u;
            __syncwarp();
            if (valid && below == 0) wc[d] += __popc(peers);
            __syncwarp();
        }
        __syncthreads();
        // digit tid: exclusive offsets of the warps, the part's count
        uint32_t cnt = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t c = wcnt[w][tid];
            wcnt[w][tid] = cnt;
            cnt += c;
        }
        uint64_t *word = words + (size_t)part * 256 + tid;
        const bool digit = tid <= (int)mask;  // (the other threads' counts are 0)
        if (digit && !(sw.withhold && part == 0)) store_word(word, (part == 0 ? kPrefix : kAggregate) | cnt);
        const uint32_t slot0 = block_exclusive_scan(cnt, unused);
        loc[tid] = slot0;
        __syncthreads();
#pragma unroll
        for (int it = 0; it < IPT; ++it) {
            if (wbase + 32 * it + lane < cn) {
                const uint32_t d = (key[it] >> shift) & mask;
                const uint32_t li = loc[d] + wc[d] + rank[it];
                skey[li] = key[it];
                sval[li] = val[it];
            }
        }
        uint32_t before = 0;
        if (part > 0 && (tid & ~31) <= (int)mask) {  // (warp-uniform)
            bool late = false;
            before = look_back(words + tid, 256, part, digit, sw, late);
            if (digit) store_word(word, kPrefix | (uint64_t)(before + cnt));
            __syncwarp();
        }
        to[tid] = first + before - slot0;
        if (clear) clear[(size_t)part * 256 + tid] = 0;
        __syncthreads();
        for (int j = tid; j < cn; j += kScanThreads) {
            const uint32_t k = skey[j];
            const uint32_t pos = to[(k >> shift) & mask] + (uint32_t)j;
            if (pos >= (uint32_t)n) continue;  // (only after a timeout)
            kout[pos] = k;
            vout[pos] = sval[j];
        }
        // (next_part's barriers order these reads before the next part's writes)
    }
}

// Splits `bits` into the fewest passes of at most max_bits bits, as evenly as possible.
static Digits split_digits(int bits, int max_bits) {
    Digits d{};
    d.n = (bits + max_bits - 1) / max_bits;
    int shift = 0;
    for (int p = 0; p < d.n; ++p) {
        const int nb = (bits - shift + (d.n - p) - 1) / (d.n - p);
        d.shift[p] = shift;
        d.mask[p] = (1u << nb) - 1u;
        shift += nb;
    }
    return d;
}

// Sorts n (device count, clamped to cap) pairs by the digits dg from (kin, vin) into
// (kout, vout) using (ktmp, vtmp) as ping-pong; kin/vin are not modified.  hist: the digits'
// histograms (256 words each); words[0]: the first pass's chained-scan words, cleared for every
// part; words[1]: the second pass's (the passes alternate between the two and each clears its
// successor's); counters: one per pass, zero; waits: one per pass.
static void radix_sort(const uint32_t *kin, const uint32_t *vin, uint32_t *kout, uint32_t *vout, uint32_t *ktmp,
                       uint32_t *vtmp, const int *n_ptr, int cap, const Digits &dg, const uint32_t *hist,
                       uint64_t *const words[2], int *counters, int grid, const StepWaits *waits, cudaStream_t st) {
    const uint32_t *ks = kin, *vs = vin;
    for (int p = 0; p < dg.n; ++p) {
        uint32_t *kd = ((dg.n - 1 - p) % 2 == 0) ? kout : ktmp;
        uint32_t *vd = ((dg.n - 1 - p) % 2 == 0) ? vout : vtmp;
        launch_pdl(sweep_kernel, grid, kScanThreads, 0, st, ks, vs, kd, vd, n_ptr, cap, dg.shift[p], dg.mask[p],
                   hist + 256 * p, words[p & 1], p + 1 < dg.n ? words[(p + 1) & 1] : (uint64_t *)nullptr, counters + p,
                   waits[p]);
        count_launches(1);
        ks = kd;
        vs = vd;
    }
}

// ---------------------------------------------------------------------------------------
// Ranges and work order
// ---------------------------------------------------------------------------------------

__device__ __forceinline__ int lower_bound_u32(const uint32_t *__restrict__ a, int lo, int hi, uint32_t key) {
    while (lo < hi) {
        const int mid = lo + ((hi - lo) >> 1);
        if (a[mid] < key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The same for a whole warp and one key, 32 probes at a time.
__device__ __forceinline__ int warp_lower_bound_u32(const uint32_t *__restrict__ a, int n, uint32_t key) {
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = n;  // the answer is in [lo, hi]
    while (hi > lo) {
        const int64_t len = hi - lo;
        const int probe = lo + (int)(len * lane / 32);  // ascending; probe of lane 0 is lo
        const uint32_t less = __ballot_sync(SG_FULL_MASK, a[probe] < key);
        const int m = __popc(less);  // probes below the key: a prefix of the lanes
        if (m == 0) return lo;
        const int nlo = lo + (int)(len * (m - 1) / 32) + 1;
        hi = m == 32 ? hi : lo + (int)(len * m / 32);
        lo = nlo;
    }
    return lo;
}

// Work-order bucket of a tile with n instances: 63 - b, b = 0 for n = 0, else
// 1 + 2 floor(log2 n) + the bit below the leading one (descending length, 6 bits).
__device__ __forceinline__ uint32_t length_bucket(int2 r) {
    const uint32_t n = (uint32_t)max(r.y - r.x, 0);
    if (n == 0) return 63u;
    const int lz = 31 - __clz(n);
    const uint32_t sub = lz >= 1 ? (n >> (lz - 1)) & 1u : 0u;
    return 63u - (1u + 2u * (uint32_t)lz + sub);
}

// [start, end) of every tile by search in the sorted tile ids ((0, 0) for a tile with no
// instance): one warp per 32 tiles finds its first and its last bound together, then each lane
// its own bound in between.  hist (or null): counts of the length buckets.  *failed: the last
// step's flag.
__global__ void __launch_bounds__(kScanThreads) ranges_kernel(const uint32_t *__restrict__ tile,
                                                              int *__restrict__ k_ptr, int cap, int n_tiles,
                                                              int2 *__restrict__ ranges, uint32_t *__restrict__ hist,
                                                              const int *__restrict__ failed) {
    pdl_begin();
    const int found = *k_ptr;
    const bool broken = *failed != 0;  // (a step gave up: no instances)
    if (broken && blockIdx.x == 0 && threadIdx.x == 0) *k_ptr = 0;
    __shared__ uint32_t s_h[64];
    if (threadIdx.x < 64) s_h[threadIdx.x] = 0;
    __syncthreads();
    const int K = broken ? 0 : min(found, cap), lane = threadIdx.x & 31;
    const int t = blockIdx.x * kScanThreads + (int)threadIdx.x, t0 = t - lane;
    if (t0 < n_tiles) {  // (warp-uniform)
        const int wlo = warp_lower_bound_u32(tile, K, (uint32_t)t0);
        const int whi = warp_lower_bound_u32(tile, K, (uint32_t)t0 + 32u);
        const int lo = lower_bound_u32(tile, wlo, whi, (uint32_t)t);
        int hi = __shfl_down_sync(SG_FULL_MASK, lo, 1);
        if (lane == 31) hi = whi;
        if (t < n_tiles) {
            const int2 r = lo < hi ? make_int2(lo, hi) : make_int2(0, 0);
            ranges[t] = r;
            if (hist) atomicAdd(&s_h[length_bucket(r)], 1u);
        }
    }
    if (hist) flush_hist(s_h, 64, hist);
}

// The work order: a stable counting sort of the tiles by length bucket.  A block's part is a
// contiguous range of tiles (grid parts, 256 tiles at a time), counted, placed by the chained
// scan (64 words per part) and written.  A part whose wait gives up counts the tiles before it
// itself, so that the order always holds every tile.
__global__ void __launch_bounds__(kScanThreads) order_kernel(const int2 *__restrict__ ranges, int n_tiles,
                                                             const uint32_t *__restrict__ hist,
                                                             uint64_t *__restrict__ words, int *__restrict__ counter,
                                                             int *__restrict__ order, StepWaits sw) {
    pdl_begin();
    constexpr int kWarps = kScanThreads / 32;
    __shared__ uint32_t s_cnt[64], s_run[64], s_w[kWarps][64];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rows = (n_tiles + kScanThreads - 1) / kScanThreads;
    const int per = (rows + (int)gridDim.x - 1) / (int)gridDim.x * kScanThreads;  // tiles of a part
    const int part = next_part(counter);
    const int64_t beg = (int64_t)part * per, end = min((int64_t)n_tiles, beg + per);
    uint32_t unused;
    const uint32_t first = block_exclusive_scan(tid < 64 ? hist[tid] : 0u, unused);
    if (tid < 64) s_cnt[tid] = 0;
    __syncthreads();
    for (int64_t i = beg + tid; i < end; i += kScanThreads) atomicAdd(&s_cnt[length_bucket(ranges[i])], 1u);
    __syncthreads();
    if (tid < 64) {
        uint64_t *word = words + (size_t)part * 64 + tid;
        if (!(sw.withhold && part == 0)) store_word(word, (part == 0 ? kPrefix : kAggregate) | s_cnt[tid]);
        uint32_t before = 0;
        if (part > 0) {
            bool late = false;
            before = look_back(words + tid, 64, part, true, sw, late);
            if (late) {
                before = 0;
                for (int64_t i = 0; i < beg; ++i) before += length_bucket(ranges[i]) == (uint32_t)tid;
            }
            store_word(word, kPrefix | (uint64_t)(before + s_cnt[tid]));
        }
        s_run[tid] = first + before;
    }
    const uint32_t lt_mask = (1u << lane) - 1u;
    for (int64_t base = beg; base < end; base += kScanThreads) {
        s_w[warp][lane] = s_w[warp][lane + 32] = 0;
        __syncwarp();
        const int64_t i = base + tid;
        const uint32_t d = i < end ? length_bucket(ranges[i]) : 64u;
        const uint32_t peers = __match_any_sync(SG_FULL_MASK, d);
        const uint32_t below = __popc(peers & lt_mask);
        if (d < 64u && below == 0) s_w[warp][d] = __popc(peers);
        __syncthreads();
        if (tid < 64) {  // the warps' first positions in this row of 256 tiles
            uint32_t run = s_run[tid];
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const uint32_t c = s_w[w][tid];
                s_w[w][tid] = run;
                run += c;
            }
            s_run[tid] = run;
        }
        __syncthreads();
        if (d < 64u) {
            const uint32_t pos = s_w[warp][d] + below;
            order[pos] = (int)i;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------
// Workspace layout
// ---------------------------------------------------------------------------------------

// Steps of a list build: its kernels with a chained scan (each has a part counter and a flag).
enum { kCtrCompact = 0, kCtrDepth = 1, kCtrSlots = 5, kCtrCull = 6, kCtrTile = 7, kCtrOrder = 11, kCtrs = 12 };

struct TileWorkspace {
    uint32_t *dkey_in, *dval_in, *dkey_out, *dval_out, *dkey_tmp, *dval_tmp;
    uint32_t *slot0;      // first (record, tile row) slot of each depth-sorted record
    uint32_t *first_rec;  // record owning the first slot of each 256-slot chunk
    uint32_t *tkey_in, *tval_in, *tkey_tmp, *tval_tmp;
    // cleared by a memset at the start of every list build, [zero, zero + zero_bytes):
    char *zero;
    size_t zero_bytes;
    int *counts;    // [0] visible records M, [1] slots S
    int *counters;  // kCtrs part counters
    int *failed;    // kCtrs flags of steps that gave up
    uint32_t *dhist, *thist, *ohist;                      // 4 x 256, 4 x 256, 64
    uint64_t *cwords, *swords, *kwords, *owords;  // chained-scan words: compaction, slots, culling, order
    uint64_t *sweep[2];  // radix passes: [0] is cleared for the depth sort's parts
};

static int sort_grid() {
    static int G = 0;
    if (!G) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        G = sms > 0 ? 4 * sms : 512;
        if (G > 4096) G = 4096;
    }
    return G;
}

static size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

static int64_t sweep_parts(int64_t n) { return (n + kSweepPart - 1) / kSweepPart; }

static size_t tile_ws_layout(int64_t R, int32_t cap, int G, TileWorkspace *ws, char *base) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *p = base ? base + off : nullptr;
        off += align_up(bytes);
        return p;
    };
    const size_t r4 = (size_t)R * 4, c4 = (size_t)cap * 4;
    TileWorkspace w{};
    w.dkey_in = (uint32_t *)take(r4);
    w.dval_in = (uint32_t *)take(r4);
    w.dkey_out = (uint32_t *)take(r4);
    w.dval_out = (uint32_t *)take(r4);
    w.dkey_tmp = (uint32_t *)take(r4);
    w.dval_tmp = (uint32_t *)take(r4);
    w.slot0 = (uint32_t *)take(r4);
    w.first_rec = (uint32_t *)take((size_t)kMaxChunks * 4);
    w.tkey_in = (uint32_t *)take(c4);
    w.tval_in = (uint32_t *)take(c4);
    w.tkey_tmp = (uint32_t *)take(c4);
    w.tval_tmp = (uint32_t *)take(c4);
    const size_t z0 = off;
    const size_t rparts = (size_t)((R + kCompactPart - 1) / kCompactPart);
    w.zero = take(0);
    w.counts = (int *)take(4 * sizeof(int));
    w.counters = (int *)take(kCtrs * sizeof(int));
    w.failed = (int *)take(kCtrs * sizeof(int));
    w.dhist = (uint32_t *)take(4 * 256 * 4);
    w.thist = (uint32_t *)take(4 * 256 * 4);
    w.ohist = (uint32_t *)take(64 * 4);
    w.cwords = (uint64_t *)take(rparts * 8);
    w.swords = (uint64_t *)take(rparts * 8);
    w.kwords = (uint64_t *)take((size_t)kMaxChunks * 8);
    w.owords = (uint64_t *)take((size_t)G * 64 * 8);
    const size_t sweep_bytes = (size_t)std::max(sweep_parts(R), sweep_parts(cap)) * 256 * 8;
    w.zero_bytes = off - z0 + (size_t)sweep_parts(R) * 256 * 8;
    w.sweep[0] = (uint64_t *)take(sweep_bytes);
    w.sweep[1] = (uint64_t *)take(sweep_bytes);
    if (ws) *ws = w;
    return off;
}

size_t tile_lists_workspace_size(int64_t R, int32_t cap) {
    return tile_ws_layout(R, cap, sort_grid(), nullptr, nullptr);
}

sg_status launch_build_tile_lists(const sg_projected *proj, int N, int n_views,
                                  const sg_view *views, int n_tiles, int tile_w, int tile_h, sg_tile_lists *lists,
                                  void *workspace, size_t ws_bytes, uint32_t *status,
                                  cudaStream_t st, int withheld_step, uint32_t polls) {
    const int G = sort_grid();
    const int64_t R = (int64_t)N * n_views;
    TileWorkspace w;
    const size_t need = tile_ws_layout(R, lists->capacity, G, &w, (char *)workspace);
    if (ws_bytes < need) {
        set_error("build_tile_lists: workspace %zu bytes < %zu needed", ws_bytes, need);
        return SG_ERR_CAPACITY;
    }
    const uint2 *rect = reinterpret_cast<const uint2 *>(proj->rect);
    const float4 *geo = reinterpret_cast<const float4 *>(proj->geo);
    const float2 *ext = reinterpret_cast<const float2 *>(proj->ext);
    auto grid = [G](int64_t parts) { return (int)std::max<int64_t>(1, std::min<int64_t>(G, parts)); };
    if (!polls) polls = kSpinLimit;
    StepWaits waits[kCtrs];
    for (int k = 0; k < kCtrs; ++k)
        waits[k] = {status, k ? w.failed + k - 1 : nullptr, w.failed + k, polls, k == withheld_step};
    cudaMemsetAsync(w.zero, 0, w.zero_bytes, st);
    // 1. compaction of the visible records (count -> counts[0])
    const int cgrid = grid((R + kCompactPart - 1) / kCompactPart);
    launch_pdl(compact_kernel, cgrid, kScanThreads, 0, st, rect, geo, (int)R, w.cwords, w.counters + kCtrCompact,
               w.dkey_in, w.dval_in, w.counts, w.dhist, lists->count, waits[kCtrCompact]);
    // 2. depth sort (32 bits)
    radix_sort(w.dkey_in, w.dval_in, w.dkey_out, w.dval_out, w.dkey_tmp, w.dval_tmp, w.counts, (int)R,
               split_digits(32, 8), w.dhist, w.sweep, w.counters + kCtrDepth, grid(sweep_parts(R)), waits + kCtrDepth, st);
    // 3. slots: the rectangle tile rows of the records in depth order (their number ->
    // counts[1]); culling and emission (K -> lists->count)
    launch_pdl(slot_prefix_kernel, cgrid, kScanThreads, 0, st, rect, w.dval_out, w.counts, w.swords,
               w.counters + kCtrSlots, w.slot0, w.first_rec, w.counts + 1, waits[kCtrSlots]);
    int bits = 1;
    while ((1ll << bits) < (long long)n_tiles) ++bits;
    const Digits dg = split_digits(bits, kTileDigitBits);
    const bool halves = lists->half_masks != 0;  // records carry half masks
    launch_pdl(halves ? cull_kernel<true> : cull_kernel<false>, G + G / 2, kScanThreads, 0, st, rect, geo, ext, w.dval_out,
               w.counts, w.counts + 1, w.slot0, w.first_rec, w.kwords, w.counters + kCtrCull, N, views, n_views, tile_w,
               tile_h, w.tkey_in, w.tval_in, lists->capacity, lists->count, dg, w.thist, w.sweep[0], kSweepPart, w.tkey_tmp, w.tval_tmp,
               lists->tile, waits[kCtrCull]);
    // 4. stable sort by tile id
    radix_sort(w.tkey_in, w.tval_in, lists->tile, lists->record, w.tkey_tmp, w.tval_tmp, lists->count,
               lists->capacity, dg, w.thist, w.sweep, w.counters + kCtrTile, grid(sweep_parts(lists->capacity)),
               waits + kCtrTile, st);
    // 5. tile ranges; 6. work order
    int2 *ranges = reinterpret_cast<int2 *>(lists->ranges);
    const int tblocks = (int)(((int64_t)n_tiles + kScanThreads - 1) / kScanThreads);
    launch_pdl(ranges_kernel, tblocks, kScanThreads, 0, st, lists->tile, lists->count, lists->capacity, n_tiles, ranges,
               lists->order ? w.ohist : (uint32_t *)nullptr, w.failed + kCtrTile + dg.n - 1);
    count_launches(4);  // compaction, slots, culling, ranges
    if (lists->order) {
        launch_pdl(order_kernel, std::min(G, tblocks), kScanThreads, 0, st, ranges, n_tiles, w.ohist,
                   w.owords, w.counters + kCtrOrder, lists->order, waits[kCtrOrder]);
        count_launches(1);
    }
    return check_launch("build_tile_lists");
}

}  // namespace sg
