// mlp.cu -- the learned Gaussian initializer (not in the paper): a 3-layer BF16 MLP with
// FP32 accumulation, 2048 (2009 used) -> 128 -> 128 -> 32 (20 used), trained and run by
// the tcgen05 GEMM of tc_gemm.cuh.
//
// Forward (per batch of B rows, B % 128 == 0):
//   H1 = relu(X W1^T + b1)      A = X [B][2048],  B-operand = W1 [128][2048]
//   H2 = relu(H1 W2^T + b2)     A = H1 [B][128],  B-operand = W2 [128][128]
//   Y  = H2 W3^T + b3           A = H2 [B][128],  B-operand = W3 [32][128]
// Backward of L = sum_o w_o mean_b (Y - T)^2:
//   dY = 2 w (Y - T) / B                               (CUDA cores)
//   dW3^T = H2^T dY   (K = B)   A = H2t [128][B],  B-operand = dYt [32][B]
//   dH2 = (dY W3) * [H2 > 0]    A = dY [B][64],    B-operand = W3t [128][64]
//   dW2^T = H1^T dH2  (K = B)   A = H1t [128][B],  B-operand = dH2t [128][B]
//   dH1 = (dH2 W2) * [H1 > 0]   A = dH2 [B][128],  B-operand = W2t [128][128]
//   dW1 = dH1^T X     (K = B)   A = dH1t [128][B], B-operand = Xt [2048][B]
// Every operand is K-major: the epilogues write the transposed copies (H1t, H2t, dYt,
// dH2t, dH1t) the later GEMMs need, and the patch extractor writes X and Xt.  The K = B
// reductions are split over CTAs.  With a workspace (sg_mlp_backward_ordered, what training uses)
// every split stores its product and the launch that sums the bias gradients adds them in split
// order, so a step gives the same bits every time; without one (sg_mlp_backward) the splits are
// atomically added into the FP32 gradients, in no fixed order.  One ulp of a weight can flip its
// bf16 copy and a ReLU with it: with atomics two runs of three steps differed by up to 1e-3 in
// the moments.
#include <cstdio>
#include <cstring>

#include "tc_gemm.cuh"

namespace sg {

using bf16 = __nv_bfloat16;

// cuTensorMapEncodeTiled from the driver, found through the runtime's entry-point query (the
// library links only the runtime).  NULL when the driver does not provide it.
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled() {
    static EncodeTiledFn fn = nullptr;
    static bool looked = false;
    if (!looked) {
        looked = true;
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
        cudaGetLastError();
    }
    return fn;
}

// Tensor map of a rows x K bf16 operand (K contiguous, leading dimension ld elements) read in
// boxes of 64 (K) x box_rows with the 128-byte swizzle; rows beyond `rows` read as zero.
static bool make_operand_map(CUtensorMap *map, const bf16 *base, long long rows, long long K, long long ld,
                             int box_rows) {
    EncodeTiledFn enc = encode_tiled();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(bf16)};
    const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1u, 1u};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16 *>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN, int STAGES, bool TMA>
static sg_status launch_gemm_kernel(const tc::GemmParams &p, int splits, const CUtensorMap &ma,
                                    const CUtensorMap &mb, cudaStream_t st) {
    constexpr size_t smem = tc::gemm_smem_bytes<BN, STAGES>();
    static bool attr = false;
    if (!attr) {
        if (cudaFuncSetAttribute(tc::gemm_kernel<BN, STAGES, TMA>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem) != cudaSuccess)
            return check_launch("gemm smem attribute");
        attr = true;
    }
    const dim3 grid((p.M + 127) / 128, (p.N + BN - 1) / BN, splits);
    launch_pdl(tc::gemm_kernel<BN, STAGES, TMA>, grid, dim3(128), smem, st, p, ma, mb);
    count_launches(1);
    return check_launch("tcgen05 gemm");
}

template <int BN, int STAGES>
static sg_status launch_gemm_t(const tc::GemmParams &p, int splits, cudaStream_t st) {
    // operands staged by TMA (tensor maps, 128-byte swizzle); by cp.async only when the driver
    // offers no tensor-map encoder
    CUtensorMap ma, mb;
    if (make_operand_map(&ma, p.A, p.M, p.K, p.lda, 128) &&
        make_operand_map(&mb, p.B, p.N, p.K, p.ldb, BN))
        return launch_gemm_kernel<BN, STAGES, true>(p, splits, ma, mb, st);
    memset(&ma, 0, sizeof(ma));
    memset(&mb, 0, sizeof(mb));
    return launch_gemm_kernel<BN, STAGES, false>(p, splits, ma, mb, st);
}

static int sm_count() {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

static int tile_width(int N) { return N <= 32 ? 32 : (N <= 128 ? 128 : 256); }

// Number of parts a K-split product's K range is cut into, so that the grid covers the SMs;
// k_per_split: the K of each (a multiple of 64; the last part may have less, never none).
static int split_count(int M, int N, int K, int max_splits, int &k_per_split) {
    const int tiles = ((M + 127) / 128) * ((N + tile_width(N) - 1) / tile_width(N)), kch = K / 64;
    int splits = (sm_count() + tiles - 1) / tiles;
    if (splits > kch) splits = kch;
    if (splits > max_splits) splits = max_splits;
    if (splits < 1) splits = 1;
    const int per = (kch + splits - 1) / splits;
    k_per_split = per * 64;
    return (kch + per - 1) / per;
}
constexpr int kMaxSplits = 64;

// Chooses the tile width from N and splits K so that the grid covers the SMs.
sg_status launch_gemm(tc::GemmParams p, cudaStream_t st, int max_splits = kMaxSplits) {
    if (p.K % 64 != 0 || p.M <= 0 || p.N <= 0 || p.K <= 0) {
        set_error("gemm: need M, N > 0 and K a positive multiple of 64 (M=%d N=%d K=%d)", p.M, p.N, p.K);
        return SG_ERR_INVALID_ARG;
    }
    const int BN = tile_width(p.N), sms = sm_count();
    const int tiles = ((p.M + 127) / 128) * ((p.N + BN - 1) / BN);
    const bool split_k = (p.f32_atomic || p.split_stride) && p.out_f32 && !p.out_bf16 && !p.out_bf16_t && !p.relu && !p.mask;
    const int splits = split_count(p.M, p.N, p.K, split_k ? max_splits : 1, p.k_per_split);
    if (splits > 1 && p.bias) {
        set_error("gemm: bias with split-K is not supported");
        return SG_ERR_INVALID_ARG;
    }
    p.vec_mask = p.mask && p.ldmask % 8 == 0 && (uintptr_t)p.mask % 16 == 0;
    p.vec_bf16 = p.out_bf16 && p.ld_bf16 % 8 == 0 && (uintptr_t)p.out_bf16 % 16 == 0;
    p.vec_f32 = p.out_f32 && p.ld_f32 % 4 == 0 && (uintptr_t)p.out_f32 % 16 == 0;
    // fewer tiles than half the SMs: narrower ones, each with the same K order, so that more SMs
    // stream the operands; the A rows they read again come from L2.  An SM then takes in 640 or
    // 768 KiB of a 2048-deep layer instead of 1 MiB, in parallel with more of the others (network
    // forward at up to 4864 rows 32.8 -> 26.7 us, at 5120 to 8192 28.7; training step at 2048
    // rows 76 -> 66; the same from 77 tiles on)
    if (BN == 128 && splits == 1 && 2 * tiles <= sms)
        return tiles * ((p.N + 31) / 32) <= sms ? launch_gemm_t<32, 8>(p, splits, st) : launch_gemm_t<64, 6>(p, splits, st);
    switch (BN) {
        case 32: return launch_gemm_t<32, 4>(p, splits, st);
        // with more tiles than SMs, 3 stages of 32 KiB: two CTAs per SM keep twice the operand
        // bytes in flight (layer 1 at 65536 rows: 133 -> 107 us against 4 stages and one CTA);
        // with fewer, one CTA per SM that keeps five chunks in flight
        case 128: return tiles * splits > sms ? launch_gemm_t<128, 3>(p, splits, st) : launch_gemm_t<128, 6>(p, splits, st);
        default: return launch_gemm_t<256, 4>(p, splits, st);
    }
}

static tc::GemmParams gemm_params(const bf16 *A, long long lda, const bf16 *B, long long ldb, int M, int N,
                                  int K, uint32_t *status) {
    tc::GemmParams p{};
    p.A = A; p.lda = lda; p.B = B; p.ldb = ldb;
    p.M = M; p.N = N; p.K = K;
    p.alpha = 1.f;
    p.status = status;
    return p;
}

// ---------------------------------------------------------------------------------------
// small CUDA-core kernels of the MLP
// ---------------------------------------------------------------------------------------

// The bf16 operand copies of the three weight matrices in one launch: fp32 [rows][cols] -> bf16
// [rows][cols], and for W2, W3 also transposed, [cols][ld_t] (columns of the transposed copy
// beyond rows are left untouched: the caller zeroes them once).
__global__ void __launch_bounds__(256) pack_weights_kernel(const float *__restrict__ W1, const float *__restrict__ W2,
                                                           const float *__restrict__ W3, bf16 *__restrict__ W1b,
                                                           bf16 *__restrict__ W2b, bf16 *__restrict__ W3b,
                                                           bf16 *__restrict__ W2t, bf16 *__restrict__ W3t) {
    pdl_begin();
    constexpr int H = SG_MLP_HIDDEN, n1 = H * SG_MLP_IN, n2 = H * H, n3 = SG_MLP_OUT * H;
    int i = blockIdx.x * 256 + threadIdx.x;
    if (i < n1) {
        W1b[i] = __float2bfloat16_rn(W1[i]);
        return;
    }
    i -= n1;
    if (i < n2) {
        const bf16 v = __float2bfloat16_rn(W2[i]);
        W2b[i] = v;
        W2t[(i % H) * H + i / H] = v;
        return;
    }
    i -= n2;
    if (i < n3) {
        const bf16 v = __float2bfloat16_rn(W3[i]);
        W3b[i] = v;
        W3t[(i % H) * 64 + i / H] = v;
    }
}

// dY = 2 w_o (Y - T) / B (bf16, [B][64] with columns >= 32 zero, and [32][B]); loss += sum, or
// the block's share of it into loss_part[block].
// A block takes 64 rows, a thread four outputs of two rows at a time (16-byte loads, 8-byte
// stores); the transposed copy goes through shared memory so that its rows are written 128
// bytes at a time (16384 rows: 27 -> 4 us against one 2-byte store per element).
__global__ void __launch_bounds__(256) mse_head_kernel(const float *__restrict__ Y, const float *__restrict__ T,
                                                       const float *__restrict__ w, int B, bf16 *__restrict__ dY,
                                                       bf16 *__restrict__ dYt, float *__restrict__ loss,
                                                       float *__restrict__ loss_part, bool vec) {
    pdl_begin();
    __shared__ uint16_t s_t[32][64 + 2];
    const int b0 = blockIdx.x * 64;
    float l = 0.f;
    for (int i = threadIdx.x; i < 64 * 8; i += 256) {
        const int r = i >> 3, o = (i & 7) * 4, b = b0 + r;  // (B is a multiple of 128)
        const float *yp = Y + (long long)b * 32 + o, *tp = T + (long long)b * 32 + o;
        float d[4];
        if (vec) {
            const float4 y = *reinterpret_cast<const float4 *>(yp), t = *reinterpret_cast<const float4 *>(tp);
            d[0] = y.x - t.x; d[1] = y.y - t.y; d[2] = y.z - t.z; d[3] = y.w - t.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) d[k] = yp[k] - tp[k];
        }
        uint16_t h[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            l += w[o + k] * d[k] * d[k] / (float)B;
            h[k] = __bfloat16_as_ushort(__float2bfloat16_rn(2.f * w[o + k] * d[k] / (float)B));
            s_t[o + k][r] = h[k];
        }
        uint2 *row = reinterpret_cast<uint2 *>(dY + (long long)b * 64 + o);
        row[0] = make_uint2(h[0] | ((uint32_t)h[1] << 16), h[2] | ((uint32_t)h[3] << 16));
        row[8] = make_uint2(0u, 0u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 32 * 32; i += 256) {
        const int o = i >> 5, r = (i & 31) * 2;
        *reinterpret_cast<uint32_t *>(dYt + (long long)o * B + b0 + r) = s_t[o][r] | ((uint32_t)s_t[o][r + 1] << 16);
    }
    for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(SG_FULL_MASK, l, off);
    if (!loss_part) {
        if ((threadIdx.x & 31) == 0 && l != 0.f) atomicAdd(loss, l);
        return;
    }
    __shared__ float s_l[8];
    if ((threadIdx.x & 31) == 0) s_l[threadIdx.x >> 5] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) t += s_l[k];
        loss_part[blockIdx.x] = t;
    }
}

// Bias gradients: out[r] += sum_c M[r][c] for the rows of three bf16 [rows][cols] matrices (one
// CTA per row; cols is a multiple of 128).  2048 columns at a time through shared memory: 16-byte
// loads, while thread t sums columns t, t + 256, ... in order.
struct RowSums {
    const bf16 *M[3];
    float *out[3];
    int rows[3];
};
__device__ __forceinline__ float block_sum_256(float s) {  // (thread 0 has the sum)
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(SG_FULL_MASK, s, off);
    __shared__ float sw[8];
    if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = s;
    __syncthreads();
    float t = 0.f;
    if (threadIdx.x == 0)
        for (int w = 0; w < 8; ++w) t += sw[w];
    return t;
}
__device__ __forceinline__ void row_sum(const RowSums &a, int cols, int i) {
    const int b1 = a.rows[0], b2 = b1 + a.rows[1];
    const bf16 *M = i < b1 ? a.M[0] : i < b2 ? a.M[1] : a.M[2];
    float *out = i < b1 ? a.out[0] : i < b2 ? a.out[1] : a.out[2];
    const int r = i < b1 ? i : i < b2 ? i - b1 : i - b2;
    const uint4 *row = reinterpret_cast<const uint4 *>(M + (long long)r * cols);
    __shared__ uint4 s_q[256];
    const uint16_t *s_c = reinterpret_cast<const uint16_t *>(s_q);
    const int n8 = cols / 8, tid = threadIdx.x;
    float s = 0.f;
    uint4 next = tid < n8 ? row[tid] : make_uint4(0u, 0u, 0u, 0u);
    for (int q0 = 0; q0 < n8; q0 += 256) {
        s_q[tid] = next;
        __syncthreads();
        const int q = q0 + 256 + tid;
        next = q < n8 ? row[q] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (8 * q0 + 256 * i + tid < cols) s += __uint_as_float((uint32_t)s_c[256 * i + tid] << 16);
        __syncthreads();
    }
    const float t = block_sum_256(s);
    if (tid == 0) out[r] += t;
}

// The splits' products of the three weight gradients, added in split order with the rounding
// errors kept beside the sums (two floats), so that only the last rounding is left of them: two
// consecutive elements per thread with ten loads in flight, or, where up to 64 splits would make
// a long chain of loads (W2, W3), four threads that take every fourth split and add their shares
// in a fixed tree.  Then the bias rows and the loss (the head's block shares, in order) in the same
// launch.  Bound by the latency and the L2 traffic of 25 MB of partials: 11.6 us at 16384 rows (four
// elements per thread 15.6, one 14.4; the bias rows alone 6.7), 8.3 at 2560; the head and the dW3
// product got 3.5 us faster without their atomics.
struct SplitSums {
    const float *part[3];  // [splits][n]
    float *out[3];
    int n[3], splits[3], lanes[3];  // n: multiples of 512; lanes: threads per two elements (1 or 4)
    const float *loss_part;
    int n_loss;
    float *loss;
    __host__ __device__ int blocks(int k) const { return n[k] / 512 * lanes[k]; }
};
__global__ void __launch_bounds__(256) gradient_sums_kernel(RowSums a, int cols, SplitSums g) {
    pdl_begin();
    constexpr int kBatch = 10;
    int blk = blockIdx.x;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (blk >= 0 && blk < g.blocks(k)) {
            const int lanes = g.lanes[k], t = blk * 256 + (int)threadIdx.x, i = t / lanes, sub = t % lanes;
            const int n2 = g.n[k] / 2, splits = g.splits[k];
            const float2 *p = reinterpret_cast<const float2 *>(g.part[k]) + i;
            float hi[2] = {0.f, 0.f}, lo[2] = {0.f, 0.f};
            auto add = [&](int c, float h, float l) {
                const DF s = two_sum(hi[c], h);
                hi[c] = s.hi;
                lo[c] += s.lo + l;
            };
            for (int s0 = sub; s0 < splits; s0 += kBatch * lanes) {
                float2 q[kBatch];
#pragma unroll
                for (int j = 0; j < kBatch; ++j) {
                    const int s = s0 + j * lanes;
                    q[j] = s < splits ? p[(size_t)s * n2] : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int j = 0; j < kBatch; ++j) {
                    add(0, q[j].x, 0.f);
                    add(1, q[j].y, 0.f);
                }
            }
            for (int o = 1; o < lanes; o <<= 1)
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    add(c, __shfl_xor_sync(SG_FULL_MASK, hi[c], o), __shfl_xor_sync(SG_FULL_MASK, lo[c], o));
            if (sub == 0) {
                float *o = g.out[k] + 2 * (size_t)i;
#pragma unroll
                for (int c = 0; c < 2; ++c) o[c] += isfinite(hi[c]) ? hi[c] + lo[c] : hi[c];  // (inf has no error term)
            }
            return;
        }
        blk -= g.blocks(k);
    }
    if (blk < a.rows[0] + a.rows[1] + a.rows[2]) {
        row_sum(a, cols, blk);
        return;
    }
    if (!g.loss) return;
    float s = 0.f;
    for (int i = threadIdx.x; i < g.n_loss; i += 256) s += g.loss_part[i];
    const float t = block_sum_256(s);
    if (threadIdx.x == 0) *g.loss += t;
}

}  // namespace sg

using namespace sg;

#define MLP_REQUIRE(cond, ...)         \
    do {                               \
        if (!(cond)) {                 \
            set_error(__VA_ARGS__);    \
            return SG_ERR_INVALID_ARG; \
        }                              \
    } while (0)
#define MLP_TRY(expr)                 \
    do {                              \
        const sg_status _s = (expr);  \
        if (_s != SG_OK) return _s;   \
    } while (0)

// Layout of the ordered backward's workspace (floats): the splits' products of W1, W2 and W3 and
// the loss shares, each a multiple of 1024 floats.
struct GradWorkspace {
    int splits[3];
    size_t at[3], loss, total;
};
static const int kGradN[3] = {SG_MLP_HIDDEN * SG_MLP_IN, SG_MLP_HIDDEN * SG_MLP_HIDDEN, SG_MLP_OUT *SG_MLP_HIDDEN};
static GradWorkspace grad_workspace(int B) {
    GradWorkspace w;
    const int N[3] = {SG_MLP_IN, SG_MLP_HIDDEN, SG_MLP_OUT};
    size_t off = 0;
    for (int k = 0; k < 3; ++k) {
        int per;
        w.splits[k] = split_count(SG_MLP_HIDDEN, N[k], B, kMaxSplits, per);
        w.at[k] = off;
        off += (size_t)w.splits[k] * kGradN[k];
    }
    w.loss = off;
    w.total = off + (size_t)((B / 64 + 1023) / 1024) * 1024;
    return w;
}

// ws: NULL, or grad_workspace(B).total floats.
static sg_status mlp_backward(const sg_mlp *net, const uint16_t *Xt, const float *target, const float *out_weight,
                              int32_t B, sg_mlp_acts *acts, sg_mlp_grads *grads, float *loss, float *ws,
                              uint32_t *status, cudaStream_t st) {
    MLP_REQUIRE(net && Xt && target && out_weight && acts && grads && loss, "mlp_backward: NULL argument");
    MLP_REQUIRE(acts->H1t && acts->H2t && acts->dY && acts->dYt && acts->dH2 && acts->dH2t && acts->dH1t,
                "mlp_backward: activation buffers are NULL");
    MLP_REQUIRE(grads->W1 && grads->W2 && grads->W3 && grads->b1 && grads->b2 && grads->b3,
                "mlp_backward: gradient buffers are NULL");
    MLP_REQUIRE(B > 0 && B % 128 == 0, "mlp_backward: B = %d must be a positive multiple of 128", B);
    const int H = SG_MLP_HIDDEN, O = SG_MLP_OUT;
    GradWorkspace w{};
    if (ws) w = grad_workspace(B);
    float *const out[3] = {grads->W1, grads->W2, grads->W3};
    // weight gradient k: atomically added, or the splits' products into the workspace
    auto to_grad = [&](tc::GemmParams &p, int k, long long ld, int transposed) {
        p.out_f32 = ws ? ws + w.at[k] : out[k];
        p.ld_f32 = ld;
        p.f32_transposed = transposed;
        p.f32_atomic = ws ? 0 : 1;
        p.split_stride = ws ? kGradN[k] : 0;
    };
    launch_pdl(mse_head_kernel, B / 64, 256, 0, st, acts->Y, target, out_weight, B, (bf16 *)acts->dY, (bf16 *)acts->dYt,
               loss, ws ? ws + w.loss : (float *)nullptr, (((uintptr_t)acts->Y | (uintptr_t)target) & 15) == 0);
    count_launches(1);
    // dW3 [32][128] += (H2^T dY)^T
    tc::GemmParams p = gemm_params((const bf16 *)acts->H2t, B, (const bf16 *)acts->dYt, B, H, O, B, status);
    to_grad(p, 2, H, 1);
    MLP_TRY(launch_gemm(p, st));
    // dH2 = (dY W3) * [H2 > 0]
    p = gemm_params((const bf16 *)acts->dY, 64, (const bf16 *)net->W3t, 64, B, H, 64, status);
    p.mask = (const bf16 *)acts->H2; p.ldmask = H;
    p.out_bf16 = (bf16 *)acts->dH2; p.ld_bf16 = H;
    p.out_bf16_t = (bf16 *)acts->dH2t; p.ld_bf16_t = B;
    MLP_TRY(launch_gemm(p, st));
    // dW2 [128][128] += (H1^T dH2)^T
    p = gemm_params((const bf16 *)acts->H1t, B, (const bf16 *)acts->dH2t, B, H, H, B, status);
    to_grad(p, 1, H, 1);
    MLP_TRY(launch_gemm(p, st));
    // dH1 = (dH2 W2) * [H1 > 0], transposed copy only
    p = gemm_params((const bf16 *)acts->dH2, H, (const bf16 *)net->W2t, H, B, H, H, status);
    p.mask = (const bf16 *)acts->H1; p.ldmask = H;
    p.out_bf16_t = (bf16 *)acts->dH1t; p.ld_bf16_t = B;
    MLP_TRY(launch_gemm(p, st));
    // dW1 [128][2048] += dH1^T X
    p = gemm_params((const bf16 *)acts->dH1t, B, (const bf16 *)Xt, B, H, SG_MLP_IN, B, status);
    to_grad(p, 0, SG_MLP_IN, 0);
    MLP_TRY(launch_gemm(p, st));
    // bias gradients: row sums of the transposed copies; with a workspace also the splits' sums
    const RowSums rs{{(const bf16 *)acts->dYt, (const bf16 *)acts->dH2t, (const bf16 *)acts->dH1t},
                     {grads->b3, grads->b2, grads->b1},
                     {O, H, H}};
    SplitSums ss{};
    int blocks = O + 2 * H;
    if (ws) {
        for (int k = 0; k < 3; ++k) {
            ss.part[k] = ws + w.at[k];
            ss.out[k] = out[k];
            ss.n[k] = kGradN[k];
            ss.splits[k] = w.splits[k];
            ss.lanes[k] = k == 0 ? 1 : 4;
            blocks += ss.blocks(k);
        }
        ss.loss_part = ws + w.loss;
        ss.n_loss = B / 64;
        ss.loss = loss;
        blocks += 1;
    }
    launch_pdl(gradient_sums_kernel, blocks, 256, 0, st, rs, B, ss);
    count_launches(1);
    return check_launch("mlp_backward");
}

extern "C" {

sg_status sg_gemm_bf16(const uint16_t *A, int64_t lda, const uint16_t *B, int64_t ldb, int32_t M, int32_t N,
                       int32_t K, float *D, int64_t ldd, int32_t accumulate, uint32_t *status,
                       sg_stream_t stream) {
    MLP_REQUIRE(A && B && D, "gemm: NULL operand");
    MLP_REQUIRE(M > 0 && N > 0 && K > 0 && K % 64 == 0, "gemm: need M, N > 0 and K %% 64 == 0");
    MLP_REQUIRE(lda % 8 == 0 && ldb % 8 == 0 && ((uintptr_t)A & 15) == 0 && ((uintptr_t)B & 15) == 0,
                "gemm: operands need 16-byte aligned rows");
    tc::GemmParams p = gemm_params((const bf16 *)A, lda, (const bf16 *)B, ldb, M, N, K, status);
    p.out_f32 = D;
    p.ld_f32 = ldd;
    p.f32_atomic = accumulate ? 1 : 0;
    return launch_gemm(p, (cudaStream_t)stream);
}

sg_status sg_gemm_bf16_timeout_probe(const uint16_t *A, int64_t lda, const uint16_t *B, int64_t ldb, int32_t M,
                                     int32_t N, int32_t K, float *D, int64_t ldd, uint32_t polls,
                                     uint32_t *status, sg_stream_t stream) {
    MLP_REQUIRE(A && B && D, "gemm: NULL operand");
    MLP_REQUIRE(M > 0 && N > 0 && K > 0 && K % 64 == 0, "gemm: need M, N > 0 and K %% 64 == 0");
    MLP_REQUIRE(lda % 8 == 0 && ldb % 8 == 0 && ((uintptr_t)A & 15) == 0 && ((uintptr_t)B & 15) == 0,
                "gemm: operands need 16-byte aligned rows");
    MLP_REQUIRE(polls >= 1 && polls <= (1u << 20), "timeout probe: polls must be in [1, 2^20]");
    tc::GemmParams p = gemm_params((const bf16 *)A, lda, (const bf16 *)B, ldb, M, N, K, status);
    p.out_f32 = D;
    p.ld_f32 = ldd;
    p.probe_polls = polls;
    return launch_gemm(p, (cudaStream_t)stream);
}

sg_status sg_mlp_pack_weights(const float *W1, const float *W2, const float *W3, uint16_t *W1b, uint16_t *W2b,
                              uint16_t *W3b, uint16_t *W2t, uint16_t *W3t, sg_stream_t stream) {
    MLP_REQUIRE(W1 && W2 && W3 && W1b && W2b && W3b && W2t && W3t, "pack_weights: NULL argument");
    cudaStream_t st = (cudaStream_t)stream;
    const int n = SG_MLP_HIDDEN * (SG_MLP_IN + SG_MLP_HIDDEN + SG_MLP_OUT);
    launch_pdl(pack_weights_kernel, (n + 255) / 256, 256, 0, st, W1, W2, W3, (bf16 *)W1b, (bf16 *)W2b, (bf16 *)W3b,
               (bf16 *)W2t, (bf16 *)W3t);
    count_launches(1);
    return check_launch("mlp_pack_weights");
}

sg_status sg_mlp_forward(const sg_mlp *net, const uint16_t *X, int32_t B, sg_mlp_acts *acts, uint32_t *status,
                         sg_stream_t stream) {
    MLP_REQUIRE(net && X && acts && acts->H1 && acts->H2 && acts->Y, "mlp_forward: NULL argument");
    MLP_REQUIRE(B > 0 && B % 128 == 0, "mlp_forward: B = %d must be a positive multiple of 128", B);
    cudaStream_t st = (cudaStream_t)stream;
    const int H = SG_MLP_HIDDEN;
    tc::GemmParams p = gemm_params((const bf16 *)X, SG_MLP_IN, (const bf16 *)net->W1, SG_MLP_IN, B, H, SG_MLP_IN,
                                   status);
    p.bias = net->b1; p.relu = 1;
    p.out_bf16 = (bf16 *)acts->H1; p.ld_bf16 = H;
    p.out_bf16_t = (bf16 *)acts->H1t; p.ld_bf16_t = B;
    MLP_TRY(launch_gemm(p, st));
    p = gemm_params((const bf16 *)acts->H1, H, (const bf16 *)net->W2, H, B, H, H, status);
    p.bias = net->b2; p.relu = 1;
    p.out_bf16 = (bf16 *)acts->H2; p.ld_bf16 = H;
    p.out_bf16_t = (bf16 *)acts->H2t; p.ld_bf16_t = B;
    MLP_TRY(launch_gemm(p, st));
    p = gemm_params((const bf16 *)acts->H2, H, (const bf16 *)net->W3, H, B, SG_MLP_OUT, H, status);
    p.bias = net->b3;
    p.out_f32 = acts->Y; p.ld_f32 = SG_MLP_OUT;
    return launch_gemm(p, st);
}

sg_status sg_mlp_backward(const sg_mlp *net, const uint16_t *Xt, const float *target, const float *out_weight,
                          int32_t B, sg_mlp_acts *acts, sg_mlp_grads *grads, float *loss, uint32_t *status,
                          sg_stream_t stream) {
    return mlp_backward(net, Xt, target, out_weight, B, acts, grads, loss, nullptr, status, (cudaStream_t)stream);
}

size_t sg_mlp_backward_workspace_size(int32_t B) {
    return B > 0 && B % 128 == 0 ? grad_workspace(B).total * sizeof(float) : 0;
}

sg_status sg_mlp_backward_ordered(const sg_mlp *net, const uint16_t *Xt, const float *target,
                                  const float *out_weight, int32_t B, sg_mlp_acts *acts, sg_mlp_grads *grads,
                                  float *loss, void *workspace, size_t workspace_bytes, uint32_t *status,
                                  sg_stream_t stream) {
    MLP_REQUIRE(B > 0 && B % 128 == 0, "mlp_backward: B = %d must be a positive multiple of 128", B);
    MLP_REQUIRE(workspace && ((uintptr_t)workspace & 15) == 0, "mlp_backward: workspace is NULL or not 16-byte aligned");
    const size_t need = sg_mlp_backward_workspace_size(B);
    if (workspace_bytes < need) {
        set_error("mlp_backward: workspace %zu bytes < %zu needed", workspace_bytes, need);
        return SG_ERR_CAPACITY;
    }
    return mlp_backward(net, Xt, target, out_weight, B, acts, grads, loss, (float *)workspace, status,
                        (cudaStream_t)stream);
}

}  // extern "C"
