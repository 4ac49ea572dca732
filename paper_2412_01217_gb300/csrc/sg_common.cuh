// sg_common.cuh -- device helpers shared by the sm_103a kernels of the pyramid splatting
// library.  Nothing here is shared with the CPU oracle.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "../../include/sg.h"

#define SG_FULL_MASK 0xffffffffu

namespace sg {

// Largest tile: 32x8 or 16x16 pixels = 256 threads per CTA.
constexpr int kMaxTileThreads = 256;

struct Float3 {
    float x, y, z;
};

// ----------------------------------------------------------------------------------------
// alpha of one Gaussian at one pixel (Eq. 3 with the anisotropic 2D covariance S).  The
// exponent sigma = 1/2 d^T S^{-1} d is evaluated in its conditional (Schur complement)
// form  sigma = (m00 dx)^2 + (m10 dx + m11 dy)^2  with m00 = 1/sqrt(2 s00),
// m10 = -s01/sqrt(2 s00 det), m11 = sqrt(s00/(2 det)): a sum of squares, so no
// cancellation for elongated footprints, and 7 flops.  The forward and backward kernels
// must take bit-identical skip/stop decisions, so every rounding step is spelled out with
// _rn intrinsics (no compiler contraction can differ between kernels).  The 2D mean is an
// integer (ui, vi) plus a float fraction (uf, vf): (px - ui) is exact in float and
// dx = (px - ui) - uf is the correctly rounded offset, whatever the tile.
// ----------------------------------------------------------------------------------------

// 2^x, approximate (results below the normal range flush to 0)
__device__ __forceinline__ float ex2_fast(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(r) : "f"(x));
    return r;
}

// alpha from dx, q = m11 dy and (m00 dx)^2, each rounded as above; 0 below alpha_min.
// exp(-sigma) = 2^(-sigma log2 e).  (A non-finite sigma gives no alpha: the comparison fails.)
__device__ __forceinline__ float entry_alpha(float m10, float dx, float q, float p1_sq, float o, float alpha_max,
                                             float alpha_min) {
    const float p2 = __fmaf_rn(m10, dx, q);
    const float sigma = __fmaf_rn(p2, p2, p1_sq);
    const float raw = __fmul_rn(o, ex2_fast(__fmul_rn(sigma, -1.4426950408889634f)));
    return raw >= alpha_min ? fminf(alpha_max, raw) : 0.f;
}

// ---- double-float (unevaluated sum hi + lo of two floats) helpers --------------------
struct DF {
    float hi, lo;
};
__device__ __forceinline__ DF two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
__device__ __forceinline__ DF two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ DF df_add(DF a, DF b) {
    DF s = two_sum(a.hi, b.hi);
    s.lo = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
    return two_sum(s.hi, s.lo);
}
__device__ __forceinline__ DF df_add_f(DF a, float b) {
    DF s = two_sum(a.hi, b);
    s.lo = __fadd_rn(s.lo, a.lo);
    return two_sum(s.hi, s.lo);
}
// (a.hi + a.lo) * f, f a float
__device__ __forceinline__ DF df_mul_f(DF a, float f) {
    DF p = two_prod(a.hi, f);
    p.lo = __fmaf_rn(a.lo, f, p.lo);
    return two_sum(p.hi, p.lo);
}
// a / b for double-floats (one Newton-style correction of the float quotient)
__device__ __forceinline__ DF df_div(DF a, DF b) {
    const float q0 = __fdiv_rn(a.hi, b.hi);
    const DF p = two_prod(q0, b.hi);
    float r = __fsub_rn(a.hi, p.hi);
    r = __fsub_rn(r, p.lo);
    r = __fadd_rn(r, a.lo);
    r = __fmaf_rn(-q0, b.lo, r);
    const float q1 = __fdiv_rn(r, b.hi);
    return two_sum(q0, q1);
}

// a*b - c*d with one rounding error (Kahan's algorithm with FMA).
__device__ __forceinline__ float diff_of_products(float a, float b, float c, float d) {
    const float w = c * d;
    const float err = __fmaf_rn(-c, d, w);
    const float dop = __fmaf_rn(a, b, -w);
    return dop + err;
}

// ----------------------------------------------------------------------------------------
// TF32 tensor-core products with FP32-level accuracy: x = hi + lo with hi = x with its 13
// low mantissa bits cleared and lo = x - hi (exact); a*b ~ hi*hi + hi*lo + lo*hi keeps about
// 22 mantissa bits of every product (the dropped lo*lo term is below 2^-22 relative).
// mma.m16n8k8 fragments (gid = lane / 4, tig = lane % 4):
//   A (16 x 8): a0 (gid, tig), a1 (gid + 8, tig), a2 (gid, tig + 4), a3 (gid + 8, tig + 4)
//   B (8 x 8):  b0 (tig, gid), b1 (tig + 4, gid)
//   D (16 x 8): d0 (gid, 2 tig), d1 (gid, 2 tig + 1), d2 (gid + 8, 2 tig), d3 (gid + 8, 2 tig + 1)
// ----------------------------------------------------------------------------------------
__device__ __forceinline__ void split_tf32(float x, uint32_t &hi, uint32_t &lo) {
    const uint32_t h = __float_as_uint(x) & 0xffffe000u;
    hi = h;
    lo = __float_as_uint(x - __uint_as_float(h));
}

// (no side effects: not volatile, so the compiler may schedule other work around it)
__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// a * b with both split (3 MMAs, small terms first)
__device__ __forceinline__ void mma_tf32x3(float (&d)[4], const uint32_t (&ah)[4], const uint32_t (&al)[4],
                                           uint32_t bh0, uint32_t bh1, uint32_t bl0, uint32_t bl1) {
    mma_tf32(d, al, bh0, bh1);
    mma_tf32(d, ah, bl0, bl1);
    mma_tf32(d, ah, bh0, bh1);
}

// The same with four-deep operands (m16n8k4): A (16 x 4) a0 (gid, tig), a1 (gid + 8, tig);
// B (4 x 8) b0 (tig, gid).
__device__ __forceinline__ void mma_tf32_k4(float (&d)[4], const uint32_t (&a)[2], uint32_t b) {
    asm(
        "mma.sync.aligned.m16n8k4.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(b));
}
__device__ __forceinline__ void mma_tf32x3_k4(float (&d)[4], const uint32_t (&ah)[2], const uint32_t (&al)[2],
                                              uint32_t bh, uint32_t bl) {
    mma_tf32_k4(d, al, bh);
    mma_tf32_k4(d, ah, bl);
    mma_tf32_k4(d, ah, bh);
}

// 32-bit operand tiles through ldmatrix: an 8 x 4 tile of 32-bit words is an 8 x 8 tile of
// 16-bit halves, and thread t receives the word at row t / 4, column t % 4 of each tile, the
// (gid, tig) element of the fragments above.  Lane 8 m + i gives the (16-byte aligned)
// address of row i of tile m.
__device__ __forceinline__ void ldsm_x2(const float *p, uint32_t &r0, uint32_t &r1) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm_x4(const float *p, uint32_t (&r)[4]) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}

// Asynchronous copies global -> shared (4 bytes, zero-filled when !valid while src must still
// be a mapped address; 16 bytes, both sides 16-byte aligned) and their group fences.
__device__ __forceinline__ void cp_async4(void *dst, const void *src, bool valid) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit_group() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>  // waits until at most the N latest groups are pending
__device__ __forceinline__ void cp_async_wait_groups() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// 1 / x, approximate (x normal; 1 ulp, exact for 1)
__device__ __forceinline__ float rcp_fast(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;\n" : "=f"(r) : "f"(x));
    return r;
}

// Two float additions to consecutive, 8-byte aligned addresses in one vector reduction.
__device__ __forceinline__ void red_add_v2(float *addr, float a, float b) {
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};\n" ::"l"(addr), "f"(a), "f"(b) : "memory");
}

// Four float additions to consecutive, 16-byte aligned addresses in one vector reduction.
__device__ __forceinline__ void red_add_v4(float *addr, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d)
                 : "memory");
}

// ----------------------------------------------------------------------------------------
// Programmatic dependent launch.  The kernels of one iteration are launched with
// launch_pdl() (programmatic stream serialisation), and every kernel starts with
// pdl_begin(): griddepcontrol.wait, which returns once the grids it depends on have completed
// and their writes are visible (at once when the launch has no such dependency).  Nothing
// before it touches global memory, so the ordering is that of plain stream order; the
// launch of each kernel is prepared while its predecessor runs.  (Letting dependents start
// early with griddepcontrol.launch_dependents was measured slower: their waiting blocks take
// SM slots from the running kernel.)
// ----------------------------------------------------------------------------------------
__device__ __forceinline__ void pdl_begin() {
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

template <typename... KArgs, typename... Args>
inline void launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

__device__ __forceinline__ int find_view(const sg_view *views, int n_views, int tile) {
    int lo = 0, hi = n_views - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (views[mid].tile_offset <= tile) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Sets `bit` in *status when `bad` holds for any active lane of the warp (one atomic per
// warp).  Safe in divergent code: only the lanes that reach it take part.
__device__ __forceinline__ void flag_status(bool bad, uint32_t *status, uint32_t bit) {
    const uint32_t m = __ballot_sync(__activemask(), bad);
    if (m && (threadIdx.x & 31) == (uint32_t)(__ffs(m) - 1)) atomicOr(status, bit);
}

__device__ __forceinline__ uint32_t pack16(int a, int b) {
    return (uint32_t)a | ((uint32_t)b << 16);
}

}  // namespace sg

// Internal launch helpers (defined in api.cu / the kernel files).
namespace sg {
void set_error(const char *fmt, ...);
void count_launches(int n);  // kernel launches issued by the library (diagnostics)
sg_status check_launch(const char *what);
}  // namespace sg
