// init.cu -- insertion of new Gaussians from a keyframe (Sec. III-A: the mapping thread
// converts keyframe data into Gaussian primitives with position, colour, semantics, depth
// and opacity) and the patch features of the learned initializer.
//
// Heuristic initializer, per inserted pixel (x, y) with valid depth D at level 0:
//   mean = back-projection of (x, y, D); rgb = pixel colour; log-scale = ln(D / fx) on all
//   three axes (a one-pixel footprint, Eq. 2's r2D = f r / d = 1); quaternion = identity;
//   opacity logit = 0 (opacity 0.5); semantic feature = kappa * code[label] (or 0).
// Patch features, per inserted pixel: the 7x7 neighbourhood, 41 channels per pixel:
//   rgb (3), depth in metres (1), one-hot label (32), unit ray direction in the camera frame
//   (3), depth-valid flag (1), 1/fx (1) -- 49 * 41 = 2009 features, zero-padded to 2048.
//   Pixels outside the image contribute zeros.
#include <cuda_bf16.h>

#include "sg_common.cuh"

namespace sg {

constexpr int kPatch = 7, kPatchCh = 41, kPatchFeat = kPatch * kPatch * kPatchCh;  // 2009
static_assert(kPatchFeat <= SG_MLP_IN, "patch features exceed the MLP input");

struct Frame {
    const float *rgb, *depth;
    const int *label;
    int W, H;
    float fx, fy, cx, cy;
};

// Patch features of ROWS pixels per block, into X [B_pad][2048] and/or Xt [2048][B_pad]
// (rows from B on are zero).  The 49 x 9 values of each pixel's patch (label channels aside) are
// formed once and kept in shared memory as bf16 next to the labels; features are then written
// 8 at a time (X: one 16-byte store per thread, a row per pass of the block; Xt: 16 rows of the
// batch, 32 bytes, per half warp).  One thread per element formed every feature from the images
// again, with two integer divisions each (5120 rows into X: 50 us).  X alone takes 4 rows per
// block, so that the gathers of 1280 blocks overlap (16 rows per block: 19 us).
constexpr int kPatchVals = 9;  // rgb, depth, ray, valid, 1/fx
template <int ROWS>
__global__ void __launch_bounds__(256) patch_kernel(Frame fr, const int2 *__restrict__ pix, int B, int B_pad,
                                                    uint16_t *__restrict__ X, uint16_t *__restrict__ Xt, bool vec) {
    pdl_begin();
    constexpr int NP = kPatch * kPatch;
    __shared__ uint16_t s_v[ROWS][NP][kPatchVals];
    __shared__ int s_lab[ROWS][NP];
    const int b0 = blockIdx.x * ROWS;
    const size_t HW = (size_t)fr.W * fr.H;
    auto bits = [](float v) { return __bfloat16_as_ushort(__float2bfloat16_rn(v)); };
    for (int i = threadIdx.x; i < ROWS * NP; i += 256) {
        const int r = i / NP, k = i % NP, b = b0 + r;
        float v[kPatchVals];
#pragma unroll
        for (int c = 0; c < kPatchVals; ++c) v[c] = 0.f;
        int lab = -1;
        if (b < B) {
            const int2 q = pix[b];
            const int x = q.x + k % kPatch - kPatch / 2, y = q.y + k / kPatch - kPatch / 2;
            if (!(x < 0 || y < 0 || x >= fr.W || y >= fr.H)) {
                const size_t p = (size_t)y * fr.W + x;
#pragma unroll
                for (int c = 0; c < 3; ++c) v[c] = fr.rgb[c * HW + p];
                const float d = fr.depth[p];
                v[3] = d > 0.f ? d : 0.f;
                if (fr.label) lab = fr.label[p];
                const float rx = (x - fr.cx) / fr.fx, ry = (y - fr.cy) / fr.fy;
                const float inv = rsqrtf(rx * rx + ry * ry + 1.f);
                v[4] = rx * inv;
                v[5] = ry * inv;
                v[6] = inv;
                v[7] = d > 0.f ? 1.f : 0.f;
                v[8] = 1.f / fr.fx;
            }
        }
#pragma unroll
        for (int c = 0; c < kPatchVals; ++c) s_v[r][k][c] = bits(v[c]);
        s_lab[r][k] = lab;
    }
    __syncthreads();
    const uint16_t one = bits(1.f);
    // channel f % 41: rgb, depth, 32 label channels, ray, valid, 1/fx; features from 2009 on are 0
    auto feature = [&](int r, int k, int ch) -> uint32_t {
        if (ch < 4) return s_v[r][k][ch];
        if (ch < 36) return s_lab[r][k] == ch - 4 ? one : 0;
        return s_v[r][k][ch - 32];
    };
    if (X) {
        const int f0 = threadIdx.x * 8;  // 256 x 8 = 2048 features
        for (int r = 0; r < ROWS; ++r) {
            int k = f0 / kPatchCh, ch = f0 % kPatchCh;
            uint32_t h[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                h[j] = f0 + j < kPatchFeat ? feature(r, k, ch) : 0u;
                if (++ch == kPatchCh) {
                    ch = 0;
                    ++k;
                }
            }
            uint16_t *o = X + (size_t)(b0 + r) * SG_MLP_IN + f0;
            if (vec) {
                *reinterpret_cast<uint4 *>(o) =
                    make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) o[j] = (uint16_t)h[j];
            }
        }
    }
    if (Xt) {
        const int r = threadIdx.x % ROWS;
        for (int f = threadIdx.x / ROWS; f < SG_MLP_IN; f += 256 / ROWS)
            Xt[(size_t)f * B_pad + b0 + r] = f < kPatchFeat ? (uint16_t)feature(r, f / kPatchCh, f % kPatchCh) : 0;
    }
}

struct InitOut {
    float *mean, *log_scale, *quat, *opacity_logit, *rgb, *sem;
};

__global__ void heuristic_init_kernel(Frame fr, sg_camera cam, const int2 *__restrict__ pix, int B, int C,
                                      const float *__restrict__ code, int n_classes, float kappa, InitOut o) {
    pdl_begin();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const int2 q = pix[b];
    const size_t p = (size_t)q.y * fr.W + q.x, HW = (size_t)fr.W * fr.H;
    float D = fr.depth[p];
    if (!(D > 0.f)) D = 1.f;  // callers insert valid-depth pixels; keep the state finite
    // camera-frame point, then world = R_cw^T (t - t_cw)
    const float xc = (q.x - cam.cx) / cam.fx * D, yc = (q.y - cam.cy) / cam.fy * D, zc = D;
    const float dx = xc - cam.t_cw[0], dy = yc - cam.t_cw[1], dz = zc - cam.t_cw[2];
    const float *R = cam.R_cw;
    o.mean[3 * b + 0] = R[0] * dx + R[3] * dy + R[6] * dz;
    o.mean[3 * b + 1] = R[1] * dx + R[4] * dy + R[7] * dz;
    o.mean[3 * b + 2] = R[2] * dx + R[5] * dy + R[8] * dz;
    const float ls = logf(D / cam.fx);
    o.log_scale[3 * b + 0] = ls;
    o.log_scale[3 * b + 1] = ls;
    o.log_scale[3 * b + 2] = ls;
    o.quat[4 * b + 0] = 1.f;
    o.quat[4 * b + 1] = 0.f;
    o.quat[4 * b + 2] = 0.f;
    o.quat[4 * b + 3] = 0.f;
    o.opacity_logit[b] = 0.f;
    for (int c = 0; c < 3; ++c) o.rgb[3 * b + c] = fr.rgb[c * HW + p];
    const int lab = fr.label ? fr.label[p] : -1;
    for (int c = 0; c < C; ++c)
        o.sem[(size_t)C * b + c] = (code && lab >= 0 && lab < n_classes) ? kappa * code[(size_t)lab * C + c] : 0.f;
}

// MLP output (standardised) -> log-scale (3), opacity logit (1), semantic feature (C)
__global__ void apply_mlp_kernel(const float *__restrict__ Y, int B, int C, const float *__restrict__ mu,
                                 const float *__restrict__ sd, float *__restrict__ log_scale,
                                 float *__restrict__ opacity_logit, float *__restrict__ sem) {
    pdl_begin();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const float *y = Y + (size_t)b * SG_MLP_OUT;
    for (int k = 0; k < 3; ++k) log_scale[3 * b + k] = y[k] * sd[k] + mu[k];
    opacity_logit[b] = y[3] * sd[3] + mu[3];
    for (int c = 0; c < C && 4 + c < SG_MLP_OUT; ++c) sem[(size_t)C * b + c] = y[4 + c] * sd[4 + c] + mu[4 + c];
}

}  // namespace sg

using namespace sg;

extern "C" {

sg_status sg_extract_patches(const float *rgb, const float *depth, const int32_t *label, const sg_camera *cam,
                             const int32_t *pixels, int32_t B, int32_t B_pad, uint16_t *X, uint16_t *Xt,
                             sg_stream_t stream) {
    if (!rgb || !depth || !cam || !pixels || (!X && !Xt) || B < 0 || B_pad < B || B_pad % 128 != 0) {
        set_error("extract_patches: bad argument (B=%d, B_pad=%d must be a multiple of 128 >= B)", B, B_pad);
        return SG_ERR_INVALID_ARG;
    }
    Frame fr{rgb, depth, label, cam->W, cam->H, cam->fx, cam->fy, cam->cx, cam->cy};
    cudaStream_t st = (cudaStream_t)stream;
    if (B_pad > 0) {
        launch_pdl(Xt ? patch_kernel<16> : patch_kernel<4>, B_pad / (Xt ? 16 : 4), 256, 0, st, fr, (const int2 *)pixels, B,
                   B_pad, X, Xt, ((uintptr_t)X & 15) == 0);
        count_launches(1);
    }
    return check_launch("extract_patches");
}

sg_status sg_init_gaussians(const float *rgb, const float *depth, const int32_t *label, const sg_camera *cam,
                            const int32_t *pixels, int32_t B, const float *sem_code, int32_t n_classes,
                            float kappa, sg_gaussian_grads *out, sg_stream_t stream) {
    if (!rgb || !depth || !cam || !pixels || !out || B < 0 || !out->mean || !out->log_scale || !out->quat ||
        !out->opacity_logit || !out->rgb || !out->sem) {
        set_error("init_gaussians: NULL argument");
        return SG_ERR_INVALID_ARG;
    }
    if (B == 0) return SG_OK;
    Frame fr{rgb, depth, label, cam->W, cam->H, cam->fx, cam->fy, cam->cx, cam->cy};
    InitOut o{out->mean, out->log_scale, out->quat, out->opacity_logit, out->rgb, out->sem};
    launch_pdl(heuristic_init_kernel, (B + 127) / 128, 128, 0, (cudaStream_t)stream, fr, *cam, (const int2 *)pixels, B,
               out->C, sem_code, n_classes, kappa, o);
    count_launches(1);
    return check_launch("init_gaussians");
}

sg_status sg_apply_mlp_init(const float *Y, int32_t B, const float *y_mean, const float *y_std,
                            sg_gaussian_grads *out, sg_stream_t stream) {
    if (!Y || !y_mean || !y_std || !out || !out->log_scale || !out->opacity_logit || !out->sem || B < 0) {
        set_error("apply_mlp_init: NULL argument");
        return SG_ERR_INVALID_ARG;
    }
    if (B == 0) return SG_OK;
    launch_pdl(apply_mlp_kernel, (B + 127) / 128, 128, 0, (cudaStream_t)stream, Y, B, out->C, y_mean, y_std,
               out->log_scale, out->opacity_logit, out->sem);
    count_launches(1);
    return check_launch("apply_mlp_init");
}

}  // extern "C"
