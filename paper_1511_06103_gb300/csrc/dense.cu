// dense.cu -- fully connected CRF with a Gaussian appearance kernel
// (the dense segmentation model of Sec. 4.2), FP32 CUDA-core form.
//
// The pairwise weights are K_ij = exp(-|p_i-p_j|^2/(2 theta_pos^2)
// - |c_i-c_j|^2/(2 theta_rgb^2)) for i != j over (x, y, r, g, b) features, each
// unordered pair counted once, with one symmetric label matrix mu.  One step:
//   a1  S = K Q (N x N times N x L), m_i = mu S_i
//   a2  g_i = U_i + m_i
//   a3  a_i = -eta g_i + (1 - eta) log q_i
//   a4  log q'_i = a_i - logsumexp(a_i)
//   a5  F = sum_i q_i . (U_i + m_i / 2 + log q_i)
//
// This file builds what the steps read: K, materialised once per model (FP32
// rows of dense_k32_pitch(N) floats for the FP32 step in dense_f32.cu, BF16
// blocks for the tensor-core step in dense_tc.cu), the column features of the
// step that computes K itself, and the copies of q.
#include <cmath>

#include "dense_common.cuh"
#include "f32x2.cuh"
#include "internal.h"

namespace proxmf {

namespace {

// ---------------------------------------------------------------- K build --

// K[b][i][j] from features [b][N][5], zero on the diagonal and past column N.
// K_ij and K_ji are the same bits: the differences only change sign and are
// squared.  The FP32 step relies on it (it reads row k for column k).
__global__ void dense_kernel_build_kernel(const float *__restrict__ feats, float *__restrict__ K, int N, int pitch,
                                          float inv2p, float inv2c) {
    const int b = blockIdx.z;
    const int i = blockIdx.y;
    const float *f = feats + (size_t)b * N * 5;
    const float xi = f[i * 5 + 0], yi = f[i * 5 + 1], ri = f[i * 5 + 2], gi = f[i * 5 + 3], bi = f[i * 5 + 4];
    float *row = K + ((size_t)b * N + i) * pitch;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < pitch; j += gridDim.x * blockDim.x) {
        if (j >= N) {
            row[j] = 0.f;
            continue;
        }
        const float dx = xi - f[j * 5 + 0], dy = yi - f[j * 5 + 1];
        const float dr = ri - f[j * 5 + 2], dg = gi - f[j * 5 + 3], db = bi - f[j * 5 + 4];
        const float p2 = dx * dx + dy * dy, c2 = dr * dr + dg * dg + db * db;
        const float v = (j == i) ? 0.f : expf(-p2 * inv2p - c2 * inv2c);
        row[j] = v;
    }
}

// The BF16 copy of K for the tensor-core step, in blocks of 128 rows by 64
// columns: block (tile, chunk) of instance b starts at element
// ((b * nchunk + chunk) * ntiles + tile) * 8192 (chunk-major, so the blocks
// that all row tiles read at the same moment lie side by side in memory and
// spread over every memory channel) and holds row r, column k at
// byte r * 128 + (((k / 8) ^ (r % 8)) * 16) + (k % 8) * 2 -- the 128-byte
// swizzled K-major layout the MMA reads from shared memory, so one block is
// one contiguous 16 KiB bulk copy.  Rows and columns past N are zero.
__global__ void dense_kernel_build_tiled_kernel(const float *__restrict__ feats, __nv_bfloat16 *__restrict__ K,
                                                int N, int ntiles, int nchunk, float inv2p, float inv2c) {
    const int b = blockIdx.z;
    const int i = blockIdx.y;                 // row, < ntiles * 128
    const float *f = feats + (size_t)b * N * 5;
    const bool row_ok = i < N;
    float xi = 0.f, yi = 0.f, ri = 0.f, gi = 0.f, bi = 0.f;
    if (row_ok) {
        xi = f[i * 5 + 0];
        yi = f[i * 5 + 1];
        ri = f[i * 5 + 2];
        gi = f[i * 5 + 3];
        bi = f[i * 5 + 4];
    }
    const int tile = i / 128, r = i % 128;
    uint8_t *tb = reinterpret_cast<uint8_t *>(K) + ((size_t)b * nchunk * ntiles + tile) * 16384 + (size_t)r * 128;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nchunk * 64; j += gridDim.x * blockDim.x) {
        float v = 0.f;
        if (row_ok && j < N && j != i) {
            const float dx = xi - f[j * 5 + 0], dy = yi - f[j * 5 + 1];
            const float dr = ri - f[j * 5 + 2], dg = gi - f[j * 5 + 3], db = bi - f[j * 5 + 4];
            const float p2 = dx * dx + dy * dy, c2 = dr * dr + dg * dg + db * db;
            v = expf(-p2 * inv2p - c2 * inv2c);
        }
        const int chunk = j / 64, k = j % 64;
        *reinterpret_cast<__nv_bfloat16 *>(tb + (size_t)chunk * ntiles * 16384 + (((k >> 3) ^ (r & 7)) << 4) +
                                           (k & 7) * 2) =
            __float2bfloat16_rn(v);
    }
}

// q = exp(log q) as FP32 rows [B][N][LP] (padding 0) and, if qt16 is given,
// BF16 label-major [B][32][pitch] (labels >= L zero) for the tensor-core form.
__global__ void dense_export_q_kernel(const float *__restrict__ s, float *__restrict__ q32,
                                      __nv_bfloat16 *__restrict__ qt16, int B, int N, int L, int LP, int pitch) {
    const long long n = (long long)B * N * LP;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int l = (int)(idx % LP);
        const long long bi = idx / LP;
        const int b = (int)(bi / N), i = (int)(bi % N);
        const float q = l < L ? expf(s[idx]) : 0.f;
        if (q32) q32[idx] = q;
        if (qt16 && l < 32) qt16[((size_t)b * 32 + l) * pitch + i] = __float2bfloat16_rn(q);
    }
}

}  // namespace

cudaError_t launch_dense_kernel_build(const float *feats, float *K32, __nv_bfloat16 *K16, int B, int N,
                                      double theta_pos, double theta_rgb, cudaStream_t st) {
    const float inv2p = (float)(1.0 / (2.0 * theta_pos * theta_pos));
    const float inv2c = (float)(1.0 / (2.0 * theta_rgb * theta_rgb));
    dim3 grid((N + 255) / 256 < 8 ? (N + 255) / 256 : 8, N, B);
    if (K32) dense_kernel_build_kernel<<<grid, 256, 0, st>>>(feats, K32, N, dense_k32_pitch(N), inv2p, inv2c);
    if (K16) {
        const int ntiles = dense_tc_tiles(N), nchunk = dense_tc_pitch(N) / 64;
        dim3 g2((nchunk * 64 + 255) / 256 < 8 ? (nchunk * 64 + 255) / 256 : 8, ntiles * 128, B);
        dense_kernel_build_tiled_kernel<<<g2, 256, 0, st>>>(feats, K16, N, ntiles, nchunk, inv2p, inv2c);
    }
    return cudaGetLastError();
}

namespace {

// One thread per (instance, chunk, column): the six rows of a chunk's column
// (see launch_dense_fly_features).
__global__ void dense_fly_features_kernel(const float *__restrict__ feats, float *__restrict__ featsT, int B, int N,
                                          int nchunk, float sp, float sc) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)B * nchunk * 64) return;
    const int j = (int)(idx % 64);
    const long long bc = idx / 64;                 // b * nchunk + chunk
    const int chunk = (int)(bc % nchunk), b = (int)(bc / nchunk);
    const int J = chunk * 64 + j;
    float *out = featsT + bc * 6 * 64 + j;
    if (J >= N) {
        for (int k = 0; k < 5; ++k) out[k * 64] = 0.f;
        out[5 * 64] = -1e30f;
        return;
    }
    const float *f = feats + ((size_t)b * N + J) * 5;
    float g[5];
    g[0] = sp * f[0];
    g[1] = sp * f[1];
    g[2] = sc * f[2];
    g[3] = sc * f[3];
    g[4] = sc * f[4];
    float n2 = 0.f;
    for (int k = 0; k < 5; ++k) {
        out[k * 64] = 1.41421356f * g[k];
        n2 = fmaf(g[k], g[k], n2);
    }
    out[5 * 64] = -n2;
}

}  // namespace

cudaError_t launch_dense_fly_features(const float *feats, float *featsT, int B, int N, double theta_pos,
                                      double theta_rgb, cudaStream_t st) {
    // K = exp(-d^2 / (2 theta^2)) = 2^(-(s d)^2) with s = sqrt(log2(e) / (2 theta^2))
    const double log2e = 1.4426950408889634;
    const float sp = (float)std::sqrt(log2e / (2.0 * theta_pos * theta_pos));
    const float sc = (float)std::sqrt(log2e / (2.0 * theta_rgb * theta_rgb));
    const int nchunk = dense_tc_pitch(N) / 64;
    const long long n = (long long)B * nchunk * 64;
    dense_fly_features_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(feats, featsT, B, N, nchunk, sp, sc);
    return cudaGetLastError();
}

cudaError_t launch_dense_export_q(const float *s, float *q32, __nv_bfloat16 *qt16, int B, int N, int L, int LP,
                                  cudaStream_t st) {
    const long long n = (long long)B * N * LP;
    const int blocks = (int)std::min<long long>((n + 255) / 256, 1 << 20);
    dense_export_q_kernel<<<blocks, 256, 0, st>>>(s, q32, qt16, B, N, L, LP, dense_tc_pitch(N));
    return cudaGetLastError();
}

}  // namespace proxmf
