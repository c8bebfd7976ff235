// layout.cu -- conversions between the external [B][N][L] row layout and the
// internal padded pixel-major [B][N][LP] layout, the initial state q^0, and
// small fills.  None of this runs inside the iteration loop.
#include <cmath>

#include "internal.h"

namespace proxmf {

namespace {

constexpr int kThreads = 256;

// The row kernels below are bound by HBM (or the host link, for page-locked
// buffers used in place).  The external rows of L floats are a contiguous
// segment per block, moved as 16-byte vectors through shared memory; the padded
// rows are 16-byte vectors of a row.  A row is handled by G lanes holding one
// vector each, so its log-sum-exp is a shuffle tree and the row is read once.
// 1 M rows of 21 labels: unaries in with q^0 (290 MB) 55 us, rows out (190 MB)
// 29 us, q^0 alone (200 MB) 38 us; with one thread per element and its 64-bit
// division, and one thread per row for q^0, 245 us (two passes), 105 and 129.
template <int LP>
struct RowGeom {
    static constexpr int V = LP == 2 ? 2 : 4;                                // floats of a vector
    static constexpr int GL = LP / V;                                        // lanes with labels
    static constexpr int G = GL <= 1 ? 1 : GL <= 2 ? 2 : GL <= 4 ? 4 : 8;    // lanes per row
    static constexpr int RB = LP <= 4 ? 512 : LP <= 8 ? 256 : 128;           // rows per block
};

template <int V>
__device__ __forceinline__ void vget(float (&v)[V], const float *p) {
    if constexpr (V == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
    } else {
        const float2 t = *reinterpret_cast<const float2 *>(p);
        v[0] = t.x, v[1] = t.y;
    }
}

template <int V>
__device__ __forceinline__ void vput(float *p, const float (&v)[V]) {
    if constexpr (V == 4)
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else
        *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
}

// n contiguous floats between global (any 4-byte alignment) and shared memory.
__device__ __forceinline__ void copy_block(float *dst, const float *src, int n, bool vec) {
    if (vec) {
        for (int i = threadIdx.x; i < n / 4; i += kThreads)
            reinterpret_cast<float4 *>(dst)[i] = reinterpret_cast<const float4 *>(src)[i];
        for (int i = n / 4 * 4 + threadIdx.x; i < n; i += kThreads) dst[i] = src[i];
    } else {
        for (int i = threadIdx.x; i < n; i += kThreads) dst[i] = src[i];
    }
}
__device__ __forceinline__ bool aligned16(const void *p) { return ((uintptr_t)p & 15) == 0; }

// log softmax(-u) of a row over the G lanes that hold it (padding kPadLogQ).
template <int LP>
__device__ __forceinline__ void row_logq(float (&s)[RowGeom<LP>::V], const float (&u)[RowGeom<LP>::V], int g, int L) {
    using R = RowGeom<LP>;
    float mx = -INFINITY, z = 0.f;
#pragma unroll
    for (int j = 0; j < R::V; ++j)
        if (g * R::V + j < L) mx = fmaxf(mx, -u[j]);
#pragma unroll
    for (int o = R::G / 2; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll
    for (int j = 0; j < R::V; ++j)
        if (g * R::V + j < L) z += expf(-u[j] - mx);
#pragma unroll
    for (int o = R::G / 2; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    const float lse = mx + logf(z);
#pragma unroll
    for (int j = 0; j < R::V; ++j) s[j] = g * R::V + j < L ? -u[j] - lse : kPadLogQ;
}

// rows [R][L] -> padded rows [R][LP]; with s also q^0 = softmax(-row) as log q.
template <int LP>
__global__ void __launch_bounds__(kThreads)
rows_to_padded_kernel(const float *__restrict__ src, float *__restrict__ dst, float *__restrict__ s, long long rows,
                      int L, float pad) {
    using R = RowGeom<LP>;
    __shared__ __align__(16) float sm[R::RB * LP];
    const long long r0 = (long long)blockIdx.x * R::RB;
    const int nr = (int)min((long long)R::RB, rows - r0);
    const float *seg = src + r0 * L;
    copy_block(sm, seg, nr * L, aligned16(seg));
    __syncthreads();
    const int g = threadIdx.x & (R::G - 1);
    for (int base = 0; base < nr; base += kThreads / R::G) {
        const int row = base + threadIdx.x / R::G;
        const bool act = row < nr;
        float v[R::V];
#pragma unroll
        for (int j = 0; j < R::V; ++j) {
            const int l = g * R::V + j;
            v[j] = act && l < L ? sm[row * L + l] : pad;
        }
        const long long o = (r0 + row) * LP + g * R::V;
        if (act && g < R::GL) vput<R::V>(dst + o, v);
        if (s != nullptr) {
            float t[R::V];
            row_logq<LP>(t, v, g, L);
            if (act && g < R::GL) vput<R::V>(s + o, t);
        }
    }
}

// padded rows [R][LP] -> rows [R][L], as they are or their exponentials.
template <int LP>
__global__ void __launch_bounds__(kThreads)
padded_to_rows_kernel(const float *__restrict__ src, float *__restrict__ dst, long long rows, int L, int mode) {
    using R = RowGeom<LP>;
    __shared__ __align__(16) float sm[R::RB * LP];
    const long long r0 = (long long)blockIdx.x * R::RB;
    const int nr = (int)min((long long)R::RB, rows - r0);
    for (int i = threadIdx.x; i < nr * R::GL; i += kThreads) {
        const int row = i / R::GL, g = i - row * R::GL;
        float v[R::V];
        vget<R::V>(v, src + (r0 + row) * LP + g * R::V);
#pragma unroll
        for (int j = 0; j < R::V; ++j) {
            const int l = g * R::V + j;
            if (l < L) sm[row * L + l] = mode == CONV_EXP ? expf(v[j]) : v[j];
        }
    }
    __syncthreads();
    float *seg = dst + r0 * L;
    copy_block(seg, sm, nr * L, aligned16(seg));
}

// q^0 = softmax(-U): unary-only marginals, written as log q (padded rows).
template <int LP>
__global__ void __launch_bounds__(kThreads)
init_logq_kernel(const float *__restrict__ U, float *__restrict__ s, long long rows, int L) {
    using R = RowGeom<LP>;
    constexpr int per = kThreads / R::G;
    const int g = threadIdx.x & (R::G - 1);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const long long row = ((long long)blockIdx.x * 4 + k) * per + threadIdx.x / R::G;
        const bool act = row < rows && g < R::GL;
        const long long o = row * LP + g * R::V;
        float u[R::V], t[R::V];
#pragma unroll
        for (int j = 0; j < R::V; ++j) u[j] = 0.f;
        if (act) vget<R::V>(u, U + o);
        row_logq<LP>(t, u, g, L);
        if (act) vput<R::V>(s + o, t);
    }
}

// Direction k of the grid: 0 right, 1 down, 2 down-right, 3 down-left.
__device__ __forceinline__ void dir_offset(int k, int *dy, int *dx) {
    *dy = k == 0 ? 0 : 1;
    *dx = k == 0 ? 1 : (k == 1 ? 0 : (k == 2 ? 1 : -1));
}

// [B][nd][H][W] -> [B][H*W][nd], zero where the edge would leave the image;
// a thread per pixel, one vector store.
template <int ND>
__global__ void __launch_bounds__(kThreads)
weights_to_pixel_major_kernel(const float *__restrict__ src, float *__restrict__ dst, int H, int W) {
    const size_t HW = (size_t)H * W, b = blockIdx.y;
    for (size_t p = (size_t)blockIdx.x * kThreads + threadIdx.x; p < HW; p += (size_t)gridDim.x * kThreads) {
        const int y = (int)(p / (unsigned)W), x = (int)(p - (size_t)y * W);
        float v[ND];
#pragma unroll
        for (int k = 0; k < ND; ++k) {
            int dy, dx;
            dir_offset(k, &dy, &dx);
            const int yy = y + dy, xx = x + dx;
            v[k] = yy < H && xx >= 0 && xx < W ? src[(b * ND + k) * HW + p] : 0.f;
        }
        vput<ND>(dst + (b * HW + p) * ND, v);
    }
}

__global__ void lambda_to_d_kernel(const double *Lambda, float *d, int B) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < B) d[i] = (float)fmax(Lambda[i], 0.0);
}

__global__ void fill_eta_kernel(float *eta, int B, float v) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < B) eta[i] = v;
}

}  // namespace

// The stored label counts (storage_labels).
#define PROXMF_LPS(X) X(2) X(4) X(8) X(12) X(16) X(20) X(24) X(28) X(32)

cudaError_t launch_rows_to_padded(const float *src, float *dst, long long rows, int L, int LP, float pad,
                                  cudaStream_t st) {
    return launch_unary_rows(src, dst, nullptr, rows, L, LP, pad, st);
}

cudaError_t launch_unary_rows(const float *src, float *dst, float *s, long long rows, int L, int LP, float pad,
                              cudaStream_t st) {
    switch (LP) {
#define PROXMF_CASE(V)                                                                                             case V:                                                                                                            rows_to_padded_kernel<V><<<(unsigned)((rows + RowGeom<V>::RB - 1) / RowGeom<V>::RB), kThreads, 0, st>>>(             src, dst, s, rows, L, pad);                                                                                break;
        PROXMF_LPS(PROXMF_CASE)
#undef PROXMF_CASE
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_padded_to_rows(const float *src, float *dst, long long rows, int L, int LP, int mode,
                                  cudaStream_t st) {
    switch (LP) {
#define PROXMF_CASE(V)                                                                                             case V:                                                                                                            padded_to_rows_kernel<V><<<(unsigned)((rows + RowGeom<V>::RB - 1) / RowGeom<V>::RB), kThreads, 0, st>>>(             src, dst, rows, L, mode);                                                                                  break;
        PROXMF_LPS(PROXMF_CASE)
#undef PROXMF_CASE
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_weights_to_pixel_major(const float *src, float *dst, int B, int nd, int H, int W,
                                          cudaStream_t st) {
    const long long nb = ((long long)H * W + kThreads - 1) / kThreads;
    const dim3 grid((unsigned)(nb < 65536 ? nb : 65536), (unsigned)B);
    if (nd == 4)
        weights_to_pixel_major_kernel<4><<<grid, kThreads, 0, st>>>(src, dst, H, W);
    else
        weights_to_pixel_major_kernel<2><<<grid, kThreads, 0, st>>>(src, dst, H, W);
    return cudaGetLastError();
}

cudaError_t launch_init_logq(const float *U, float *s, long long rows, int L, int LP, cudaStream_t st) {
    switch (LP) {
#define PROXMF_CASE(V)                                                                               case V: {                                                                                            constexpr int per = 4 * kThreads / RowGeom<V>::G;                                                init_logq_kernel<V><<<(unsigned)((rows + per - 1) / per), kThreads, 0, st>>>(U, s, rows, L);         break;                                                                                       }
        PROXMF_LPS(PROXMF_CASE)
#undef PROXMF_CASE
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_lambda_to_d(const double *Lambda, float *d, int B, cudaStream_t st) {
    lambda_to_d_kernel<<<(B + 127) / 128, 128, 0, st>>>(Lambda, d, B);
    return cudaGetLastError();
}

namespace {

// A thread per 8 labels of a row: one 16-byte store.
__global__ void __launch_bounds__(kThreads)
to_bf16_kernel(const float *__restrict__ src, __nv_bfloat16 *__restrict__ dst, long long rows, int LP, int pitch) {
    const unsigned per = (unsigned)pitch / 8;
    for (long long r0 = (long long)blockIdx.x * kThreads; r0 < rows; r0 += (long long)gridDim.x * kThreads) {
        const unsigned nr = (unsigned)min((long long)kThreads, rows - r0);
        for (unsigned i = threadIdx.x; i < nr * per; i += kThreads) {
            const unsigned row = i / per, l0 = (i - row * per) * 8;
            const float *p = src + (r0 + row) * LP;
            __align__(16) __nv_bfloat16 v[8];
#pragma unroll
            for (unsigned j = 0; j < 8; ++j)
                v[j] = __float2bfloat16_rn(l0 + j < (unsigned)LP ? p[l0 + j] : 0.f);
            *reinterpret_cast<uint4 *>(dst + (r0 + row) * pitch + l0) = *reinterpret_cast<const uint4 *>(v);
        }
    }
}

}  // namespace

cudaError_t launch_to_bf16(const float *src, __nv_bfloat16 *dst, long long rows, int LP, int pitch,
                           cudaStream_t st) {
    const long long nb = (rows + kThreads - 1) / kThreads;
    to_bf16_kernel<<<(unsigned)(nb < 65536 ? nb : 65536), kThreads, 0, st>>>(src, dst, rows, LP, pitch);
    return cudaGetLastError();
}

cudaError_t launch_fill_eta(float *eta, int B, double value, cudaStream_t st) {
    fill_eta_kernel<<<(B + 127) / 128, 128, 0, st>>>(eta, B, (float)value);
    return cudaGetLastError();
}

}  // namespace proxmf
