// nn.cu -- the learned warm start (not in the paper): the entry points of the
// 3x3x3 convolutions, whose tensor-core kernels are in nn_tc.cu, the bias
// gradient and the elementwise steps of training.  See include/lbm_nn.h.
#include <cuda_bf16.h>

#include <cstdint>

#include "internal.h"
#include "lbm_nn.h"
#include "tc.cuh"

namespace lbm {
namespace nn {

using bf16 = __nv_bfloat16;

// Partial bias gradients of blocks of kBiasRows rows: part[blockIdx.x][c] = sum
// of dy over the block's rows, in row order (one FP32 chain per channel: the
// order is part of the result's rounding).  The block's threads bring the rows
// to shared memory, tile after tile, 16 bytes at a time where VEC (C % 8 == 0,
// aligned), the next tile in flight while one thread per channel walks the
// last.  Bound by that chain, 4096 additions, about 10 us for any layer; walking
// memory instead of shared memory the 15 layers of a training step on 8 x 64^3
// voxels took 5.4 ms with their chunk sums.
constexpr int kBiasThreads = 256;
constexpr int kBiasRows = 4096;
constexpr int kBiasTile = 8192;  // values of a tile, at most (a row wider than that takes several passes)

template <bool VEC>
__global__ void __launch_bounds__(kBiasThreads) k_bias_grad(const bf16* __restrict__ dy, long long M, int C,
                                                            float* __restrict__ part) {
    __shared__ __align__(16) bf16 sm[2][kBiasTile];
    const long long r0 = (long long)blockIdx.x * kBiasRows;
    const int rows = (int)(M - r0 < kBiasRows ? M - r0 : kBiasRows);
    // the channels from blockIdx.y * kBiasThreads, one per thread
    const int c0 = blockIdx.y * kBiasThreads, cn = C - c0 < kBiasThreads ? C - c0 : kBiasThreads;
    const int tr = kBiasTile / cn, tiles = (rows + tr - 1) / tr;
    const bf16* src = dy + r0 * C + c0;
    auto load = [&](int t) {
        bf16* dst = sm[t & 1];
        const int n = rows - t * tr < tr ? rows - t * tr : tr;
        if constexpr (VEC) {
            const int g8 = cn / 8;
            for (int e = threadIdx.x; e < n * g8; e += kBiasThreads) {
                const int r = e / g8, g = e - r * g8;
                tc::cp_async16(dst + (size_t)e * 8, src + (long long)(t * tr + r) * C + g * 8, true);
            }
        } else {
            for (int e = threadIdx.x; e < n * cn; e += kBiasThreads) {
                const int r = e / cn, c = e - r * cn;
                dst[e] = src[(long long)(t * tr + r) * C + c];
            }
        }
        tc::cp_async_commit();
    };
    float s = 0.f;
    load(0);
    for (int t = 0; t < tiles; t++) {
        if (t + 1 < tiles) load(t + 1);
        else tc::cp_async_commit();
        tc::cp_async_wait<1>();
        __syncthreads();
        const int n = rows - t * tr < tr ? rows - t * tr : tr;
        if ((int)threadIdx.x < cn) {
            const bf16* p = sm[t & 1] + threadIdx.x;
#pragma unroll 16
            for (int r = 0; r < n; r++) s += __bfloat162float(p[r * cn]);
        }
        __syncthreads();
    }
    if ((int)threadIdx.x < cn) part[(long long)blockIdx.x * C + c0 + threadIdx.x] = s;
}

__global__ void k_weight_flip(const bf16* __restrict__ w, int Cin, int Cout, bf16* __restrict__ wt) {
    const long long n = 27ll * Cin * Cout;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int co = (int)(e % Cout);
        const long long t = e / Cout;
        const int ci = (int)(t % Cin), tap = (int)(t / Cin);
        wt[((long long)(26 - tap) * Cout + co) * Cin + ci] = w[e];
    }
}

__global__ void k_relu_mask(bf16* __restrict__ g, const bf16* __restrict__ act, size_t n) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
        if (!(__bfloat162float(act[e]) > 0.f)) g[e] = __float2bfloat16(0.f);
}

__global__ void k_pool2(const bf16* __restrict__ x, int N, int D, int H, int W, int C, bf16* __restrict__ y) {
    const int d = D / 2, h = H / 2, w = W / 2;
    const long long n = (long long)N * d * h * w * C;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(e % C);
        long long t = e / C;
        const int xx = (int)(t % w);
        t /= w;
        const int yy = (int)(t % h);
        t /= h;
        const int zz = (int)(t % d);
        const int nn = (int)(t / d);
        float s = 0.f;
        for (int k = 0; k < 8; k++) {
            const int z = 2 * zz + (k >> 2), y_ = 2 * yy + ((k >> 1) & 1), x_ = 2 * xx + (k & 1);
            s += __bfloat162float(x[((((long long)nn * D + z) * H + y_) * W + x_) * C + c]);
        }
        y[e] = __float2bfloat16(0.125f * s);
    }
}

__global__ void k_pool2_bwd(const bf16* __restrict__ dy, int N, int D, int H, int W, int C, bf16* __restrict__ dx) {
    const long long n = (long long)N * D * H * W * C;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(e % C);
        long long t = e / C;
        const int x_ = (int)(t % W);
        t /= W;
        const int y_ = (int)(t % H);
        t /= H;
        const int z = (int)(t % D);
        const int nn = (int)(t / D);
        const long long src = ((((long long)nn * (D / 2) + z / 2) * (H / 2) + y_ / 2) * (W / 2) + x_ / 2) * C + c;
        dx[e] = __float2bfloat16(0.125f * __bfloat162float(dy[src]));
    }
}

__global__ void k_up2(const bf16* __restrict__ x, int N, int D, int H, int W, int C, bf16* __restrict__ y) {
    const long long n = (long long)N * 8 * D * H * W * C;
    const int D2 = 2 * D, H2 = 2 * H, W2 = 2 * W;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(e % C);
        long long t = e / C;
        const int x_ = (int)(t % W2);
        t /= W2;
        const int y_ = (int)(t % H2);
        t /= H2;
        const int z = (int)(t % D2);
        const int nn = (int)(t / D2);
        y[e] = x[((((long long)nn * D + z / 2) * H + y_ / 2) * W + x_ / 2) * C + c];
    }
}

__global__ void k_up2_bwd(const bf16* __restrict__ dy, int N, int D, int H, int W, int C, bf16* __restrict__ dx) {
    const long long n = (long long)N * D * H * W * C;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(e % C);
        long long t = e / C;
        const int x_ = (int)(t % W);
        t /= W;
        const int y_ = (int)(t % H);
        t /= H;
        const int z = (int)(t % D);
        const int nn = (int)(t / D);
        float s = 0.f;
        for (int k = 0; k < 8; k++) {
            const int zz = 2 * z + (k >> 2), yy = 2 * y_ + ((k >> 1) & 1), xx = 2 * x_ + (k & 1);
            s += __bfloat162float(dy[((((long long)nn * 2 * D + zz) * 2 * H + yy) * 2 * W + xx) * C + c]);
        }
        dx[e] = __float2bfloat16(s);
    }
}

__global__ void k_concat(const bf16* __restrict__ a, int ca, const bf16* __restrict__ b, int cb, size_t vox,
                         bf16* __restrict__ y) {
    const int c = ca + cb;
    const size_t n = vox * c;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const size_t v = e / c;
        const int k = (int)(e - v * c);
        y[e] = k < ca ? a[v * ca + k] : b[v * cb + (k - ca)];
    }
}

__global__ void k_split(const bf16* __restrict__ y, int ca, int cb, size_t vox, bf16* __restrict__ a,
                        bf16* __restrict__ b) {
    const int c = ca + cb;
    const size_t n = vox * c;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const size_t v = e / c;
        const int k = (int)(e - v * c);
        if (k < ca) {
            if (a) a[v * ca + k] = y[e];
        } else if (b) {
            b[v * cb + (k - ca)] = y[e];
        }
    }
}

__global__ void k_mse(const float* __restrict__ pred, const float* __restrict__ tgt, const uint8_t* __restrict__ mask,
                      size_t vox, int c, float inv_count, double* __restrict__ loss, bf16* __restrict__ dpred) {
    double s = 0.0;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < vox * c; e += (size_t)gridDim.x * blockDim.x) {
        const size_t v = e / c;
        float d = 0.f;
        if (mask[v]) d = pred[e] - tgt[e];
        s += (double)d * d;
        dpred[e] = __float2bfloat16(2.f * d * inv_count);
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0) atomicAdd(loss, s * inv_count);
}

__global__ void k_adam(float* __restrict__ p, float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       bf16* __restrict__ pb, size_t n, float lr, float b1, float b2, float eps, float c1, float c2) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const float gr = g[e];
        const float mm = b1 * m[e] + (1.f - b1) * gr;
        const float vv = b2 * v[e] + (1.f - b2) * gr * gr;
        m[e] = mm;
        v[e] = vv;
        const float q = p[e] - lr * (mm * c1) / (sqrtf(vv * c2) + eps);
        p[e] = q;
        g[e] = 0.f;
        if (pb) pb[e] = __float2bfloat16(q);
    }
}

__global__ void k_add(const bf16* __restrict__ a, const bf16* __restrict__ b, size_t n, bf16* __restrict__ y) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
        y[e] = __float2bfloat16(__bfloat162float(a[e]) + __bfloat162float(b[e]));
}

__global__ void k_mask_input(const uint8_t* __restrict__ mask, size_t vox, float value, bf16* __restrict__ x) {
    for (size_t v = (size_t)blockIdx.x * blockDim.x + threadIdx.x; v < vox; v += (size_t)gridDim.x * blockDim.x) {
        x[2 * v] = __float2bfloat16(mask[v] ? 1.f : 0.f);
        x[2 * v + 1] = __float2bfloat16(value);
    }
}

__global__ void k_fields_to_target(const double* __restrict__ rho, const double* __restrict__ u, size_t vox,
                                   double rho0, double inv_s_rho, double inv_s_u, float* __restrict__ t) {
    for (size_t v = (size_t)blockIdx.x * blockDim.x + threadIdx.x; v < vox; v += (size_t)gridDim.x * blockDim.x) {
        double r = rho[v];
        const bool ok = isfinite(r);
        t[4 * v] = ok ? (float)((r - rho0) * inv_s_rho) : 0.f;
        for (int c = 0; c < 3; c++) {
            const double uc = u[c * vox + v];
            t[4 * v + 1 + c] = ok && isfinite(uc) ? (float)(uc * inv_s_u) : 0.f;
        }
    }
}

__global__ void k_target_to_fields(const float* __restrict__ t, size_t vox, double rho0, double s_rho, double s_u,
                                   double* __restrict__ rho, double* __restrict__ u) {
    for (size_t v = (size_t)blockIdx.x * blockDim.x + threadIdx.x; v < vox; v += (size_t)gridDim.x * blockDim.x) {
        rho[v] = rho0 + s_rho * (double)t[4 * v];
        for (int c = 0; c < 3; c++) u[c * vox + v] = s_u * (double)t[4 * v + 1 + c];
    }
}

__global__ void k_f2b(const float* __restrict__ x, size_t n, bf16* __restrict__ y) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
        y[e] = __float2bfloat16(x[e]);
}

__global__ void k_b2f(const bf16* __restrict__ x, size_t n, float* __restrict__ y) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
        y[e] = __bfloat162float(x[e]);
}

static unsigned grid_for(size_t n) {
    const size_t b = (n + 255) / 256;
    return (unsigned)(b < 4096 ? (b ? b : 1) : 4096);
}

static cudaStream_t S(void* s) { return static_cast<cudaStream_t>(s); }

static int check(cudaError_t e, const char* what) { return e == cudaSuccess ? LBM_OK : cuda_fail(e, what); }

}  // namespace nn
}  // namespace lbm

using namespace lbm;
using namespace lbm::nn;

namespace lbm {
namespace nn {
int conv3d(const void* x, int n, int d, int h, int w, int cin, const void* wgt, const float* bias, int cout, int relu,
           int wrap, void* y, float* y32, cudaStream_t s);
float* chunk_scratch(size_t floats);
int sum_few(const float* part, long long chunks, long long E, float* dst, cudaStream_t s);
int wgrad_tc(const void* x, const void* dy, int n, int d, int h, int w, int cin, int cout, int wrap, float* dw,
             cudaStream_t s);
}  // namespace nn
}  // namespace lbm

extern "C" int lbm_nn_conv3d(const void* x, int n, int d, int h, int w, int cin, const void* wgt,
                             const float* bias, int cout, int relu, int wrap, void* y, float* y32, void* stream) {
    if (!x || !wgt || n < 1 || d < 1 || h < 1 || w < 1 || cin < 1 || cout < 1 || (!y && !y32) || (wrap & ~7))
        return fail(LBM_ERR_ARG, "lbm_nn_conv3d: bad arguments");
    return conv3d(x, n, d, h, w, cin, wgt, bias, cout, relu, wrap, y, y32, S(stream));
}

extern "C" int lbm_nn_weight_flip(const void* wgt, int cin, int cout, void* wt, void* stream) {
    if (!wgt || !wt || cin < 1 || cout < 1) return fail(LBM_ERR_ARG, "lbm_nn_weight_flip: bad arguments");
    k_weight_flip<<<grid_for(27ull * cin * cout), 256, 0, S(stream)>>>(static_cast<const bf16*>(wgt), cin, cout,
                                                                       static_cast<bf16*>(wt));
    return check(cudaGetLastError(), "k_weight_flip launch");
}

extern "C" int lbm_nn_conv3d_wgrad(const void* x, const void* dy, int n, int d, int h, int w, int cin, int cout,
                                   int wrap, float* dw, float* dbias, void* stream) {
    if (!x || !dy || !dw || n < 1 || d < 1 || h < 1 || w < 1 || cin < 1 || cout < 1 || (wrap & ~7))
        return fail(LBM_ERR_ARG, "lbm_nn_conv3d_wgrad: bad arguments");
    // per-chunk partial sums that are added in chunk order (the result does
    // not depend on the order blocks finish in)
    int rc = wgrad_tc(x, dy, n, d, h, w, cin, cout, wrap, dw, S(stream));
    const long long M = (long long)n * d * h * w;
    if (rc || !dbias) return rc;
    const long long nb = (M + kBiasRows - 1) / kBiasRows;
    float* part = chunk_scratch((size_t)nb * cout);  // the weight gradient's sums are already in dw
    if (!part) return fail(LBM_ERR_OOM, "bias-gradient partial sums");
    const dim3 grid((unsigned)nb, (unsigned)((cout + kBiasThreads - 1) / kBiasThreads));
    // 16-byte copies where every row's channels allow them (row starts are cout values apart)
    if (cout % 8 == 0 && reinterpret_cast<uintptr_t>(dy) % 16 == 0)
        k_bias_grad<true><<<grid, kBiasThreads, 0, S(stream)>>>(static_cast<const bf16*>(dy), M, cout, part);
    else
        k_bias_grad<false><<<grid, kBiasThreads, 0, S(stream)>>>(static_cast<const bf16*>(dy), M, cout, part);
    rc = check(cudaGetLastError(), "k_bias_grad launch");
    return rc ? rc : sum_few(part, nb, cout, dbias, S(stream));
}

extern "C" int lbm_nn_relu_mask(void* g, const void* act, size_t count, void* stream) {
    if (!g || !act) return fail(LBM_ERR_ARG, "lbm_nn_relu_mask: NULL");
    k_relu_mask<<<grid_for(count), 256, 0, S(stream)>>>(static_cast<bf16*>(g), static_cast<const bf16*>(act), count);
    return check(cudaGetLastError(), "k_relu_mask launch");
}

extern "C" int lbm_nn_pool2(const void* x, int n, int d, int h, int w, int c, void* y, void* stream) {
    if (!x || !y || (d | h | w) & 1) return fail(LBM_ERR_ARG, "lbm_nn_pool2: bad arguments");
    k_pool2<<<grid_for((size_t)n * d * h * w * c / 8), 256, 0, S(stream)>>>(static_cast<const bf16*>(x), n, d, h, w,
                                                                            c, static_cast<bf16*>(y));
    return check(cudaGetLastError(), "k_pool2 launch");
}

extern "C" int lbm_nn_pool2_bwd(const void* dy, int n, int d, int h, int w, int c, void* dx, void* stream) {
    if (!dy || !dx || (d | h | w) & 1) return fail(LBM_ERR_ARG, "lbm_nn_pool2_bwd: bad arguments");
    k_pool2_bwd<<<grid_for((size_t)n * d * h * w * c), 256, 0, S(stream)>>>(static_cast<const bf16*>(dy), n, d, h, w,
                                                                            c, static_cast<bf16*>(dx));
    return check(cudaGetLastError(), "k_pool2_bwd launch");
}

extern "C" int lbm_nn_up2(const void* x, int n, int d, int h, int w, int c, void* y, void* stream) {
    if (!x || !y) return fail(LBM_ERR_ARG, "lbm_nn_up2: NULL");
    k_up2<<<grid_for((size_t)n * 8 * d * h * w * c), 256, 0, S(stream)>>>(static_cast<const bf16*>(x), n, d, h, w, c,
                                                                           static_cast<bf16*>(y));
    return check(cudaGetLastError(), "k_up2 launch");
}

extern "C" int lbm_nn_up2_bwd(const void* dy, int n, int d, int h, int w, int c, void* dx, void* stream) {
    if (!dy || !dx) return fail(LBM_ERR_ARG, "lbm_nn_up2_bwd: NULL");
    k_up2_bwd<<<grid_for((size_t)n * d * h * w * c), 256, 0, S(stream)>>>(static_cast<const bf16*>(dy), n, d, h, w, c,
                                                                           static_cast<bf16*>(dx));
    return check(cudaGetLastError(), "k_up2_bwd launch");
}

extern "C" int lbm_nn_concat(const void* a, int ca, const void* b, int cb, size_t voxels, void* y, void* stream) {
    if (!a || !b || !y) return fail(LBM_ERR_ARG, "lbm_nn_concat: NULL");
    k_concat<<<grid_for(voxels * (ca + cb)), 256, 0, S(stream)>>>(static_cast<const bf16*>(a), ca,
                                                                 static_cast<const bf16*>(b), cb, voxels,
                                                                 static_cast<bf16*>(y));
    return check(cudaGetLastError(), "k_concat launch");
}

extern "C" int lbm_nn_split(const void* y, int ca, int cb, size_t voxels, void* a, void* b, void* stream) {
    if (!y) return fail(LBM_ERR_ARG, "lbm_nn_split: NULL");
    k_split<<<grid_for(voxels * (ca + cb)), 256, 0, S(stream)>>>(static_cast<const bf16*>(y), ca, cb, voxels,
                                                                static_cast<bf16*>(a), static_cast<bf16*>(b));
    return check(cudaGetLastError(), "k_split launch");
}

extern "C" int lbm_nn_mse(const float* pred, const float* target, const uint8_t* mask, size_t voxels, int c,
                          size_t count, double* loss, void* dpred, void* stream) {
    if (!pred || !target || !mask || !loss || !dpred || c < 1) return fail(LBM_ERR_ARG, "lbm_nn_mse: bad arguments");
    const float inv = count ? 1.f / ((float)count * c) : 0.f;
    LBM_CUDA_TRY(cudaMemsetAsync(loss, 0, sizeof(double), S(stream)));
    k_mse<<<grid_for(voxels * c), 256, 0, S(stream)>>>(pred, target, mask, voxels, c, inv, loss,
                                                       static_cast<bf16*>(dpred));
    return check(cudaGetLastError(), "k_mse launch");
}

extern "C" int lbm_nn_adam(float* p, float* g, float* m, float* v, void* pb, size_t count, float lr, float beta1,
                           float beta2, float eps, int t, void* stream) {
    if (!p || !g || !m || !v || t < 1) return fail(LBM_ERR_ARG, "lbm_nn_adam: bad arguments");
    const float c1 = 1.f / (1.f - powf(beta1, (float)t)), c2 = 1.f / (1.f - powf(beta2, (float)t));
    k_adam<<<grid_for(count), 256, 0, S(stream)>>>(p, g, m, v, static_cast<bf16*>(pb), count, lr, beta1, beta2, eps,
                                                   c1, c2);
    return check(cudaGetLastError(), "k_adam launch");
}

extern "C" int lbm_nn_add(const void* a, const void* b, size_t count, void* y, void* stream) {
    if (!a || !b || !y) return fail(LBM_ERR_ARG, "lbm_nn_add: NULL");
    k_add<<<grid_for(count), 256, 0, S(stream)>>>(static_cast<const bf16*>(a), static_cast<const bf16*>(b), count,
                                                  static_cast<bf16*>(y));
    return check(cudaGetLastError(), "k_add launch");
}

extern "C" int lbm_nn_mask_input(const uint8_t* mask, size_t voxels, float value, void* x, void* stream) {
    if (!mask || !x) return fail(LBM_ERR_ARG, "lbm_nn_mask_input: NULL");
    k_mask_input<<<grid_for(voxels), 256, 0, S(stream)>>>(mask, voxels, value, static_cast<bf16*>(x));
    return check(cudaGetLastError(), "k_mask_input launch");
}

extern "C" int lbm_nn_fields_to_target(const double* rho, const double* u, size_t voxels, double rho0,
                                       double s_rho, double s_u, float* t, void* stream) {
    if (!rho || !u || !t || !(s_rho != 0.0) || !(s_u != 0.0))
        return fail(LBM_ERR_ARG, "lbm_nn_fields_to_target: bad arguments");
    k_fields_to_target<<<grid_for(voxels), 256, 0, S(stream)>>>(rho, u, voxels, rho0, 1.0 / s_rho, 1.0 / s_u, t);
    return check(cudaGetLastError(), "k_fields_to_target launch");
}

extern "C" int lbm_nn_target_to_fields(const float* t, size_t voxels, double rho0, double s_rho, double s_u,
                                       double* rho, double* u, void* stream) {
    if (!t || !rho || !u) return fail(LBM_ERR_ARG, "lbm_nn_target_to_fields: NULL");
    k_target_to_fields<<<grid_for(voxels), 256, 0, S(stream)>>>(t, voxels, rho0, s_rho, s_u, rho, u);
    return check(cudaGetLastError(), "k_target_to_fields launch");
}

extern "C" int lbm_nn_f32_to_bf16(const float* x, size_t count, void* y, void* stream) {
    if (!x || !y) return fail(LBM_ERR_ARG, "lbm_nn_f32_to_bf16: NULL");
    k_f2b<<<grid_for(count), 256, 0, S(stream)>>>(x, count, static_cast<bf16*>(y));
    return check(cudaGetLastError(), "k_f2b launch");
}

extern "C" int lbm_nn_bf16_to_f32(const void* x, size_t count, float* y, void* stream) {
    if (!x || !y) return fail(LBM_ERR_ARG, "lbm_nn_bf16_to_f32: NULL");
    k_b2f<<<grid_for(count), 256, 0, S(stream)>>>(static_cast<const bf16*>(x), count, y);
    return check(cudaGetLastError(), "k_b2f launch");
}
