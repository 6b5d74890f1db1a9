// nn.cu -- the learned warm start (not in the paper): the entry points of the
// 3x3x3 convolutions, whose tcgen05 kernels are in nn_tc.cu, their mma.sync form
// for few channels and thin boxes, the bias gradient and the elementwise steps
// of training.  See include/lbm_nn.h.
#include <cuda_bf16.h>

#include <cstdint>
#include <type_traits>

#include "internal.h"
#include "lbm_nn.h"
#include "tc.cuh"

namespace lbm {
namespace nn {

using bf16 = __nv_bfloat16;

__device__ __forceinline__ void mma_bf16(float (&c)[4], const unsigned (&a)[4], const unsigned (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ unsigned lds32(const bf16* p) { return *reinterpret_cast<const unsigned*>(p); }

constexpr int BM = 64;  // GEMM rows per block
constexpr int BK = 32;  // reduction depth per shared-memory stage
constexpr int LD = BK + 8;

// Neighbour coordinate along one axis with zero padding (returns -1 outside)
// or periodic wrap.
__device__ __forceinline__ int nb_coord(int c, int d, int n, bool wrap) {
    c += d;
    if (wrap) return c < 0 ? c + n : (c >= n ? c - n : c);
    return (c < 0 || c >= n) ? -1 : c;
}

// C[p][co] = sum_k A[p][k] B[k][co], A[p][(tap,ci)] = x[p + off(tap)][ci] (0 outside,
// or wrapped on the axes set in `wrap`), B[(tap,ci)][co] = wgt[tap][ci][co]; one
// block computes 64 voxels x NF*8 outputs starting at channel blockIdx.y * NF*8.
// VEC: Cin % 16 == 0, so that a thread's 16 consecutive k share one tap and are
// read as two 16-byte vectors.  For the shapes of by_warps().
template <int NF, bool VEC>
__global__ void __launch_bounds__(128) k_conv(const bf16* __restrict__ x, int N, int D, int H, int W, int Cin,
                                              const bf16* __restrict__ wgt, const float* __restrict__ bias,
                                              int Cout, int relu, int wrap, bf16* __restrict__ y,
                                              float* __restrict__ y32) {
    constexpr int BN = NF * 8;
    __shared__ __align__(16) bf16 As[BM][LD];
    __shared__ __align__(16) bf16 Bs[BN][LD];
    const long long M = (long long)N * D * H * W;
    const int K = 27 * Cin;
    const long long m0 = (long long)blockIdx.x * BM;
    const int n0 = blockIdx.y * BN;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float acc[NF][4];
#pragma unroll
    for (int f = 0; f < NF; f++) acc[f][0] = acc[f][1] = acc[f][2] = acc[f][3] = 0.f;

    // this thread gathers row ar, columns ak .. ak+15 of every A stage
    const int ar = tid >> 1, ak = (tid & 1) * 16;
    const long long am = m0 + ar;
    const bool arow = am < M;
    int an = 0, az = 0, ay = 0, ax = 0;
    if (arow) {
        long long t = am;
        ax = (int)(t % W);
        t /= W;
        ay = (int)(t % H);
        t /= H;
        az = (int)(t % D);
        an = (int)(t / D);
    }
    const bool wx = wrap & 1, wy = wrap & 2, wz = wrap & 4;
    const bf16 zero = __float2bfloat16(0.f);
    for (int k0 = 0; k0 < K; k0 += BK) {
        int k = k0 + ak;
        int tap = k / Cin, ci = k - tap * Cin;
        if constexpr (VEC) {
            uint4 v0 = make_uint4(0, 0, 0, 0), v1 = v0;
            if (arow && k < K) {
                const int zz = nb_coord(az, tap / 9 - 1, D, wz), yy = nb_coord(ay, (tap / 3) % 3 - 1, H, wy),
                          xx = nb_coord(ax, tap % 3 - 1, W, wx);
                if ((zz | yy | xx) >= 0) {
                    const uint4* src =
                        reinterpret_cast<const uint4*>(x + ((((long long)an * D + zz) * H + yy) * W + xx) * Cin + ci);
                    v0 = src[0];
                    v1 = src[1];
                }
            }
            *reinterpret_cast<uint4*>(&As[ar][ak]) = v0;
            *reinterpret_cast<uint4*>(&As[ar][ak + 8]) = v1;
        } else {
#pragma unroll
            for (int j = 0; j < 16; j++) {
                bf16 v = zero;
                if (arow && k < K) {
                    const int zz = nb_coord(az, tap / 9 - 1, D, wz), yy = nb_coord(ay, (tap / 3) % 3 - 1, H, wy),
                              xx = nb_coord(ax, tap % 3 - 1, W, wx);
                    if ((zz | yy | xx) >= 0) v = x[((((long long)an * D + zz) * H + yy) * W + xx) * Cin + ci];
                }
                As[ar][ak + j] = v;
                k++;
                if (++ci == Cin) {
                    ci = 0;
                    tap++;
                }
            }
        }
        for (int e = tid; e < BN * BK; e += 128) {
            const int kk = e / BN, nn = e - kk * BN;
            const int kg = k0 + kk;
            Bs[nn][kk] = (kg < K && n0 + nn < Cout) ? wgt[(long long)kg * Cout + n0 + nn] : zero;
        }
        __syncthreads();
#pragma unroll
        for (int ks = 0; ks < BK; ks += 16) {
            const int r = warp * 16 + (lane >> 2), c = ks + (lane & 3) * 2;
            const unsigned a[4] = {lds32(&As[r][c]), lds32(&As[r + 8][c]), lds32(&As[r][c + 8]),
                                   lds32(&As[r + 8][c + 8])};
#pragma unroll
            for (int f = 0; f < NF; f++) {
                const int nn = f * 8 + (lane >> 2);
                const unsigned b[2] = {lds32(&Bs[nn][c]), lds32(&Bs[nn][c + 8])};
                mma_bf16(acc[f], a, b);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int f = 0; f < NF; f++)
#pragma unroll
        for (int h2 = 0; h2 < 2; h2++)
#pragma unroll
            for (int j = 0; j < 2; j++) {
                const long long row = m0 + warp * 16 + (lane >> 2) + h2 * 8;
                const int co = n0 + f * 8 + (lane & 3) * 2 + j;
                if (row < M && co < Cout) {
                    float v = acc[f][h2 * 2 + j] + (bias ? bias[co] : 0.f);
                    if (relu) v = fmaxf(v, 0.f);
                    if (y) y[row * Cout + co] = __float2bfloat16(v);
                    if (y32) y32[row * Cout + co] = v;
                }
            }
}

// Partial bias gradients of blocks of kBiasRows rows: part[blockIdx.x][c] = sum
// of dy over the block's rows, in row order (one FP32 chain per channel: the
// order is part of the result's rounding).  The block's threads bring the rows
// to shared memory, tile after tile, 16 bytes at a time where VEC (C % 8 == 0,
// aligned), else 4 (up to 256 channels: a tile is one run of values then), the next
// tile in flight while one thread per channel walks the last.  Bound by that chain,
// 4096 additions, about 10 us for 16 channels, and by the copies of one block per 4096
// rows with many (128 channels on 16^3 voxels 53 us; off by one value 74, value by
// value 310); walking memory instead of shared memory the 15 layers of a training step
// on 8 x 64^3 voxels took 5.4 ms with their chunk sums.
constexpr int kBiasThreads = 256;
constexpr int kBiasRows = 4096;
constexpr int kBiasTile = 8192;  // values of a tile, at most (a row holds the block's 256 channels at most)

// 1 where a value is the upper half of its 4-byte word.
__device__ __forceinline__ int odd_start(const bf16* p) { return (int)(reinterpret_cast<uintptr_t>(p) >> 1) & 1; }

template <bool VEC>
__global__ void __launch_bounds__(kBiasThreads) k_bias_grad(const bf16* __restrict__ dy, long long M, int C,
                                                            float* __restrict__ part) {
    __shared__ __align__(16) bf16 sm[2][kBiasTile + 8];
    const long long r0 = (long long)blockIdx.x * kBiasRows;
    const int rows = (int)(M - r0 < kBiasRows ? M - r0 : kBiasRows);
    // the channels from blockIdx.y * kBiasThreads, one per thread
    const int c0 = blockIdx.y * kBiasThreads, cn = C - c0 < kBiasThreads ? C - c0 : kBiasThreads;
    const int tr = kBiasTile / cn, tiles = (rows + tr - 1) / tr;
    const bf16* src = dy + r0 * C + c0;
    auto load = [&](int t) {
        bf16* dst = sm[t & 1];
        const int n = rows - t * tr < tr ? rows - t * tr : tr;
        if (!VEC && cn == C) {
            // the tile is one run of values: whole words, and the values at its ends that share theirs
            const bf16* from = src + (long long)t * tr * C;
            const int odd = odd_start(from), total = n * C;
            dst += odd;
            for (int e = odd + 2 * threadIdx.x; e + 2 <= total; e += 2 * kBiasThreads) tc::cp_async4(dst + e, from + e);
            if (threadIdx.x == 0 && odd) dst[0] = from[0];
            if (threadIdx.x == 0 && (total - odd) % 2) dst[total - 1] = from[total - 1];
        } else if constexpr (VEC) {
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
            const bf16* p = sm[t & 1] + threadIdx.x + (!VEC && cn == C ? odd_start(src + (long long)t * tr * C) : 0);
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

// ---- elementwise passes over activations ------------------------------------
// All are bound by memory.  A thread takes V consecutive channels of a voxel, 8
// (16 bytes) where the channel counts and addresses allow, and finds its voxel
// with indices of type I, 32 bits where the tensors allow: one channel per
// thread with 64-bit divisions these passes took 1.9 ms of a training step on 8
// x 64^3 voxels, several times their memory time.
template <int V>
struct alignas(2 * V) Pack {
    bf16 v[V];
};

template <int V>
__device__ __forceinline__ Pack<V> load_pack(const bf16* p) {
    return *reinterpret_cast<const Pack<V>*>(p);
}
template <int V>
__device__ __forceinline__ void store_pack(bf16* p, const Pack<V>& x) {
    *reinterpret_cast<Pack<V>*>(p) = x;
}

// (n packs and, behind them, `rest` < V values, the first threads' own)
template <int V, class I>
__global__ void k_relu_mask(bf16* __restrict__ g, const bf16* __restrict__ act, I n, int rest) {
    const I t = blockIdx.x * (I)blockDim.x + threadIdx.x;
    for (I e = t; e < n; e += (I)gridDim.x * blockDim.x) {
        const Pack<V> a = load_pack<V>(act + (size_t)e * V);
        Pack<V> x = load_pack<V>(g + (size_t)e * V);
#pragma unroll
        for (int k = 0; k < V; k++)
            if (!(__bfloat162float(a.v[k]) > 0.f)) x.v[k] = __float2bfloat16(0.f);
        store_pack(g + (size_t)e * V, x);
    }
    const size_t at = (size_t)n * V + t;
    if (t < (I)rest && !(__bfloat162float(act[at]) > 0.f)) g[at] = __float2bfloat16(0.f);
}

// The group of channels e of a tensor [.][D][H][W][G groups]: its sample, voxel
// and group.
template <class I>
struct Cell {
    I n;
    int z, y, x, g;
    __device__ __forceinline__ Cell(I e, int D, int H, int W, int G) {
        I t = e / G;
        g = (int)(e - t * G);
        I u = t / W;
        x = (int)(t - u * W);
        t = u / H;
        y = (int)(u - t * H);
        n = t / D;
        z = (int)(t - n * D);
    }
};

// y[n][z][y][x] = the mean (MEAN) or sum of the eight voxels of a D x H x W box of
// twice the size.
template <int V, class I, bool MEAN>
__global__ void k_down2(const bf16* __restrict__ x, I total, int D, int H, int W, int G, bf16* __restrict__ y) {
    for (I e = blockIdx.x * (I)blockDim.x + threadIdx.x; e < total; e += (I)gridDim.x * blockDim.x) {
        const Cell<I> c(e, D, H, W, G);
        float s[V];
#pragma unroll
        for (int j = 0; j < V; j++) s[j] = 0.f;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const size_t at = ((((size_t)c.n * 2 * D + 2 * c.z + (k >> 2)) * 2 * H + 2 * c.y + ((k >> 1) & 1)) * 2 * W + 2 * c.x + (k & 1)) * G + c.g;
            const Pack<V> v = load_pack<V>(x + at * V);
#pragma unroll
            for (int j = 0; j < V; j++) s[j] += __bfloat162float(v.v[j]);
        }
        Pack<V> o;
#pragma unroll
        for (int j = 0; j < V; j++) o.v[j] = __float2bfloat16(MEAN ? 0.125f * s[j] : s[j]);
        store_pack(y + (size_t)e * V, o);
    }
}

// y (D x H x W) from a box of half the size: each voxel's parent, an eighth of it (SCALE).
template <int V, class I, bool SCALE>
__global__ void k_up2(const bf16* __restrict__ x, I total, int D, int H, int W, int G, bf16* __restrict__ y) {
    for (I e = blockIdx.x * (I)blockDim.x + threadIdx.x; e < total; e += (I)gridDim.x * blockDim.x) {
        const Cell<I> c(e, D, H, W, G);
        const size_t at = ((((size_t)c.n * (D / 2) + c.z / 2) * (H / 2) + c.y / 2) * (W / 2) + c.x / 2) * G + c.g;
        Pack<V> v = load_pack<V>(x + at * V);
        if constexpr (SCALE) {
#pragma unroll
            for (int j = 0; j < V; j++) v.v[j] = __float2bfloat16(0.125f * __bfloat162float(v.v[j]));
        }
        store_pack(y + (size_t)e * V, v);
    }
}

// ga and gb groups of channels per voxel
template <int V, class I>
__global__ void k_concat(const bf16* __restrict__ a, int ga, const bf16* __restrict__ b, int gb, I total,
                         bf16* __restrict__ y) {
    for (I e = blockIdx.x * (I)blockDim.x + threadIdx.x; e < total; e += (I)gridDim.x * blockDim.x) {
        const I v = e / (ga + gb);
        const int k = (int)(e - v * (ga + gb));
        store_pack(y + (size_t)e * V, k < ga ? load_pack<V>(a + ((size_t)v * ga + k) * V)
                                             : load_pack<V>(b + ((size_t)v * gb + (k - ga)) * V));
    }
}

template <int V, class I>
__global__ void k_split(const bf16* __restrict__ y, int ga, int gb, I total, bf16* __restrict__ a, bf16* __restrict__ b) {
    for (I e = blockIdx.x * (I)blockDim.x + threadIdx.x; e < total; e += (I)gridDim.x * blockDim.x) {
        const I v = e / (ga + gb);
        const int k = (int)(e - v * (ga + gb));
        if (k < ga) {
            if (a) store_pack(a + ((size_t)v * ga + k) * V, load_pack<V>(y + (size_t)e * V));
        } else if (b) {
            store_pack(b + ((size_t)v * gb + (k - ga)) * V, load_pack<V>(y + (size_t)e * V));
        }
    }
}

// The block's squared errors are added up before its one atomic addition (one
// per warp made 32,768 additions to one address).
template <class I>
__global__ void __launch_bounds__(256) k_mse(const float* __restrict__ pred, const float* __restrict__ tgt,
                                             const uint8_t* __restrict__ mask, I total, int c, float inv_count,
                                             double* __restrict__ loss, bf16* __restrict__ dpred) {
    __shared__ double sm[8];
    double s = 0.0;
    for (I e = blockIdx.x * (I)blockDim.x + threadIdx.x; e < total; e += (I)gridDim.x * blockDim.x) {
        float d = 0.f;
        if (mask[e / c]) d = pred[e] - tgt[e];
        s += (double)d * d;
        dpred[e] = __float2bfloat16(2.f * d * inv_count);
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; w++) s += sm[w];
        atomicAdd(loss, s * inv_count);
    }
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

template <int V, class I>
__global__ void k_add(const bf16* a, const bf16* b, I n, int rest, bf16* y) {  // y may be a or b; as k_relu_mask
    const I t = blockIdx.x * (I)blockDim.x + threadIdx.x;
    for (I e = t; e < n; e += (I)gridDim.x * blockDim.x) {
        const Pack<V> p = load_pack<V>(a + (size_t)e * V), q = load_pack<V>(b + (size_t)e * V);
        Pack<V> o;
#pragma unroll
        for (int k = 0; k < V; k++) o.v[k] = __float2bfloat16(__bfloat162float(p.v[k]) + __bfloat162float(q.v[k]));
        store_pack(y + (size_t)e * V, o);
    }
    const size_t at = (size_t)n * V + t;
    if (t < (I)rest) y[at] = __float2bfloat16(__bfloat162float(a[at]) + __bfloat162float(b[at]));
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

// Output-channel tiling of k_conv: the channels are split into equal tiles of at most 128, each a multiple of 8.
static int pick_nf(int cout, int* n_tiles) {
    const int tiles = (cout + 127) / 128;
    const int per = (cout + tiles - 1) / tiles;
    const int need = (per + 7) / 8;
    static const int sizes[] = {1, 2, 4, 6, 8, 12, 16};
    int nf = 16;
    for (int s : sizes)
        if (s >= need) {
            nf = s;
            break;
        }
    *n_tiles = (cout + nf * 8 - 1) / (nf * 8);
    return nf;
}

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

// The convolutions that k_conv does faster than the tcgen05 kernels (on both, us):
// - voxels that start at odd addresses, for an odd number of input channels or a
//   tensor off by one value: gathered value by value either way (1 -> 16 channels on
//   4 x 32^3 voxels 21 and 47, 7 -> 9 84 and 171; from odd addresses 24 -> 32 285 and
//   559, 104 -> 128 2051 and 3273);
// - other voxels that allow no 8-channel loads, where both channels are few or the
//   outputs are up to 8 (6 -> 4 on 16^3 23 and 27, 10 -> 32 36 and 41, 20 -> 4 61 and 66;
//   but 26 -> 16 89 and 80, 10 -> 64 52 and 46);
// - boxes so thin along x or y that most of the 8 x 16 columns of the halo kernels is
//   padding, once that is what they spend their time on (2 -> 16 on 512 x 1 x 512 49
//   and 76, on 512 x 512 x 1, half as empty, 56 and 50; 16 -> 16 on 256 x 1 x 256 23
//   and 77, 64 -> 64 154 and 256), and boxes of one plane of 16 channels, each plane
//   with its two neighbours in z (16 -> 4 on 1 x 256 x 256 19 and 25).  Of multiples of
//   16 channels only boxes of up to 4 voxels along x or y, or one plane: any other
//   keeps the halo kernel's sums.
static bool by_warps(const void* x, int n, int d, int h, int w, int cin, int cout) {
    const uintptr_t at = reinterpret_cast<uintptr_t>(x);
    if (cin % 2) return true;
    const double voxels = (double)n * d * h * w;
    const double column = (double)n * ((h + 15) / 16) * ((w + 7) / 8) * 128;  // positions of one plane
    if ((cin == 2 || cin == 4) && at % (2 * cin) == 0) return column * d > 8 * voxels && column * d >= 1 << 18;
    if (cin % 16) return at % 4 || ((cin % 8 || at % 16) && (cout <= 8 || (cin <= 24 && cout <= 32)));
    if (at % 16 || (w > 4 && h > 4 && d > 1)) return false;
    const double read = column * (d + 2 * ((d + 15) / 16));  // positions that the halo planes hold
    if (cin == 16 && cout <= 16) return read > 2.75 * voxels && read >= 1 << 17;
    return read > (cin == 16 ? 8.5 : 16) * voxels && read >= 400e3;
}

extern "C" int lbm_nn_conv3d(const void* x, int n, int d, int h, int w, int cin, const void* wgt,
                             const float* bias, int cout, int relu, int wrap, void* y, float* y32, void* stream) {
    if (!x || !wgt || n < 1 || d < 1 || h < 1 || w < 1 || cin < 1 || cout < 1 || (!y && !y32) || (wrap & ~7))
        return fail(LBM_ERR_ARG, "lbm_nn_conv3d: bad arguments");
    if (!by_warps(x, n, d, h, w, cin, cout))
        return conv3d(x, n, d, h, w, cin, wgt, bias, cout, relu, wrap, y, y32, S(stream));
    const long long M = (long long)n * d * h * w;
    int ny = 0;
    const int nf = pick_nf(cout, &ny);
    const dim3 grid((unsigned)((M + BM - 1) / BM), (unsigned)ny);
    auto go = [&](auto kern) {
        kern<<<grid, 128, 0, S(stream)>>>(static_cast<const bf16*>(x), n, d, h, w, cin, static_cast<const bf16*>(wgt),
                                          bias, cout, relu, wrap, static_cast<bf16*>(y), y32);
    };
    const bool vec = cin % 16 == 0;
    switch (nf) {
        case 1: vec ? go(k_conv<1, true>) : go(k_conv<1, false>); break;
        case 2: vec ? go(k_conv<2, true>) : go(k_conv<2, false>); break;
        case 4: vec ? go(k_conv<4, true>) : go(k_conv<4, false>); break;
        case 6: vec ? go(k_conv<6, true>) : go(k_conv<6, false>); break;
        case 8: vec ? go(k_conv<8, true>) : go(k_conv<8, false>); break;
        case 12: vec ? go(k_conv<12, true>) : go(k_conv<12, false>); break;
        default: vec ? go(k_conv<16, true>) : go(k_conv<16, false>); break;
    }
    return check(cudaGetLastError(), "k_conv launch");
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

// Runs go(V, I) with the widest pack that the channel counts `c` (0: any) and
// the addresses `at` (ORed) allow, and indices wide enough for `total` values
// plus a grid's stride.
template <class F>
static void by_width(unsigned long long c, uintptr_t at, size_t total, F go) {
    const bool wide = c % 8 == 0 && at % 16 == 0, small = total < (1ull << 31);
    using W8 = std::integral_constant<int, 8>;
    using W1 = std::integral_constant<int, 1>;
    if (wide && small) go(W8{}, unsigned{});
    else if (wide) go(W8{}, (unsigned long long)0);
    else if (small) go(W1{}, unsigned{});
    else go(W1{}, (unsigned long long)0);
}
static uintptr_t adr(const void* p) { return reinterpret_cast<uintptr_t>(p); }

extern "C" int lbm_nn_relu_mask(void* g, const void* act, size_t count, void* stream) {
    if (!g || !act) return fail(LBM_ERR_ARG, "lbm_nn_relu_mask: NULL");
    by_width(0, adr(g) | adr(act), count, [&](auto V, auto I) {
        constexpr int v = decltype(V)::value;
        k_relu_mask<v, decltype(I)><<<grid_for(count / v), 256, 0, S(stream)>>>(
            static_cast<bf16*>(g), static_cast<const bf16*>(act), (decltype(I))(count / v), (int)(count % v));
    });
    return check(cudaGetLastError(), "k_relu_mask launch");
}

// One thread per pack of the result, of voxels n x d x h x w and c channels.
template <class K>
static void over_cells(const void* x, int n, int d, int h, int w, int c, void* y, K launch) {
    const size_t total = (size_t)n * d * h * w * c;
    by_width((unsigned)c, adr(x) | adr(y), total, [&](auto V, auto I) {
        constexpr int v = decltype(V)::value;
        launch(V, I, (decltype(I))(total / v), c / v, grid_for(total / v));
    });
}

extern "C" int lbm_nn_pool2(const void* x, int n, int d, int h, int w, int c, void* y, void* stream) {
    if (!x || !y || (d | h | w) & 1) return fail(LBM_ERR_ARG, "lbm_nn_pool2: bad arguments");
    over_cells(x, n, d / 2, h / 2, w / 2, c, y, [&](auto V, auto I, auto total, int groups, unsigned grid) {
        k_down2<decltype(V)::value, decltype(I), true><<<grid, 256, 0, S(stream)>>>(
            static_cast<const bf16*>(x), total, d / 2, h / 2, w / 2, groups, static_cast<bf16*>(y));
    });
    return check(cudaGetLastError(), "k_down2 launch");
}

extern "C" int lbm_nn_pool2_bwd(const void* dy, int n, int d, int h, int w, int c, void* dx, void* stream) {
    if (!dy || !dx || (d | h | w) & 1) return fail(LBM_ERR_ARG, "lbm_nn_pool2_bwd: bad arguments");
    over_cells(dy, n, d, h, w, c, dx, [&](auto V, auto I, auto total, int groups, unsigned grid) {
        k_up2<decltype(V)::value, decltype(I), true><<<grid, 256, 0, S(stream)>>>(
            static_cast<const bf16*>(dy), total, d, h, w, groups, static_cast<bf16*>(dx));
    });
    return check(cudaGetLastError(), "k_up2 launch");
}

extern "C" int lbm_nn_up2(const void* x, int n, int d, int h, int w, int c, void* y, void* stream) {
    if (!x || !y) return fail(LBM_ERR_ARG, "lbm_nn_up2: NULL");
    over_cells(x, n, 2 * d, 2 * h, 2 * w, c, y, [&](auto V, auto I, auto total, int groups, unsigned grid) {
        k_up2<decltype(V)::value, decltype(I), false><<<grid, 256, 0, S(stream)>>>(
            static_cast<const bf16*>(x), total, 2 * d, 2 * h, 2 * w, groups, static_cast<bf16*>(y));
    });
    return check(cudaGetLastError(), "k_up2 launch");
}

extern "C" int lbm_nn_up2_bwd(const void* dy, int n, int d, int h, int w, int c, void* dx, void* stream) {
    if (!dy || !dx) return fail(LBM_ERR_ARG, "lbm_nn_up2_bwd: NULL");
    over_cells(dy, n, d, h, w, c, dx, [&](auto V, auto I, auto total, int groups, unsigned grid) {
        k_down2<decltype(V)::value, decltype(I), false><<<grid, 256, 0, S(stream)>>>(
            static_cast<const bf16*>(dy), total, d, h, w, groups, static_cast<bf16*>(dx));
    });
    return check(cudaGetLastError(), "k_down2 launch");
}

extern "C" int lbm_nn_concat(const void* a, int ca, const void* b, int cb, size_t voxels, void* y, void* stream) {
    if (!a || !b || !y) return fail(LBM_ERR_ARG, "lbm_nn_concat: NULL");
    const size_t total = voxels * (ca + cb);
    by_width((unsigned)(ca | cb), adr(a) | adr(b) | adr(y), total, [&](auto V, auto I) {
        constexpr int v = decltype(V)::value;
        k_concat<v, decltype(I)><<<grid_for(total / v), 256, 0, S(stream)>>>(
            static_cast<const bf16*>(a), ca / v, static_cast<const bf16*>(b), cb / v, (decltype(I))(total / v),
            static_cast<bf16*>(y));
    });
    return check(cudaGetLastError(), "k_concat launch");
}

extern "C" int lbm_nn_split(const void* y, int ca, int cb, size_t voxels, void* a, void* b, void* stream) {
    if (!y) return fail(LBM_ERR_ARG, "lbm_nn_split: NULL");
    const size_t total = voxels * (ca + cb);
    by_width((unsigned)(ca | cb), adr(a) | adr(b) | adr(y), total, [&](auto V, auto I) {
        constexpr int v = decltype(V)::value;
        k_split<v, decltype(I)><<<grid_for(total / v), 256, 0, S(stream)>>>(
            static_cast<const bf16*>(y), ca / v, cb / v, (decltype(I))(total / v), static_cast<bf16*>(a),
            static_cast<bf16*>(b));
    });
    return check(cudaGetLastError(), "k_split launch");
}

extern "C" int lbm_nn_mse(const float* pred, const float* target, const uint8_t* mask, size_t voxels, int c,
                          size_t count, double* loss, void* dpred, void* stream) {
    if (!pred || !target || !mask || !loss || !dpred || c < 1) return fail(LBM_ERR_ARG, "lbm_nn_mse: bad arguments");
    const float inv = count ? 1.f / ((float)count * c) : 0.f;
    LBM_CUDA_TRY(cudaMemsetAsync(loss, 0, sizeof(double), S(stream)));
    const size_t total = voxels * c;
    if (total < (1ull << 31))
        k_mse<unsigned><<<grid_for(total), 256, 0, S(stream)>>>(pred, target, mask, (unsigned)total, c, inv, loss,
                                                                static_cast<bf16*>(dpred));
    else
        k_mse<unsigned long long><<<grid_for(total), 256, 0, S(stream)>>>(pred, target, mask, total, c, inv, loss,
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
    by_width(0, adr(a) | adr(b) | adr(y), count, [&](auto V, auto I) {
        constexpr int v = decltype(V)::value;
        k_add<v, decltype(I)><<<grid_for(count / v), 256, 0, S(stream)>>>(
            static_cast<const bf16*>(a), static_cast<const bf16*>(b), (decltype(I))(count / v), (int)(count % v),
            static_cast<bf16*>(y));
    });
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
