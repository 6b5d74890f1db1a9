// nn_tc.cu -- GEMMs of the learned warm start on the 5th-generation tensor
// cores (tcgen05): operands staged in shared memory by the block's threads,
// the FP32 accumulator in tensor memory (TMEM), one thread issuing the MMAs
// and an mbarrier reporting their completion.  A plain BF16 GEMM, the 3x3x3
// convolution (as an implicit GEMM, and reading a shared-memory halo tile)
// and its weight gradient (reducing over the voxels of such tiles).  See
// include/lbm_nn.h.
#include <cuda_bf16.h>

#include <cstdint>
#include <mutex>
#include <type_traits>

#include "internal.h"
#include "lbm_nn.h"
#include "tc.cuh"

namespace lbm {
namespace nn {

using bf16 = __nv_bfloat16;

__device__ unsigned g_tc_timeouts;  // blocks of the tensor-core kernels whose waits ran out

constexpr int TC_M = 128;                        // rows per block = accumulator lanes
constexpr int TC_BK = 64;                        // reduction depth of one stage: four K = 16 MMAs
constexpr uint32_t TC_KGAP = 128;                // core matrices adjacent along K (leading byte offset)
constexpr uint32_t TC_RGAP = (TC_BK / 8) * 128;  // 8-row groups (stride byte offset)
constexpr uint32_t TC_WAIT = 1u << 24;           // polls before a wait gives up

__host__ __device__ constexpr uint32_t tc_stage_bytes(int n) { return (uint32_t)(TC_M + n) * TC_BK * 2; }
constexpr int TC_STAGES = 3;  // operand stages in flight

// The pipeline of one block: `nk` stages of depth 64 in a ring of TC_STAGES
// shared-memory buffers.  fill(a, b, kc) stages A (128 x 64) and B (n x 64),
// K-major, 16-byte row segments at tc::tile_off, with cp.async or plain
// stores; the copies of the next TC_STAGES - 1 stages are in flight while the
// tensor cores work on the current one.  Thread 0 issues a stage's four MMAs
// into the TMEM accumulator and commits them to the stage's mbarrier; a
// buffer is refilled once the MMAs that read it have completed.  Then every
// thread reads its accumulator row, 16 columns at a time, into
// out(row_in_tile, first_column, values, ok).  `n` is a multiple of 16 in
// 16 .. 256.
template <class Fill, class Out>
__device__ __forceinline__ void tc_pipeline(unsigned char* smem, uint64_t* mbar, uint32_t* tmem_slot, int n, int nk,
                                            Fill fill, Out out) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t a_bytes = TC_M * TC_BK * 2;
    const uint32_t stage_bytes = tc_stage_bytes(n);
    uint32_t ncols = 32;
    while (ncols < (uint32_t)n) ncols <<= 1;
    if (warp == 0) tc::tmem_alloc(tmem_slot, ncols);
    if (tid == 0)
        for (int s = 0; s < TC_STAGES; s++) tc::mbar_init(&mbar[s], 1);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    const uint32_t idesc = tc::idesc_bf16_f32(TC_M, n);
    bool ok = true;
    // one cp.async group per stage, empty past the end, so that "all but the
    // newest TC_STAGES - 2 groups complete" always means "this stage landed"
    for (int p = 0; p < TC_STAGES - 1; p++) {
        if (p < nk) fill(smem + p * stage_bytes, smem + p * stage_bytes + a_bytes, p);
        tc::cp_async_commit();
    }
    for (int kc = 0; kc < nk; kc++) {
        const int s = kc % TC_STAGES;
        unsigned char* sa = smem + s * stage_bytes;
        tc::cp_async_wait<TC_STAGES - 2>();
        tc::fence_smem_to_async();
        __syncthreads();
        if (tid == 0) {
            tc::fence_after_sync();
            const uint32_t a0 = tc::smem_u32(sa), b0 = a0 + a_bytes;
#pragma unroll
            for (int j = 0; j < TC_BK / 16; j++)
                tc::mma_bf16(tmem, tc::smem_desc(a0 + 2 * j * TC_KGAP, TC_KGAP, TC_RGAP),
                             tc::smem_desc(b0 + 2 * j * TC_KGAP, TC_KGAP, TC_RGAP), idesc, kc > 0 || j > 0);
            tc::mma_commit(&mbar[s]);
        }
        // refill the buffer of stage kc - 1 with stage kc + TC_STAGES - 1, once its MMAs are done
        const int nxt = kc + TC_STAGES - 1;
        if (nxt < nk) {
            const int r = nxt % TC_STAGES;
            if (kc >= 1) ok &= tc::mbar_wait(&mbar[r], ((kc - 1) / TC_STAGES) & 1, TC_WAIT);
            fill(smem + r * stage_bytes, smem + r * stage_bytes + a_bytes, nxt);
        }
        tc::cp_async_commit();
    }
    // the last commit arrives once every MMA of the block has completed
    const int last = nk - 1;
    bool done = tc::mbar_wait(&mbar[last % TC_STAGES], (last / TC_STAGES) & 1, TC_WAIT);
    if (!done) done = tc::mbar_wait(&mbar[last % TC_STAGES], (last / TC_STAGES) & 1, TC_WAIT);
    ok &= done;
    tc::cp_async_wait<0>();
    if (!ok && lane == 0) atomicAdd(&g_tc_timeouts, 1u);
    tc::fence_after_sync();
    for (int c0 = 0; c0 < n; c0 += 16) {
        float v[16];
        tc::tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
        out(warp * 32 + lane, c0, v, ok);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, ncols);
    }
}

// C[m][n] = sum_k A[m][k] B[n][k]: A, B BF16 with K contiguous, C FP32;
// M % 128 == 0, N % 16 == 0 (16 .. 256), K % 64 == 0.
__global__ void __launch_bounds__(128) k_gemm_tc(const bf16* __restrict__ A, const bf16* __restrict__ B,
                                                 float* __restrict__ C, int N, int K) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ uint64_t mbar[TC_STAGES];
    __shared__ uint32_t tmem_slot;
    const int m0 = blockIdx.x * TC_M;
    auto fill = [&](unsigned char* sa, unsigned char* sb, int kc) {
        for (int e = threadIdx.x; e < TC_M * 8; e += 128) {
            const int r = e >> 3, g = e & 7;
            tc::cp_async16(sa + tc::tile_off(r, g, TC_KGAP, TC_RGAP), A + (size_t)(m0 + r) * K + kc * TC_BK + g * 8,
                           true);
        }
        for (int e = threadIdx.x; e < N * 8; e += 128) {
            const int r = e >> 3, g = e & 7;
            tc::cp_async16(sb + tc::tile_off(r, g, TC_KGAP, TC_RGAP), B + (size_t)r * K + kc * TC_BK + g * 8, true);
        }
    };
    auto out = [&](int r, int c0, float (&v)[16], bool ok) {
#pragma unroll
        for (int k = 0; k < 16; k++) C[(size_t)(m0 + r) * N + c0 + k] = ok ? v[k] : __int_as_float(0x7fc00000);
    };
    tc_pipeline(smem, mbar, &tmem_slot, N, K / TC_BK, fill, out);
}

// 16 output channels from co0 of one voxel: their bias (in shared memory), ReLU,
// and the stores that the tensors allow (vy: 8, 4, 2 or 1 values of y at a time, vy32: 16 bytes of y32, else value by
// value: a row of 100 channels by single values took 12 -> 100 channels on 7 x 27 x 42 x 24 voxels from 362 us to 443);
// `at`: offset of (voxel, co0).  NaN where the sums are not there, with or without ReLU.
__device__ __forceinline__ void conv_out(float (&v)[16], bool ok, const float* bias, int relu, int co0,
                                         int Cout, size_t at, int vy, bool vy32, bf16* __restrict__ y,
                                         float* __restrict__ y32) {
#pragma unroll
    for (int k = 0; k < 16; k++) {
        v[k] += bias[k];
        if (relu) v[k] = fmaxf(v[k], 0.f);
        if (!ok) v[k] = __int_as_float(0x7fc00000);
    }
    if (y) {
        uint32_t h[8];
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const __nv_bfloat162 p = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
            h[j] = *reinterpret_cast<const uint32_t*>(&p);
        }
        if (vy == 8) {
#pragma unroll
            for (int k = 0; k < 16; k += 8)
                if (co0 + k < Cout)
                    *reinterpret_cast<uint4*>(y + at + k) = make_uint4(h[k / 2], h[k / 2 + 1], h[k / 2 + 2], h[k / 2 + 3]);
        } else if (vy == 4) {
#pragma unroll
            for (int k = 0; k < 16; k += 4)
                if (co0 + k < Cout) *reinterpret_cast<uint2*>(y + at + k) = make_uint2(h[k / 2], h[k / 2 + 1]);
        } else if (vy == 2) {
#pragma unroll
            for (int k = 0; k < 16; k += 2)
                if (co0 + k < Cout) *reinterpret_cast<uint32_t*>(y + at + k) = h[k / 2];
        } else {
#pragma unroll
            for (int k = 0; k < 16; k++)
                if (co0 + k < Cout) y[at + k] = __ushort_as_bfloat16((unsigned short)(h[k / 2] >> (k % 2 * 16)));
        }
    }
    if (y32 && vy32) {
#pragma unroll
        for (int k = 0; k < 16; k += 4)
            if (co0 + k < Cout) *reinterpret_cast<float4*>(y32 + at + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
    } else if (y32) {
#pragma unroll
        for (int k = 0; k < 16; k++)
            if (co0 + k < Cout) y32[at + k] = v[k];
    }
}

// Neighbour coordinate along one axis: zero padding (-1 outside) or periodic.
__device__ __forceinline__ int tc_nb(int c, int d, int n, bool wrap) {
    c += d;
    if (wrap) return c < 0 ? c + n : (c >= n ? c - n : c);
    return (c < 0 || c >= n) ? -1 : c;
}

// The 3x3x3 convolution of lbm_nn_conv3d as an implicit GEMM, for input
// channels that do not fill K = 16 steps of one tap (Cin % 16 != 0):
// y[p][co] = act(sum_k A[p][k] B[co][k] + bias[co]) with k = (tap, ci),
// A[p][(tap, ci)] = x[p + off(tap)][ci] (zero outside, or wrapped on the axes
// of `wrap`) and B[co][(tap, ci)] = wgt[tap][ci][co].  One block computes 128
// voxels x NT output channels from blockIdx.y * NT, NT % 16 == 0.  A is read G
// channels at a time: 8 (Cin % 8 == 0, 16-byte aligned) or 2 (even Cin, 4-byte
// aligned).  Rows k >= 27 Cin of the last stage are zero; `n_stages` stages
// are reserved.
//
// Bound by the addresses and the latency of the gathers.
template <int G>
__global__ void __launch_bounds__(128) k_conv_tc(const bf16* __restrict__ x, int N, int D, int H, int W, int Cin,
                                                 const bf16* __restrict__ wgt, const float* __restrict__ bias,
                                                 int Cout, int NT, int relu, int wrap, int vy, bool vy32,
                                                 bf16* __restrict__ y, float* __restrict__ y32) {
    static_assert(G == 8 || G == 2, "16- or 4-byte loads");
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ uint64_t mbar[TC_STAGES];
    __shared__ uint32_t tmem_slot;
    const long long M = (long long)N * D * H * W;
    const int K = 27 * Cin;
    const long long m0 = (long long)blockIdx.x * TC_M;
    const int n0 = blockIdx.y * NT;
    const bool wx = wrap & 1, wy = wrap & 2, wz = wrap & 4;
    // voxel (n, z, y, x) of each of the block's rows (n < 0: past the end)
    __shared__ int4 vox[TC_M];
    __shared__ float sbias[128];
    sbias[threadIdx.x] = bias && n0 + (int)threadIdx.x < Cout ? bias[n0 + threadIdx.x] : 0.f;
    {
        const long long p = m0 + threadIdx.x;
        int4 c = make_int4(-1, 0, 0, 0);
        if (p < M) {
            long long t = p;
            c.w = (int)(t % W);
            t /= W;
            c.z = (int)(t % H);
            t /= H;
            c.y = (int)(t % D);
            c.x = (int)(t / D);
        }
        vox[threadIdx.x] = c;
    }
    __syncthreads();
    // source of channel ci of tap `tap` for voxel c; null: zero
    auto source = [&](const int4& c, int tap, int ci) -> const bf16* {
        if (c.x < 0) return nullptr;
        const int zz = tc_nb(c.y, tap / 9 - 1, D, wz), yy = tc_nb(c.z, (tap / 3) % 3 - 1, H, wy),
                  xx = tc_nb(c.w, tap % 3 - 1, W, wx);
        return (zz | yy | xx) < 0 ? nullptr : x + ((((long long)c.x * D + zz) * H + yy) * W + xx) * Cin + ci;
    };
    // a thread fills K group g = tid % 8 of rows tid / 8 + 16 j, j = 0 .. 7
    auto fill = [&](unsigned char* sa, unsigned char* sb, int kc) {
        const int g = threadIdx.x & 7;
        const int k0 = kc * TC_BK + g * 8;
        int tap[8 / G], ci[8 / G];
#pragma unroll
        for (int q = 0; q < 8 / G; q++) {
            const int k = k0 + q * G;
            tap[q] = k < K ? k / Cin : -1;
            ci[q] = k - tap[q] * Cin;
        }
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const int r = (threadIdx.x >> 3) + 16 * j;
            const int4 c = vox[r];
            unsigned char* dst = sa + tc::tile_off(r, g, TC_KGAP, TC_RGAP);
            if constexpr (G == 8) {
                const bf16* src = tap[0] >= 0 ? source(c, tap[0], ci[0]) : nullptr;
                tc::cp_async16(dst, src ? src : x, src != nullptr);  // a zero fill reads nothing
            } else {
                uint32_t h[4];
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const bf16* src = tap[q] >= 0 ? source(c, tap[q], ci[q]) : nullptr;
                    h[q] = src ? __ldg(reinterpret_cast<const uint32_t*>(src)) : 0u;
                }
                *reinterpret_cast<uint4*>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
            }
        }
        // B[co][k] from wgt[k][co], 8 consecutive k of one co per 16-byte row segment
        const unsigned short* wv = reinterpret_cast<const unsigned short*>(wgt);
        for (int e = threadIdx.x; e < NT * 8; e += 128) {
            const int co = n0 + e % NT, gk = e / NT;
            unsigned short h[8];
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const int kk = kc * TC_BK + gk * 8 + k;
                h[k] = kk < K && co < Cout ? __ldg(wv + (size_t)kk * Cout + co) : 0;
            }
            *reinterpret_cast<uint4*>(sb + tc::tile_off(e % NT, gk, TC_KGAP, TC_RGAP)) =
                make_uint4(h[0] | (uint32_t)h[1] << 16, h[2] | (uint32_t)h[3] << 16, h[4] | (uint32_t)h[5] << 16,
                           h[6] | (uint32_t)h[7] << 16);
        }
    };
    auto out = [&](int r, int c0, float (&v)[16], bool ok) {
        const long long row = m0 + r;
        const int co0 = n0 + c0;
        if (row >= M || co0 >= Cout) return;
        conv_out(v, ok, sbias + c0, relu, co0, Cout, (size_t)row * Cout + co0, vy, vy32, y, y32);
    };
    tc_pipeline(smem, mbar, &tmem_slot, NT, (K + TC_BK - 1) / TC_BK, fill, out);
}

constexpr int HX = 10, HY = 18;      // halo tile extent in x and y
constexpr int HPLANE = HX * HY;      // cells of one z plane of the tile
constexpr int HMB_MAX = 16;          // z planes of a brick, at most
constexpr int HZ_MAX = HMB_MAX + 2;  // planes of a halo tile, at most

// Halo-tile coordinate c (the box's coordinate, possibly -1 .. n) along an
// axis of n voxels: periodic or zero padding; -1 (a zero cell) as well beyond
// one voxel past either edge, where only rows outside the box would read it.
__device__ __forceinline__ int halo_nb(int c, int n, bool wrap) {
    if (c < -1 || c > n) return -1;
    if (wrap) return c < 0 ? c + n : (c >= n ? c - n : c);
    return (c < 0 || c >= n) ? -1 : c;
}

// ---- copies of bricks and their halos by warp-specialised blocks -------------
//
// Where the tiles of a block lie: bricks of 8 x 16 x mb voxels, x fastest.
struct Brick {
    int x0, y0, z0, n;
};
__device__ __forceinline__ Brick brick_at(long long t, int BX, int BY, int BZ, int mb) {
    Brick b;
    b.x0 = (int)(t % BX) * 8;
    t /= BX;
    b.y0 = (int)(t % BY) * 16;
    t /= BY;
    b.z0 = (int)(t % BZ) * mb;
    b.n = (int)(t / BZ);
    return b;
}

constexpr int FILL_THREADS = 256;  // copying threads of a block (eight warps)

// The source of a brick's halo cells along each axis, one entry per tile
// coordinate: the plane's address (null: a plane of zeros) and voxel offsets
// within the plane (negative: a zero cell).  The copying threads write it once
// per brick; a cell's address is then two additions and a multiplication
// (recomputed per cell from its coordinates, the copies took 0.7 to 1 us per
// 16 bytes and thread, more than the MMAs they fed).
struct HaloAxes {
    const bf16* z[HZ_MAX];
    long long y[HY];
    int x[HX];
};

__device__ __forceinline__ void halo_axes(HaloAxes& ax, int ft, const bf16* src, const Brick& b, int mb, int D, int H,
                                          int W, int C, int wrap) {
    if (ft < HX) ax.x[ft] = halo_nb(b.x0 + ft - 1, W, wrap & 1);
    const int yi = ft - 32;
    if (yi >= 0 && yi < HY) {
        const int yy = halo_nb(b.y0 + yi - 1, H, wrap & 2);
        ax.y[yi] = yy < 0 ? -1 : (long long)yy * W;
    }
    const int zi = ft - 64;
    if (zi >= 0 && zi < mb + 2) {
        const int zz = halo_nb(b.z0 + zi - 1, D, wrap & 4);
        ax.z[zi] = zz < 0 ? nullptr : src + (size_t)((long long)b.n * D + zz) * H * W * C;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(FILL_THREADS) : "memory");
}

// Copies planes z0 .. z1 - 1 of the halo tile, channels c0 .. c0 + 8 ncg - 1,
// to [z][channel group][y][x] cells of 16 bytes at `dst`, `plane` cells from
// one (z, channel group) plane to the next: cp.async (VEC: C % 8 == 0, 16-byte
// aligned source), else value by value.  Lanes run over the channel groups of
// a cell first, then over the cells of a line.
template <bool VEC>
__device__ __forceinline__ void fill_halo(unsigned char* dst, const HaloAxes& ax, const bf16* any, int ft, int ncg,
                                          int z0, int z1, int plane, int c0, int C) {
    const int step = FILL_THREADS / ncg, cell0 = ft / ncg, cg = ft - cell0 * ncg;
    int hx = cell0 % HX, hy = cell0 / HX % HY, hz = cell0 / HPLANE;
    const int sx = step % HX, sy = step / HX % HY, sz = step / HPLANE;
    const int ci = c0 + cg * 8, cells = (z1 - z0) * HPLANE;
    const bool cin = ci < C;
#pragma unroll 4
    for (int e = cell0 < step ? cell0 : cells; e < cells; e += step) {
        const bf16* zp = ax.z[z0 + hz];
        const long long yo = ax.y[hy];
        const int xo = ax.x[hx];
        const bool get = zp && yo >= 0 && xo >= 0 && cin;
        const bf16* src = zp + (yo + xo) * C + ci;
        unsigned char* to = dst + (uint32_t)((hz * ncg + cg) * plane + hy * HX + hx) * 16u;
        if constexpr (VEC) {
            tc::cp_async16(to, get ? src : any, get);
        } else {
            uint4 v = make_uint4(0, 0, 0, 0);
            if (get) v = tc::load8(src, C - ci);
            *reinterpret_cast<uint4*>(to) = v;
        }
        hx += sx;
        hy += sy;
        hz += sz;
        if (hx >= HX) hx -= HX, hy++;
        if (hy >= HY) hy -= HY, hz++;
    }
}

// ---- the 3x3x3 convolution ----------------------------------------------------
//
// y[p][co] = act(sum_{tap, ci} x[p + off(tap)][ci] wgt[tap][ci][co] + bias[co])
// with the activations read by the tensor cores straight from halo planes (no
// im2col copy), Cin % 16 == 0.  A brick of 8 (x) x 16 (y) x mb (z) voxels has
// one accumulator of 128 rows (x fastest) by nt output channels per z plane,
// the planes side by side in TMEM.  Input channels come in chunks of 64 (the
// last one may be shorter).  A stage holds a few input planes of the brick's
// halo, 10 x 18 cells of 8 channels per [z][channel group]: the 8 voxels of a
// brick line are one core matrix, and a tap is a start address.  The weights of
// a chunk stay in shared memory in nine slots, one per (dy, dx): per 16
// channels the 3 nt columns (dz = 2, 1, 0; co).  Input plane z of the tile adds
// to the output planes z - 2, z - 1 and z with its dz = 2, 1 and 0 taps: their
// accumulators are neighbours, so one MMA of N = 3 nt columns takes all three,
// and the tensor cores read an input plane 9 times instead of 27.  An output's
// sum runs in the order (chunk, dz, dy, dx, 16 channels).
//
// What bounds it: the copies of the halo planes (about 16 bytes per cycle and SM) and,
// beside them, the MMAs with their reads of 128 A rows from shared memory (an MMA of
// 128 x N x 16 takes max(N / 2, 32 + N / 4) cycles); no unit is saturated.  Before and
// after (blocks of up to four planes that copied, multiplied and stored in turn, 27
// MMAs per plane): 48 -> 16 channels on 8 x 64^3 voxels 639 and 218 us, 96 -> 32 on 8
// x 32^3 292 and 88, 192 -> 64 on 8 x 16^3 149 and 51, 192 -> 128 on 8 x 48^3 6411 and
// 1300; 16 -> 16 on 8 x 64^3, bound by its outputs, 136 and 129.
//
// Blocks are persistent: each keeps one tile of output channels and walks over
// bricks.  One warp issues the MMAs, eight copy the planes (the stages that
// shared memory holds in flight), one the weights (bulk copies, slot by slot as
// the last plane of a chunk releases them), eight write the outputs plane by
// plane as they complete, while the next brick uses the other of two accumulator
// sets.
constexpr int CV_STAGES = 8;
constexpr int CV_CC = 64;    // input channels per chunk
constexpr int CV_EPI = 256;  // output threads (two warps per TMEM lane quadrant)
constexpr int CV_THREADS = 32 + CV_EPI + FILL_THREADS + 32;

struct CvShape {
    int nt;      // output channels per block: a multiple of 16 up to 64
    int mb;      // z planes of a brick
    int chunks;  // ceil(Cin / 64)
    int planes;  // input planes per stage
    int pc;      // cells from one (z, channel group) plane to the next
    int stages;
    uint32_t slot_bytes, stage_bytes, smem, ncols;
};

// False where two stages or two accumulator sets do not fit.
static bool cv_shape(int cin, int nt, int mb, CvShape* s) {
    s->nt = nt;
    s->mb = mb;
    s->chunks = (cin + CV_CC - 1) / CV_CC;
    const int cc = cin < CV_CC ? cin : CV_CC, ncg = cc / 8;
    s->planes = CV_CC / cc;
    // strides that put the cells a warp stores together into different banks
    s->pc = ncg == 2 ? HPLANE : (ncg == 4 ? HPLANE + 2 : HPLANE + 1);
    s->slot_bytes = (uint32_t)(cc * 6 * nt);
    s->stage_bytes = (uint32_t)(s->planes * ncg * s->pc * 16 + 127) / 128 * 128;
    const uint32_t all = 224u * 1024u, b = 9 * s->slot_bytes;
    s->stages = b < all ? (int)((all - b) / s->stage_bytes) : 0;
    if (s->stages > CV_STAGES) s->stages = CV_STAGES;
    s->smem = b + (uint32_t)s->stages * s->stage_bytes;
    s->ncols = 32;
    while ((int)s->ncols < 2 * mb * nt) s->ncols <<= 1;
    return s->stages >= 2 && s->ncols <= 512;
}

// 16-byte units of the weights of a chunk of cc input channels: [(dy, dx)][cc /
// 16][8-channel group][dz = 2, 1, 0][co], 8 consecutive input channels each,
// zero past Cout.
__device__ __forceinline__ uint4 cv_weights(const bf16* __restrict__ wgt, int Cin, int Cout, int nt, int c0, int cc,
                                            int ct, int u) {
    const int col = u % (3 * nt), t = u / (3 * nt), g = t % (cc / 8), tap = (2 - col / nt) * 9 + t / (cc / 8);
    const int co = ct * nt + col % nt;
    unsigned short h[8];
    const unsigned short* w = reinterpret_cast<const unsigned short*>(wgt) + ((size_t)tap * Cin + c0 + g * 8) * Cout + co;
#pragma unroll
    for (int k = 0; k < 8; k++) h[k] = co < Cout ? __ldg(w + (size_t)k * Cout) : 0;
    return make_uint4(h[0] | (uint32_t)h[1] << 16, h[2] | (uint32_t)h[3] << 16, h[4] | (uint32_t)h[5] << 16,
                      h[6] | (uint32_t)h[7] << 16);
}

// The weights of every output tile and chunk as the blocks copy them, tile by
// tile, chunk by chunk (27 nt 16-byte units per 8 input channels).
__global__ void k_pack_weights(const bf16* __restrict__ wgt, int Cin, int Cout, int nt, int tiles,
                               uint4* __restrict__ wpack) {
    const int per_tile = 27 * nt * (Cin / 8), per_chunk = 27 * nt * (CV_CC / 8);
    const long long total = (long long)tiles * per_tile;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const int ct = (int)(e / per_tile), in = (int)(e - (long long)ct * per_tile), c = in / per_chunk;
        const int c0 = c * CV_CC, cc = Cin - c0 < CV_CC ? Cin - c0 : CV_CC;
        wpack[e] = cv_weights(wgt, Cin, Cout, nt, c0, cc, ct, in - c * per_chunk);
    }
}

// The MMAs of (dy, dx) tap t of input plane hz (a: its descriptor, at the tap's
// offset; b: the tap's slot), ks steps of 16 channels, into the accumulators of
// the output planes hz - 2 .. hz that the brick of nz planes has; called by one
// lane.  `first`: the plane's first MMAs of the brick's first chunk, which
// overwrite the accumulator of plane hz.
__device__ __forceinline__ void cv_issue(uint32_t acc, uint64_t a, uint64_t b, int hz, int nz, int nt, int ks, int pc,
                                         bool first) {
    const int lo = hz < 2 ? 0 : hz - 2, hi = hz < nz ? hz : nz - 1;  // output planes
    const uint64_t bo = b + (uint64_t)((lo - hz + 2) * nt);
    const uint32_t d = acc + (uint32_t)(lo * nt);
    const uint32_t id = tc::idesc_bf16_f32(TC_M, (hi - lo + 1) * nt);
    int k = 0;
    if (first && hz < nz) {
        if (hz > lo) tc::mma_bf16(d, a, bo, tc::idesc_bf16_f32(TC_M, (hz - lo) * nt), true);
        tc::mma_bf16(acc + (uint32_t)(hz * nt), a, b + (uint64_t)(2 * nt), tc::idesc_bf16_f32(TC_M, nt), false);
        k = 1;
    }
    for (; k < ks; k++) tc::mma_bf16(d, a + (uint64_t)(k * 2 * pc), bo + (uint64_t)(k * 6 * nt), id, true);
}

// Grid: x = bricks (blockIdx.x, + gridDim.x, ..), y = output-channel tiles.
// wpack NULL (few weights, or no room for it): weights of one chunk are gathered by
// the whole block before it starts, those of several by the weights' warp.
template <bool VX>
__global__ void __launch_bounds__(CV_THREADS, 1) k_conv_halo(const bf16* __restrict__ x, int N, int D, int H, int W, int Cin,
                                                             const bf16* __restrict__ wgt, const uint4* __restrict__ wpack,
                                                             const float* __restrict__ bias, int Cout, int relu, int wrap,
                                                             CvShape sh, int vy, bool vy32, bf16* __restrict__ y,
                                                             float* __restrict__ y32) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ HaloAxes axes[2];
    __shared__ uint64_t full[CV_STAGES], empty[CV_STAGES], wfull[9], wempty[9], accf[2][HMB_MAX], acce[2], done;
    __shared__ float sbias[64];
    __shared__ uint32_t tmem_slot;
    __shared__ int stop[2];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int BX = (W + 7) / 8, BY = (H + 15) / 16, BZ = (D + sh.mb - 1) / sh.mb;
    const long long tiles = (long long)N * BZ * BY * BX;
    unsigned char* const ring = smem + 9 * sh.slot_bytes;
    if (warp == 0) tc::tmem_alloc(&tmem_slot, sh.ncols);
    if (tid >= 64 && tid < 128) {
        const int co = blockIdx.y * sh.nt + tid - 64;
        sbias[tid - 64] = bias && co < Cout ? bias[co] : 0.f;
    }
    if (tid == 0) {
        for (int s = 0; s < sh.stages; s++) {
            tc::mbar_init(&full[s], FILL_THREADS / 32);
            tc::mbar_init(&empty[s], 1);
        }
        for (int t = 0; t < 9; t++) {
            tc::mbar_init(&wfull[t], 1);
            tc::mbar_init(&wempty[t], 1);
        }
        for (int s = 0; s < 2; s++) {
            for (int m = 0; m < sh.mb; m++) tc::mbar_init(&accf[s][m], 1);
            tc::mbar_init(&acce[s], CV_EPI / 32);
        }
        tc::mbar_init(&done, 1);
        stop[0] = stop[1] = 0;
    }
    const bool held = !wpack && sh.chunks == 1;  // the weights are in their slots when the block starts
    if (held) {
        const int units = 27 * sh.nt * (Cin / 8);
#pragma unroll 2
        for (int u = tid; u < units; u += CV_THREADS)
            reinterpret_cast<uint4*>(smem)[u] = cv_weights(wgt, Cin, Cout, sh.nt, 0, Cin, blockIdx.y, u);
        tc::fence_smem_to_async();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_slot;
    bool ok = true;
    if (warp == 0) {
        // the waits' results are made uniform over the warp, so that the elected
        // lane's descriptors stay in uniform registers (a lane picked by its
        // index issues an MMA every 45 cycles at best)
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            return __all_sync(0xffffffffu, tc::mbar_wait(bar, parity, TC_WAIT));
        };
        const uint32_t wslots = tc::smem_u32(smem), rg = tc::smem_u32(ring);
        int s = 0, it = 0;
        uint32_t ph = 0, wph = 0;  // phases of the stages and of the weights' slots
        for (long long t = blockIdx.x; t < tiles && ok; t += gridDim.x, it++) {
            const Brick b = brick_at(t, BX, BY, BZ, sh.mb);
            const int nz = D - b.z0 < sh.mb ? D - b.z0 : sh.mb, buf = it & 1;
            const uint32_t acc = tmem + (uint32_t)(buf * sh.mb * sh.nt);
            if (it >= 2) ok = wait(&acce[buf], ((it >> 1) - 1) & 1);
            for (int c = 0; c < sh.chunks && ok; c++) {
                const int cc = Cin - c * CV_CC < CV_CC ? Cin - c * CV_CC : CV_CC, ks = cc / 16;
                const bool fresh = !held && (sh.chunks > 1 || it == 0);  // the weights' slots are filled anew
                for (int h0 = 0; h0 < nz + 2 && ok; h0 += sh.planes) {
                    if (!(ok = wait(&full[s], ph))) break;
                    tc::fence_after_sync();
                    const int h1 = h0 + sh.planes < nz + 2 ? h0 + sh.planes : nz + 2;
                    for (int hz = h0; hz < h1 && ok; hz++) {
                        const uint64_t a0 = tc::smem_desc(rg + s * sh.stage_bytes + (uint32_t)((hz - h0) * (cc / 8) * sh.pc) * 16,
                                                          (uint32_t)sh.pc * 16, HX * 16);
                        const uint64_t b0 = tc::smem_desc(wslots, (uint32_t)(3 * sh.nt) * 16, 128);
                        const uint64_t bt = sh.slot_bytes / 16;
                        const bool last = sh.chunks > 1 && hz == nz + 1;  // releases the slots
                        if ((hz == 0 && fresh) || last) {
                            for (int t9 = 0; t9 < 9; t9++) {
                                if (hz == 0 && fresh) {
                                    if (!(ok = wait(&wfull[t9], wph))) break;
                                    tc::fence_after_sync();
                                }
                                if (tc::elect_one()) {
                                    cv_issue(acc, a0 + (uint64_t)((t9 / 3) * HX + t9 % 3), b0 + t9 * bt, hz, nz, sh.nt, ks,
                                             sh.pc, c == 0 && t9 == 0);
                                    if (last) tc::mma_commit(&wempty[t9]);
                                }
                                __syncwarp();
                            }
                        } else if (tc::elect_one()) {
#pragma unroll
                            for (int t9 = 0; t9 < 9; t9++)
                                cv_issue(acc, a0 + (uint64_t)((t9 / 3) * HX + t9 % 3), b0 + t9 * bt, hz, nz, sh.nt, ks, sh.pc,
                                         c == 0 && t9 == 0);
                        }
                        __syncwarp();
                        // output plane hz - 2 is complete (with the last one, those that the brick lacks)
                        if (c == sh.chunks - 1 && hz >= 2 && tc::elect_one())
                            for (int m = hz - 2; m < (hz == nz + 1 ? sh.mb : hz - 1); m++) tc::mma_commit(&accf[buf][m]);
                        __syncwarp();
                    }
                    if (tc::elect_one()) tc::mma_commit(&empty[s]);
                    __syncwarp();
                    if (++s == sh.stages) s = 0, ph ^= 1;
                }
                if (fresh) wph ^= 1;
            }
        }
        // whatever ran out, the MMAs issued are over before the block gives up its TMEM and shared memory
        if (tc::elect_one()) tc::mma_commit(&done);
        __syncwarp();
        ok = (wait(&done, 0) || wait(&done, 0)) && ok;
    } else if (warp <= CV_EPI / 32) {
        const int quad = warp & 3, half = (warp - 1) >> 2, r = quad * 32 + lane;
        int it = 0;
        for (long long t = blockIdx.x; t < tiles; t += gridDim.x, it++) {
            const Brick b = brick_at(t, BX, BY, BZ, sh.mb);
            const int nz = D - b.z0 < sh.mb ? D - b.z0 : sh.mb, buf = it & 1;
            const int vx = b.x0 + (r & 7), vy_ = b.y0 + (r >> 3);
            const bool inside = vx < W && vy_ < H;
            for (int m = half; m < nz; m += 2) {
                // once a wait has run out: NaN for this and the remaining planes
                if (ok) ok = __all_sync(0xffffffffu, tc::mbar_wait(&accf[buf][m], (it >> 1) & 1, TC_WAIT));
                tc::fence_after_sync();
                const size_t at = ((((size_t)b.n * D + b.z0 + m) * H + vy_) * W + vx) * Cout;
                for (int q = 0; q < sh.nt; q += 16) {
                    __syncwarp();
                    const int co0 = blockIdx.y * sh.nt + q;
                    float v[16];
                    tc::tmem_ld16(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)((buf * sh.mb + m) * sh.nt + q), v);
                    if (inside && co0 < Cout) conv_out(v, ok, sbias + q, relu, co0, Cout, at + co0, vy, vy32, y, y32);
                }
            }
            // Every warp's arrival has to belong to this brick: a warp without a plane of it (half 1 of a brick of
            // one plane) waits for the brick's sums as well.  Arriving at once, it ran ahead of the others, and its
            // arrivals for later bricks handed over accumulators that were still being read.
            if (half >= nz && ok) ok = __all_sync(0xffffffffu, tc::mbar_wait(&accf[buf][0], (it >> 1) & 1, TC_WAIT));
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&acce[buf]);
        }
    } else if (warp <= (CV_EPI + FILL_THREADS) / 32) {
        const int ft = tid - 32 - CV_EPI;
        constexpr int LAG = 2;  // stages whose copies are in flight before the oldest is waited for
        int it = 0, fills = 0, s = 0, pending = 0;
        uint32_t ph = 0;
        bool stopped = false;
        auto hand_over = [&]() {  // the oldest pending stage: this warp's copies to it have completed
            tc::fence_smem_to_async();
            __syncwarp();
            const int o = s - pending;
            if (lane == 0) tc::mbar_arrive(&full[o < 0 ? o + sh.stages : o]);
            pending--;
        };
        auto hand_over_all = [&]() {
            tc::cp_async_wait<0>();
            while (pending > 0) hand_over();
        };
        for (long long t = blockIdx.x; t < tiles && !stopped; t += gridDim.x, it++) {
            const Brick b = brick_at(t, BX, BY, BZ, sh.mb);
            const int nz = D - b.z0 < sh.mb ? D - b.z0 : sh.mb;
            // a wait that ran out stops every copying warp behind the barrier of halo_axes
            if (!ok) stop[it & 1] = 1;
            halo_axes(axes[it & 1], ft, x, b, sh.mb, D, H, W, Cin, wrap);
            stopped = *(volatile int*)&stop[it & 1];
            if (stopped) break;
            for (int c = 0; c < sh.chunks; c++) {
                const int cc = Cin - c * CV_CC < CV_CC ? Cin - c * CV_CC : CV_CC;
                for (int h0 = 0; h0 < nz + 2; h0 += sh.planes, fills++) {
                    // while the stage is still read, first hand over those before it
                    if (fills >= sh.stages && !__all_sync(0xffffffffu, tc::mbar_test(&empty[s], ph ^ 1))) {
                        hand_over_all();
                        if (ok) ok = tc::mbar_wait(&empty[s], ph ^ 1, TC_WAIT);
                    }
                    const int h1 = h0 + sh.planes < nz + 2 ? h0 + sh.planes : nz + 2;
                    if (ok) fill_halo<VX>(ring + s * sh.stage_bytes, axes[it & 1], x, ft, cc / 8, h0, h1, sh.pc, c * CV_CC, Cin);
                    __syncwarp();
                    tc::cp_async_commit();
                    pending++;
                    if (++s == sh.stages) s = 0, ph ^= 1;
                    if (pending > LAG) {
                        tc::cp_async_wait<LAG>();
                        hand_over();
                    }
                }
            }
        }
        hand_over_all();
        ok &= !stopped;
    } else {
        uint32_t ph = 0, copies = 0;  // to the slots, in turn
        bool again = false;
        const uint4* tile = wpack ? wpack + (size_t)blockIdx.y * 27 * sh.nt * (Cin / 8) : nullptr;
        for (long long t = blockIdx.x; t < tiles && ok && !held; t += gridDim.x) {
            if (again && sh.chunks == 1) break;  // the weights stay
            for (int c = 0; c < sh.chunks && ok; c++) {
                const int c0 = c * CV_CC, cc = Cin - c0 < CV_CC ? Cin - c0 : CV_CC;
                const int units = 3 * sh.nt * (cc / 8);  // of a slot
                for (int t9 = 0; t9 < 9; t9++, copies++) {
                    if (again && !(ok = __all_sync(0xffffffffu, tc::mbar_wait(&wempty[t9], ph, TC_WAIT)))) break;
                    unsigned char* slot = smem + t9 * sh.slot_bytes;
                    if (wpack) {
                        if (lane == 0)
                            tc::bulk_copy(slot, tile + (size_t)27 * sh.nt * (c0 / 8) + (size_t)t9 * units, (uint32_t)units * 16,
                                          &wfull[t9]);
                    } else {
                        for (int u = lane; u < units; u += 32)
                            reinterpret_cast<uint4*>(slot)[u] =
                                cv_weights(wgt, Cin, Cout, sh.nt, c0, cc, blockIdx.y, t9 * units + u);
                        tc::fence_smem_to_async();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(&wfull[t9]);
                    }
                    __syncwarp();
                }
                if (again) ph ^= 1;
                again = true;
            }
        }
        // bulk copies in flight land before the block ends, also when no MMA waits for them any more
        for (uint32_t c = copies < 9 ? 0 : copies - 9; c < copies; c++)
            ok = __all_sync(0xffffffffu, tc::mbar_wait(&wfull[c % 9], (c / 9) & 1, TC_WAIT)) && ok;
    }
    if (!ok && lane == 0) atomicAdd(&g_tc_timeouts, 1u);
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, sh.ncols);
    }
}

// ---- the 3x3x3 convolution of two or four input channels ---------------------
//
// The implicit GEMM of k_conv_tc, k = (tap, ci), where 27 CI fits one operand
// tile: a block copies the halo of a column of 8 x 16 x FEW_Z voxels once, and
// each thread puts one voxel's row together from it, plane by plane.  Bound by
// the chain of a plane (rows, MMAs, outputs), which as many blocks as an SM
// holds overlap; k_conv_tc spent it on the addresses of 27 CI separate loads per
// voxel: 2 -> 16 channels on 8 x 64^3 voxels 334 and 53 us, 4 -> 16
// 615 and 86.  Small boxes take shallower columns, one plane each at the least (2 -> 16
// on 8^3 voxels 14.7 us with eight planes to a block, now 7.4; on 24^3 16.6 and 8.5).
constexpr int FEW_Z = 8;  // planes of a brick, at most
__host__ __device__ constexpr int few_groups(int ci) { return (27 * ci + 15) / 16 * 2; }  // 8-value groups of a row
__host__ __device__ constexpr uint32_t few_smem(int ci, int nt, int mb) {
    return (uint32_t)((TC_M + nt) * few_groups(ci) * 16 + (mb + 2) * HPLANE * 2 * ci);
}

template <int CI>
__global__ void __launch_bounds__(TC_M) k_conv_few(const bf16* __restrict__ x, int N, int D, int H, int W,
                                                   const bf16* __restrict__ wgt, const float* __restrict__ bias, int Cout,
                                                   int nt, int mb, int relu, int wrap, int vy, bool vy32,
                                                   bf16* __restrict__ y, float* __restrict__ y32) {
    static_assert(CI == 2 || CI == 4, "a cell of 4 or 8 bytes");
    using Cell = typename std::conditional<CI == 2, uint32_t, uint2>::type;
    constexpr int KG = few_groups(CI), K = 27 * CI;
    constexpr uint32_t RGAP = KG * 128;
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char* const sb = smem + TC_M * KG * 16;
    Cell* const halo = reinterpret_cast<Cell*>(sb + nt * KG * 16);
    __shared__ uint64_t mbar;
    __shared__ uint32_t tmem_slot;
    __shared__ float sbias[64];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n0 = blockIdx.y * nt;
    uint32_t ncols = 32;
    while (ncols < (uint32_t)nt) ncols <<= 1;
    if (warp == 0) tc::tmem_alloc(&tmem_slot, ncols);
    if (tid == 0) tc::mbar_init(&mbar, 1);
    if (tid < 64) sbias[tid] = bias && n0 + tid < Cout ? bias[n0 + tid] : 0.f;
    const unsigned short* wv = reinterpret_cast<const unsigned short*>(wgt);
    for (int e = tid; e < nt * KG; e += TC_M) {
        const int c = e % nt, g = e / nt, co = n0 + c;
        unsigned short h[8];
#pragma unroll
        for (int k = 0; k < 8; k++) h[k] = g * 8 + k < K && co < Cout ? __ldg(wv + (size_t)(g * 8 + k) * Cout + co) : 0;
        *reinterpret_cast<uint4*>(sb + tc::tile_off(c, g, TC_KGAP, RGAP)) =
            make_uint4(h[0] | (uint32_t)h[1] << 16, h[2] | (uint32_t)h[3] << 16, h[4] | (uint32_t)h[5] << 16,
                       h[6] | (uint32_t)h[7] << 16);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_slot, idesc = tc::idesc_bf16_f32(TC_M, nt);
    const int BX = (W + 7) / 8, BY = (H + 15) / 16, BZ = (D + mb - 1) / mb;
    const long long tiles = (long long)N * BZ * BY * BX;
    const int lx = tid & 7, ly = tid >> 3;
    bool ok = true;
    uint32_t ph = 0;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const Brick b = brick_at(t, BX, BY, BZ, mb);
        const int nz = D - b.z0 < mb ? D - b.z0 : mb;
#pragma unroll 4
        for (int e = tid; e < (nz + 2) * HPLANE; e += TC_M) {
            const int hx = e % HX, hy = e / HX % HY, hz = e / HPLANE;
            const int xx = halo_nb(b.x0 + hx - 1, W, wrap & 1), yy = halo_nb(b.y0 + hy - 1, H, wrap & 2),
                      zz = halo_nb(b.z0 + hz - 1, D, wrap & 4);
            Cell v{};
            if ((xx | yy | zz) >= 0)
                v = __ldg(reinterpret_cast<const Cell*>(x) + (((long long)b.n * D + zz) * H + yy) * W + xx);
            halo[e] = v;
        }
        __syncthreads();
        const int vx = b.x0 + lx, vy_ = b.y0 + ly;
        for (int z = 0; z < nz; z++) {
            Cell w[KG * 8 / CI];
#pragma unroll
            for (int k = 0; k < KG * 8 / CI; k++)
                w[k] = k < 27 ? halo[((z + k / 9) * HY + ly + k / 3 % 3) * HX + lx + k % 3] : Cell{};
#pragma unroll
            for (int g = 0; g < KG; g++) {
                uint4 u;
                if constexpr (CI == 2) u = make_uint4(w[4 * g], w[4 * g + 1], w[4 * g + 2], w[4 * g + 3]);
                else u = make_uint4(w[2 * g].x, w[2 * g].y, w[2 * g + 1].x, w[2 * g + 1].y);
                *reinterpret_cast<uint4*>(smem + tc::tile_off(tid, g, TC_KGAP, RGAP)) = u;
            }
            tc::fence_smem_to_async();
            __syncthreads();
            if (tid == 0 && ok) {
                tc::fence_after_sync();
                const uint32_t a0 = tc::smem_u32(smem), b0 = tc::smem_u32(sb);
#pragma unroll
                for (int j = 0; j < KG / 2; j++)
                    tc::mma_bf16(tmem, tc::smem_desc(a0 + 2 * j * TC_KGAP, TC_KGAP, RGAP),
                                 tc::smem_desc(b0 + 2 * j * TC_KGAP, TC_KGAP, RGAP), idesc, j > 0);
                tc::mma_commit(&mbar);
            }
            bool landed = ok;
            if (ok) landed = __all_sync(0xffffffffu, tc::mbar_wait(&mbar, ph, TC_WAIT));
            tc::fence_after_sync();
            const size_t at = ((((size_t)b.n * D + b.z0 + z) * H + vy_) * W + vx) * Cout;
            for (int q = 0; q < nt; q += 16) {
                float v[16];
                __syncwarp();
                tc::tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)q, v);
                if (vx < W && vy_ < H && n0 + q < Cout)
                    conv_out(v, landed, sbias + q, relu, n0 + q, Cout, at + n0 + q, vy, vy32, y, y32);
            }
            tc::fence_before_sync();
            // the rows and the accumulator are free; a wait that ran out in any warp stops the MMAs
            ok = __syncthreads_and(landed);
            if (ok) ph ^= 1;
            tc::fence_after_sync();
        }
    }
    if (!ok) {  // the last MMAs issued may still run
        (void)tc::mbar_wait(&mbar, ph, TC_WAIT);
        if (lane == 0) atomicAdd(&g_tc_timeouts, 1u);
        __syncthreads();
    }
    if (warp == 0) tc::tmem_dealloc(tmem, ncols);
}

// ---- weight gradient on the tensor cores ------------------------------------
//
// dw[tap][ci][co] = sum_p x[p + off(tap)][ci] dy[p][co]: GEMMs that reduce over
// the positions of a padded grid, (D + 2) x (H + 2) x Wp with Wp >= W + 2 a
// multiple of 8: position q holds x at q minus one voxel on each axis (wrapped
// on periodic axes, zero outside) and dy at interior positions (zero on the
// padding), so a tap is a shift of q by (dz Hp + dy) Wp + dx.  Both operands
// are read by the tensor cores where the channels-last tensors put them: a
// stage holds T consecutive positions as cells of 8 channels (16 bytes), dy as
// [channel group][q], x as [dz][channel group][q] with the rows that the dy and
// dx shifts reach (one window of T + 2 Wp + 2 cells, or three of T + 2 for the
// dy of wide rows).  8 consecutive cells are one core matrix of an MN-major
// operand (8 positions of K by 8 channels): no transposed or shifted copy is
// made, a tap is a start address.  The (dz, channel group) planes are one stride
// apart, so one MMA of K = 16 positions gives the sums of 3 cc (dz, ci) rows by
// NT output channels for one (dy, dx), into that tap's TMEM columns.  (Rows past
// 3 cc read whatever lies behind; their sums are not used.)  Sixteen warps copy
// the stages, one issues the MMAs; each block keeps its sums over its chunk of
// positions in TMEM and stores them once.  Stages without an interior row are left
// out.
//
// What bounds it: the tensor cores' reads of the 128 or 64 (dz, ci) rows from
// shared memory, once per (dy, dx) (an MMA of 64 x 16 x 16 takes 23 cycles, of
// 128 x 32 x 16 40), and the copies of x, three or more for its halo.
// With operands packed channel-major in memory (three copies of x) a layer wrote
// and read 4 to 8 times its tensors: 16 -> 16 channels on 8 x 64^3 voxels 1082
// us, now 157; 48 -> 16 2636, now 417; 96 -> 32 on 8 x 32^3 914, now 181; 192 ->
// 128 on 8 x 48^3 5012, now 4102; 2 -> 16 on 8 x 64^3 (gathered for mma.sync,
// 1275) 189.
constexpr int WG_FILL = 512;               // copying threads (16 warps)
constexpr int WG_THREADS = WG_FILL + 32;  // and the warp that issues the MMAs
constexpr int WG_STAGES = 4;
constexpr int WG_T = 512;                // positions of a stage, at most
constexpr int WG_ROWS = WG_T / 8 + 6;    // rows of the padded grid that a stage reaches, at most

// Shape of one launch, shared by the host and the kernel.
struct WgShape {
    int cc;       // input channels per block: 8, 16 or 32
    int ncg;      // cc / 8
    int nt;       // output channels per block: 16, 32 or 48
    int T;        // positions of a stage: a multiple of 64
    int win;      // windows of x: 1, or 3 (one per dy)
    int len;      // cells of a window
    int plane;    // cells from one (z, channel group) plane of the x tile to the next
    int gstride;  // cells from one channel group of the dy tile to the next
    int stages;   // 2 .. WG_STAGES
    uint32_t a_bytes, stage_bytes, smem, ncols;
};

// Output tiles of at most 48 channels, whose nine (dy, dx) accumulators fit the
// 512 TMEM columns.  Input channels per block: 32 (rows 3 * 32 of 128), or 16
// (3 * 16 of 64) up to 32 output channels, where the MMA of 64 rows takes little
// more than half the time (24 against 40 cycles) and twice as many blocks fill
// the chip.  Of the stage lengths and windows of which two stages fit, the one
// that copies least per position.  The plane and group strides put the 16-byte
// cells that a warp stores together (channel groups fastest) into different
// banks.
static WgShape wg_shape(int cin, int cout, int Wp) {
    WgShape best{};
    double least = 0;
    const int mt = (cout + 47) / 48;
    for (int T = WG_T; T >= 64; T -= 64)
        for (int win = 1; win <= 3; win += 2) {
            WgShape s;
            s.nt = ((cout + mt - 1) / mt + 15) / 16 * 16;
            s.cc = cin <= 8 ? 8 : (cin <= 16 || cout <= 32 || (cin % 32 && cin % 32 <= 16) ? 16 : 32);
            s.ncg = s.cc / 8;
            s.T = T;
            s.win = win;
            const long long len = T + 2 + (win == 1 ? 2ll * Wp : 0);
            if (len > 8192) continue;
            s.len = (int)len;
            const int at = s.ncg == 4 ? 2 : (s.ncg == 2 ? 4 : 0);
            s.plane = (s.len + 7 - at) / 8 * 8 + at;
            s.gstride = T + (s.nt == 16 ? 4 : (s.nt == 32 ? 2 : 1));
            s.a_bytes = (uint32_t)(win * 3 * s.ncg * s.plane) * 16;
            const uint32_t g_bytes = (uint32_t)(s.nt / 8 * s.gstride) * 16;
            s.stage_bytes = (s.a_bytes + g_bytes + 127) / 128 * 128;
            // the unused rows of an MMA reach past the last window's planes
            const uint32_t over = (uint32_t)(((3 * s.ncg > 8 ? 16 : 8) - 3 * s.ncg) * s.plane) * 16;
            const uint32_t tail = over > g_bytes ? over - g_bytes : 0;
            if (tail >= 220u * 1024u) continue;
            s.stages = (int)((220u * 1024u - tail) / s.stage_bytes);
            if (s.stages < 2) continue;
            if (s.stages > WG_STAGES) s.stages = WG_STAGES;
            s.smem = (uint32_t)s.stages * s.stage_bytes + tail;
            s.ncols = 32;
            while ((int)s.ncols < 9 * s.nt) s.ncols <<= 1;
            const double cost = (3.0 * win * s.ncg * s.len + s.nt / 8.0 * T + 400.0) / T;  // cells copied, and a stage's overhead
            if (least == 0 || cost < least) least = cost, best = s;
        }
    return best;
}

// The MMAs of one stage: ks K steps, nine (dy, dx) each (dy steps `dyoff`
// descriptor units apart); called by one lane.
__device__ __forceinline__ void wg_issue(uint32_t tmem, uint64_t a0, uint64_t g0, int ks, uint32_t dyoff, int nt,
                                         uint32_t idesc, bool first) {
    for (int k = 0; k < ks; k++) {
        const uint64_t a = a0 + (uint64_t)(k * 16), g = g0 + (uint64_t)(k * 16);
        const bool acc = !first || k > 0;
#pragma unroll
        for (int t = 0; t < 9; t++)
            tc::mma_bf16(tmem + (uint32_t)(t * nt), a + (uint64_t)((t / 3) * dyoff + t % 3), g, idesc, acc);
    }
}

// Grid: x = chunks of spc * 64 positions, y = input-channel chunks, z =
// output-channel tiles.  part[blockIdx.x][tap][ci][co] takes the block's sums
// (NaN when a wait ran out); k_sum_chunks adds the chunks to dw in order, so the
// gradient does not depend on the order in which blocks finish.
template <bool VX, bool VG>
__global__ void __launch_bounds__(WG_THREADS, 1) k_wgrad_tc(const bf16* __restrict__ x, const bf16* __restrict__ dy, int N,
                                                            int D, int H, int W, int Cin, int Cout, int wrap, int Wp,
                                                            long long nsteps, long long spc, WgShape sh,
                                                            float* __restrict__ part) {
    extern __shared__ __align__(128) unsigned char smem[];
    // sources of the padded grid's rows near a stage: x for each dz, dy (null: zeros)
    __shared__ const bf16* xrow[2][3][WG_ROWS];
    __shared__ const bf16* grow[2][WG_ROWS];
    __shared__ int used[WG_STAGES];  // the stage holds an interior row
    __shared__ uint64_t full[WG_STAGES], empty[WG_STAGES], done;
    __shared__ uint32_t tmem_slot;
    __shared__ int failed, stop[2];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int c0 = blockIdx.y * sh.cc;
    const int n0 = blockIdx.z * sh.nt;
    const int Hp = H + 2, Dp = D + 2;
    const long long begin = blockIdx.x * spc * 64, last_step = (blockIdx.x + 1) * spc,
                    end = (last_step < nsteps ? last_step : nsteps) * 64;
    if (warp == 0) tc::tmem_alloc(&tmem_slot, sh.ncols);
    if (tid == 0) {
        for (int s = 0; s < sh.stages; s++) {
            tc::mbar_init(&full[s], WG_FILL / 32);
            tc::mbar_init(&empty[s], 1);
        }
        tc::mbar_init(&done, 1);
        failed = stop[0] = stop[1] = 0;
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_slot;
    const int rows = 3 * sh.ncg > 8 ? 128 : 64;  // (dz, ci) rows of an MMA
    bool ok = true, any = false;                 // any (the issuing warp): the accumulators were written
    __shared__ int written;
    if (warp == 0) {
        // the waits' results are made uniform over the warp, so that the elected
        // lane's descriptors stay in uniform registers (a lane picked by its
        // index issues an MMA every 45 cycles at best; these need 23 to 48)
        const uint32_t idesc = tc::idesc_bf16_f32(rows, sh.nt) | tc::IDESC_MN_MAJOR;
        const uint32_t dyoff = (uint32_t)(sh.win == 1 ? Wp : 3 * sh.ncg * sh.plane);
        int s = 0;        // stage
        uint32_t ph = 0;  // its phase
        for (long long q = begin; q < end; q += sh.T) {
            if (!__all_sync(0xffffffffu, tc::mbar_wait(&full[s], ph, TC_WAIT))) {
                ok = false;
                break;
            }
            tc::fence_after_sync();
            const uint32_t st = tc::smem_u32(smem + s * sh.stage_bytes);
            const uint64_t a0 = tc::smem_desc(st, 128, (uint32_t)sh.plane * 16);
            const uint64_t g0 = tc::smem_desc(st + sh.a_bytes, 128, (uint32_t)sh.gstride * 16);
            const int ks = (int)(end - q < sh.T ? end - q : sh.T) / 16;
            if (__any_sync(0xffffffffu, used[s])) {
                if (tc::elect_one()) wg_issue(tmem, a0, g0, ks, dyoff, sh.nt, idesc, !any);
                __syncwarp();
                any = true;
            }
            if (tc::elect_one()) tc::mma_commit(&empty[s]);
            __syncwarp();
            if (++s == sh.stages) s = 0, ph ^= 1;
        }
        if (tc::elect_one()) tc::mma_commit(&done);
        __syncwarp();
        if (lane == 0) written = any;
    } else {
        const int ft = tid - 32;
        // this thread's channel groups of x and dy, its first position and the step between its positions
        const int xstep = WG_FILL / sh.ncg, xpos = ft / sh.ncg, xcg = ft - xpos * sh.ncg, ci = c0 + xcg * 8;
        const int groups = sh.nt / 8, gstep = WG_FILL / groups;
        const int gpos = ft / groups, gcg = ft - gpos * groups, co = n0 + gcg * 8;
        const int xsi = xstep / Wp, xsx = xstep - xsi * Wp, gsi = gstep / Wp, gsx = gstep - gsi * Wp;
        // row and position in it of the segment's start; rows are decoded in 32 bits where they fit
        long long row0 = begin / Wp;
        int x0 = (int)(begin - row0 * Wp);
        const int ti = sh.T / Wp, tx = sh.T - ti * Wp;
        const long long all_rows = (long long)N * Dp * Hp;
        const bool small_rows = all_rows < 0x7fffffffll;
        int it = 0, s = 0, last = -1;  // segments so far, stage, the stage copied but not handed over
        uint32_t ph = 0;
        auto hand_over = [&](int stage) {  // this warp's copies to it have completed
            tc::fence_smem_to_async();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&full[stage]);
        };
        auto hand_over_all = [&]() {
            tc::cp_async_wait<0>();
            if (last >= 0) hand_over(last);
            last = -1;
        };
        for (long long q = begin; q < end; q += sh.T, it++) {
            // with two stages the one before is handed over as soon as it has landed (the MMAs
            // would otherwise wait for the copies of this one as well), with more at the
            // latest while this one is still read; a wait that runs out stops every copying
            // warp behind the barrier below
            if (sh.stages == 2) hand_over_all();
            if (it >= sh.stages && !__all_sync(0xffffffffu, tc::mbar_test(&empty[s], ph ^ 1))) {
                hand_over_all();
                if (!tc::mbar_wait(&empty[s], ph ^ 1, TC_WAIT)) stop[it & 1] = 1;
            }
            const long long rb = row0 - 2;  // first row of the tables
            const int off = x0 + 2 * Wp;    // the segment's start from there
            const int nr = (x0 + sh.T - 1) / Wp + 5;
            for (int e = ft; e < 3 * nr; e += WG_FILL) {
                const int dz = e / nr, i = e - dz * nr;
                const long long r = rb + i + (long long)(dz - 1) * Hp;
                const bf16 *px = nullptr, *pg = nullptr;
                if (r >= 0 && r < all_rows) {
                    int yp, zp;
                    long long n;
                    if (small_rows) {
                        const unsigned u = (unsigned)r, v = u / (unsigned)Hp;
                        yp = (int)(u - v * (unsigned)Hp);
                        n = v / (unsigned)Dp;
                        zp = (int)(v - (unsigned)n * (unsigned)Dp);
                    } else {
                        yp = (int)(r % Hp);
                        zp = (int)(r / Hp % Dp);
                        n = r / Hp / Dp;
                    }
                    const int zs = halo_nb(zp - 1, D, wrap & 4), ys = halo_nb(yp - 1, H, wrap & 2);
                    if ((zs | ys) >= 0) px = x + ((n * D + zs) * H + ys) * (long long)W * Cin;
                    if (zp >= 1 && zp <= D && yp >= 1 && yp <= H) pg = dy + ((n * D + zp - 1) * H + yp - 1) * (long long)W * Cout;
                }
                xrow[it & 1][dz][i] = px;
                if (dz == 1) grow[it & 1][i] = pg;
            }
            asm volatile("bar.sync 1, %0;" ::"n"(WG_FILL) : "memory");
            if (*(volatile int*)&stop[it & 1]) {
                ok = false;
                break;
            }
            // nothing to copy or multiply where no row is interior
            bool use = false;
            for (int i = lane; i < nr; i += 32) use |= i >= 2 && i < nr - 2 && grow[it & 1][i] != nullptr;
            use = __any_sync(0xffffffffu, use);
            if (ft == 0) used[s] = use;
            if (use) {
                unsigned char* sa = smem + s * sh.stage_bytes;
                unsigned char* sg = sa + sh.a_bytes;
                const int held = end - q < sh.T ? (int)(end - q) : sh.T, cells = sh.len - (sh.T - held);  // of this segment
                for (int pl = 0; pl < 3 * sh.win; pl++) {
                    const int dz = pl % 3;
                    // position of the window's first cell from the tables' first row
                    const int rel = off - 1 + (sh.win == 1 ? -Wp : (pl / 3 - 1) * Wp) + xpos;
                    int i = rel / Wp, xp = rel - i * Wp;
                    unsigned char* to = sa + (uint32_t)((pl * sh.ncg + xcg) * sh.plane) * 16u;
#pragma unroll 4
                    for (int e = xpos < xstep ? xpos : cells; e < cells; e += xstep) {
                        const bf16* row = xrow[it & 1][dz][i];
                        const int xx = xp > W + 1 ? -1 : halo_nb(xp - 1, W, wrap & 1);
                        const bool get = row && xx >= 0 && ci < Cin;
                        const bf16* src = row + (long long)xx * Cin + ci;
                        if constexpr (VX) {
                            tc::cp_async16(to + (uint32_t)e * 16u, get ? src : x, get);
                        } else {
                            uint4 v = make_uint4(0, 0, 0, 0);
                            if (get) v = tc::load8(src, Cin - ci);
                            *reinterpret_cast<uint4*>(to + (uint32_t)e * 16u) = v;
                        }
                        xp += xsx;
                        i += xsi;
                        if (xp >= Wp) xp -= Wp, i++;
                    }
                }
                const int rel = off + gpos;
                int i = rel / Wp, xp = rel - i * Wp;
                unsigned char* to = sg + (uint32_t)(gcg * sh.gstride) * 16u;
#pragma unroll 4
                for (int e = gpos < gstep ? gpos : held; e < held; e += gstep) {
                    const bf16* row = grow[it & 1][i];
                    const bool get = row && xp >= 1 && xp <= W && co < Cout;
                    const bf16* src = row + (long long)(xp - 1) * Cout + co;
                    if constexpr (VG) {
                        tc::cp_async16(to + (uint32_t)e * 16u, get ? src : dy, get);
                    } else {
                        uint4 v = make_uint4(0, 0, 0, 0);
                        if (get) v = tc::load8(src, Cout - co);
                        *reinterpret_cast<uint4*>(to + (uint32_t)e * 16u) = v;
                    }
                    xp += gsx;
                    i += gsi;
                    if (xp >= Wp) xp -= Wp, i++;
                }
            }
            __syncwarp();
            tc::cp_async_commit();
            if (last >= 0) {  // the stage before this one has landed
                tc::cp_async_wait<1>();
                hand_over(last);
            }
            last = s;
            if (++s == sh.stages) s = 0, ph ^= 1;
            row0 += ti;
            x0 += tx;
            if (x0 >= Wp) x0 -= Wp, row0++;
        }
        hand_over_all();
    }
    bool fin = tc::mbar_wait(&done, 0, TC_WAIT);
    if (!fin) fin = tc::mbar_wait(&done, 0, TC_WAIT);
    ok &= fin;
    if (!ok && lane == 0) {
        atomicAdd(&g_tc_timeouts, 1u);
        failed = 1;
    }
    __syncthreads();
    const bool good = failed == 0, none = written == 0;  // none: sums of zero
    tc::fence_after_sync();
    if (warp > 0) {
        // row r of the accumulator lies in TMEM lane r (128 rows) or 32 (r / 16) + r % 16 (64 rows); the
        // copying warps of a lane quadrant take turns with the chunks of 16 columns
        const int quad = warp & 3, half = (warp - 1) >> 2;
        const int r = rows == 128 ? quad * 32 + lane : (lane < 16 ? quad * 16 + lane : 128);
        const int dz = r / sh.cc, ci = c0 + r % sh.cc;
        const bool mine = r < 3 * sh.cc && ci < Cin;
        for (int col = half * 16; col < 9 * sh.nt; col += 16 * (WG_FILL / 128)) {
            float v[16];
            __syncwarp();
            tc::tmem_ld16(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)col, v);
            const int t = col / sh.nt, co0 = n0 + col - t * sh.nt;
            if (!mine || co0 >= Cout) continue;
#pragma unroll
            for (int k = 0; k < 16; k++) v[k] = !good ? __int_as_float(0x7fc00000) : (none ? 0.f : v[k]);
            float* dst = part + (((size_t)blockIdx.x * 27 + dz * 9 + t) * Cin + ci) * Cout + co0;
            if (Cout % 4 == 0) {
#pragma unroll
                for (int k = 0; k < 16; k += 4)
                    if (co0 + k < Cout) *reinterpret_cast<float4*>(dst + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
            } else {
#pragma unroll
                for (int k = 0; k < 16; k++)
                    if (co0 + k < Cout) dst[k] = v[k];
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, sh.ncols);
    }
}

}  // namespace nn
}  // namespace lbm

using namespace lbm;
using namespace lbm::nn;

static int tc_launch_ok(const void* kernel, uint32_t smem, const char* what) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return e == cudaSuccess ? LBM_OK : cuda_fail(e, what);
}

extern "C" int lbm_nn_gemm_bf16(const void* a, const void* b, float* c, int m, int n, int k, void* stream) {
    if (!a || !b || !c || m < 1 || n < 16 || n > 256 || k < 1 || m % TC_M || n % 16 || k % TC_BK)
        return fail(LBM_ERR_ARG, "lbm_nn_gemm_bf16: needs m %% 128 == 0, n %% 16 == 0 in 16..256, k %% 64 == 0");
    const uint32_t smem = TC_STAGES * tc_stage_bytes(n);
    int rc = tc_launch_ok((const void*)k_gemm_tc, smem, "cudaFuncSetAttribute(k_gemm_tc)");
    if (rc) return rc;
    k_gemm_tc<<<m / TC_M, 128, smem, static_cast<cudaStream_t>(stream)>>>(static_cast<const bf16*>(a),
                                                                           static_cast<const bf16*>(b), c, n, k);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LBM_OK : cuda_fail(e, "k_gemm_tc launch");
}

namespace lbm {
namespace nn {
static int g_halo_mb = 0, g_halo_nt = 0;  // fixed by lbm_nn_conv_tune; 0 = chosen per shape

// Device memory of one call, in the order of its stream: taken before the kernel
// that writes it, given back behind the one that reads it.  Calls on other
// streams, threads and devices have memory of their own, and a call under capture
// leaves the two as nodes of its graph.  It comes from a pool per device that
// keeps up to kPoolKeep bytes between calls and gives back what is beyond them
// when the device is next synchronised.  NULL where there is no room.
class StreamBuffer {
public:
    StreamBuffer(size_t bytes, cudaStream_t s) : stream_(s) {
        if (!bytes) return;
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        cudaError_t e = cudaStreamIsCapturing(s, &cap);
        cudaMemPool_t pool = nullptr;
        if (e == cudaSuccess && cap != cudaStreamCaptureStatusNone)
            e = cudaMallocAsync(&p_, bytes, s);  // the graph's own memory, whatever the pool
        else if (e == cudaSuccess && (e = pool_of_device(&pool)) == cudaSuccess)
            e = cudaMallocFromPoolAsync(&p_, bytes, pool, s);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            p_ = nullptr;
        }
    }
    ~StreamBuffer() {
        if (p_) (void)cudaFreeAsync(p_, stream_);
    }
    StreamBuffer(const StreamBuffer&) = delete;
    StreamBuffer& operator=(const StreamBuffer&) = delete;
    void* get() const { return p_; }

private:
    static constexpr uint64_t kPoolKeep = 64ull << 20;
    static cudaError_t pool_of_device(cudaMemPool_t* pool) {
        static std::mutex lock;
        static cudaMemPool_t pools[64] = {};
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev >= 64) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> hold(lock);
        if (!pools[dev]) {
            cudaMemPoolProps props{};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            cudaMemPool_t made = nullptr;
            e = cudaMemPoolCreate(&made, &props);
            if (e != cudaSuccess) return e;
            uint64_t keep = kPoolKeep;
            int no = 0;  // memory of another stream is taken once that stream is past it, never by waiting for it
            (void)cudaMemPoolSetAttribute(made, cudaMemPoolAttrReleaseThreshold, &keep);
            (void)cudaMemPoolSetAttribute(made, cudaMemPoolReuseAllowInternalDependencies, &no);
            pools[dev] = made;
        }
        *pool = pools[dev];
        return cudaSuccess;
    }
    void* p_ = nullptr;
    cudaStream_t stream_;
};

static int sm_count() {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            (void)cudaGetLastError();
            sms = 148;
        }
    }
    return sms;
}

// The convolution of two or four input channels (x aligned to a voxel).
template <int CI>
static int conv3d_few(const void* x, int n, int d, int h, int w, const void* wgt, const float* bias, int cout, int relu,
                      int wrap, void* y, float* y32, int vy, bool vy32, cudaStream_t s) {
    const int want = (cout + 15) / 16 * 16, nt = want < 64 ? want : 64, gy = (cout + nt - 1) / nt;
    // shallower bricks while they are fewer than the SMs: a block works through its planes in turn
    const long long columns = (long long)n * ((h + 15) / 16) * ((w + 7) / 8);
    int mb = FEW_Z;
    while (mb > 1 && columns * ((d + mb - 1) / mb) * gy < sm_count()) mb /= 2;
    const long long tiles = columns * ((d + mb - 1) / mb);
    const uint32_t smem = few_smem(CI, nt, mb);
    uint32_t cols = 32;
    while (cols < (uint32_t)nt) cols <<= 1;
    long long per_sm = (224 << 10) / (smem + 2048);  // by shared memory, TMEM columns and threads
    if (per_sm > 512 / cols) per_sm = 512 / cols;
    if (per_sm > 8) per_sm = 8;
    const long long most = per_sm * sm_count(), gx = tiles < most ? tiles : most;
    if (gy > 65535) return fail(LBM_ERR_ARG, "convolution: %d output channels exceed the grid", cout);
    int rc = tc_launch_ok((const void*)k_conv_few<CI>, smem, "cudaFuncSetAttribute(k_conv_few)");
    if (rc) return rc;
    k_conv_few<CI><<<dim3((unsigned)gx, (unsigned)gy), TC_M, smem, s>>>(
        static_cast<const bf16*>(x), n, d, h, w, static_cast<const bf16*>(wgt), bias, cout, nt, mb, relu, wrap, vy, vy32,
        static_cast<bf16*>(y), y32);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LBM_OK : cuda_fail(e, "k_conv_few launch");
}

// The convolution as an implicit GEMM, an even number of input channels, x 4-byte aligned.
static int conv3d_im2col(const void* x, int n, int d, int h, int w, int cin, const void* wgt, const float* bias, int cout,
                         int relu, int wrap, void* y, float* y32, int vy, bool vy32, cudaStream_t s) {
    const int tiles = (cout + 127) / 128;
    const int nt = ((cout + tiles - 1) / tiles + 15) / 16 * 16;
    const long long M = (long long)n * d * h * w;
    const long long gx = (M + TC_M - 1) / TC_M;
    if (gx > 0x7fffffff || tiles > 65535) return fail(LBM_ERR_ARG, "convolution: grid of %lld x %d blocks", gx, tiles);
    const int nk = (27 * cin + TC_BK - 1) / TC_BK;  // a block's stages: the ring holds no more
    const uint32_t smem = (nk < TC_STAGES ? nk : TC_STAGES) * tc_stage_bytes(nt);
    auto go = [&](auto kern) -> int {
        int rc = tc_launch_ok((const void*)kern, smem, "cudaFuncSetAttribute(k_conv_tc)");
        if (rc) return rc;
        kern<<<dim3((unsigned)gx, (unsigned)((cout + nt - 1) / nt)), 128, smem, s>>>(
            static_cast<const bf16*>(x), n, d, h, w, cin, static_cast<const bf16*>(wgt), bias, cout, nt, relu, wrap, vy, vy32,
            static_cast<bf16*>(y), y32);
        const cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? LBM_OK : cuda_fail(e, "k_conv_tc launch");
    };
    if (cin % 8 == 0 && (uintptr_t)x % 16 == 0) return go(k_conv_tc<8>);
    return go(k_conv_tc<2>);
}

// Launch shape: the output-channel tile nt and brick depth mb of the least
// time by the model below, in SM cycles: bricks per block times the MMAs (9 per
// input plane and 16 channels, of 128 x 3 nt x 16) or the copies of the planes
// (near 24 bytes a cycle), whichever is longer, some cycles per plane and
// brick, and the weights at a block's start.
static CvShape cv_pick(int n, int d, int h, int w, int cin, int cout, int* grid_x) {
    CvShape best{};
    double least = 0;
    const int want = (cout + 15) / 16 * 16, most = want < 64 ? want : 64;
    for (int nt = most; nt >= 16; nt -= 16) {
        if (g_halo_nt && (nt > g_halo_nt || least > 0)) continue;  // fixed: the widest that fits, up to it
        const long long gy = (cout + nt - 1) / nt;
        for (int mb = HMB_MAX; mb >= 1; mb = mb > 4 ? mb / 2 : mb - 1) {
            CvShape s;
            if ((g_halo_mb ? mb != g_halo_mb : mb == 3) || !cv_shape(cin, nt, mb, &s)) continue;
            const long long tiles = (long long)n * ((d + mb - 1) / mb) * ((h + 15) / 16) * ((w + 7) / 8);
            long long gx = sm_count() / gy;
            if (gx < 1) gx = 1;
            if (gx > tiles) gx = tiles;
            const long long per = (tiles + gx - 1) / gx, waves = (gx * gy + sm_count() - 1) / sm_count();
            const int planes = (mb < d ? mb : d) + 2;
            const double mma = 9.0 * (cin / 16) * (1.5 * nt > 32 + 0.75 * nt ? 1.5 * nt : 32 + 0.75 * nt);
            const double copy = (double)(cin / 8) * HPLANE * 16 / 24.0;
            const double fill = 9.0 * s.slot_bytes / 40.0;  // a chunk's weights
            const double cost = (double)waves * (per * (planes * ((mma > copy ? mma : copy) + 60.0) + 800.0 * s.chunks) + 6000.0 + fill);
            if (least == 0 || cost < least) least = cost, best = s, *grid_x = (int)gx;
        }
    }
    return best;
}

// Up to so many 16-byte units of an output tile's weights (of one chunk of input
// channels) each block gathers them itself, eight rounds of its threads, instead of a
// packing launch before it: 16 -> 4 channels on 8^3 voxels 17.2 and 10.9 us, 48 -> 16
// 19.2 and 15.1, on 8 x 64^3 222 and 218; with 6912 units, 64 -> 32 on 32^3, 21.3 and
// 23.1.
constexpr size_t kGatherUnits = 4096;

// The convolution: halo planes for cin % 16 == 0, rows put together from a halo
// for two or four input channels, else the gathering implicit GEMM (an even number
// of input channels, x 4-byte aligned).  16-byte copies and stores where a tensor's
// channels and address allow, else narrower ones.
int conv3d(const void* x, int n, int d, int h, int w, int cin, const void* wgt, const float* bias, int cout, int relu,
           int wrap, void* y, float* y32, cudaStream_t s) {
    int vy = 8;
    while (vy > 1 && (cout % vy || (uintptr_t)y % (2 * vy))) vy /= 2;
    const bool vy32 = cout % 4 == 0 && (uintptr_t)y32 % 16 == 0;
    if (cin == 2 && (uintptr_t)x % 4 == 0)
        return conv3d_few<2>(x, n, d, h, w, wgt, bias, cout, relu, wrap, y, y32, vy, vy32, s);
    if (cin == 4 && (uintptr_t)x % 8 == 0)
        return conv3d_few<4>(x, n, d, h, w, wgt, bias, cout, relu, wrap, y, y32, vy, vy32, s);
    if (cin % 16 && (cin % 2 || (uintptr_t)x % 4))
        return fail(LBM_ERR_ARG, "convolution: %d input channels at an odd address on the tcgen05 kernels", cin);
    if (cin % 16) return conv3d_im2col(x, n, d, h, w, cin, wgt, bias, cout, relu, wrap, y, y32, vy, vy32, s);
    int gx = 1;
    const CvShape sh = cv_pick(n, d, h, w, cin, cout, &gx);
    const long long gy = sh.nt ? (cout + sh.nt - 1) / sh.nt : 0;
    if (gy < 1 || gy > 65535) return fail(LBM_ERR_ARG, "convolution: %d output channels exceed the grid", cout);
    // The weights packed as the blocks' slots, except where a block gathers them as fast (or where there is no room).
    const size_t per_tile = (size_t)27 * sh.nt * (cin / 8), units = gy * per_tile;
    const bool gather = sh.chunks == 1 && per_tile <= kGatherUnits;
    const StreamBuffer packed(gather ? 0 : units * 16, s);
    uint4* const wpack = static_cast<uint4*>(packed.get());
    if (wpack) {
        k_pack_weights<<<(unsigned)((units + 127) / 128 < 1216 ? (units + 127) / 128 : 1216), 128, 0, s>>>(
            static_cast<const bf16*>(wgt), cin, cout, sh.nt, (int)gy, wpack);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "k_pack_weights launch");
    }
    auto go = [&](auto kern) -> int {
        int rc = tc_launch_ok((const void*)kern, sh.smem, "cudaFuncSetAttribute(k_conv_halo)");
        if (rc) return rc;
        kern<<<dim3((unsigned)gx, (unsigned)gy), CV_THREADS, sh.smem, s>>>(
            static_cast<const bf16*>(x), n, d, h, w, cin, static_cast<const bf16*>(wgt), wpack, bias, cout, relu, wrap, sh,
            vy, vy32, static_cast<bf16*>(y), y32);
        const cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? LBM_OK : cuda_fail(e, "k_conv_halo launch");
    };
    return (uintptr_t)x % 16 == 0 ? go(k_conv_halo<true>) : go(k_conv_halo<false>);
}
}  // namespace nn
}  // namespace lbm

namespace lbm {
namespace nn {
// Per-chunk partial sums of the weight and bias gradients (k_wgrad_tc,
// k_bias_grad), summed in chunk order by k_sum_chunks: kept for the process
// and grown on demand (calls on one stream reuse it in order).
static float* g_part_buf = nullptr;
static size_t g_part_floats = 0;

float* chunk_scratch(size_t floats) {
    if (floats > g_part_floats) {
        if (g_part_buf) cudaFree(g_part_buf);
        g_part_buf = nullptr;
        g_part_floats = 0;
        if (cudaMalloc(&g_part_buf, floats * sizeof(float)) != cudaSuccess) {
            (void)cudaGetLastError();
            g_part_buf = nullptr;
            return nullptr;
        }
        g_part_floats = floats;
    }
    return g_part_buf;
}

// dst[e] += sum over c = 0 .. chunks-1 of part[c][e], in that order, one thread
// per element.  Bound by the chain of loads where there are few elements: 16 are
// in flight at a time.
__global__ void __launch_bounds__(64) k_sum_chunks(const float* __restrict__ part, long long chunks, long long E,
                                                   float* __restrict__ dst) {
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < E; e += (long long)gridDim.x * blockDim.x) {
        float s = 0.f;
        long long c = 0;
        for (; c + 16 <= chunks; c += 16) {
            float v[16];
#pragma unroll
            for (int k = 0; k < 16; k++) v[k] = __ldg(part + (c + k) * E + e);
#pragma unroll
            for (int k = 0; k < 16; k++) s += v[k];
        }
        for (; c < chunks; c++) s += __ldg(part + c * E + e);
        dst[e] += s;
    }
}

// The same for few elements (bias gradients: 512 chunks of a handful of
// channels), whose chain of loads is what it costs: a block's threads bring 256
// chunks of eight elements to shared memory at once, eight of them add.
__global__ void __launch_bounds__(256) k_sum_few(const float* __restrict__ part, long long chunks, long long E,
                                                 float* __restrict__ dst) {
    __shared__ float sm[256][8];
    const int i = threadIdx.x % 8, j = threadIdx.x / 8;
    for (long long e0 = (long long)blockIdx.x * 8; e0 < E; e0 += (long long)gridDim.x * 8) {
        const long long e = e0 + i;
        float s = 0.f;
        for (long long c0 = 0; c0 < chunks; c0 += 256) {
            const int n = (int)(chunks - c0 < 256 ? chunks - c0 : 256);
#pragma unroll
            for (int c = j; c < 256; c += 32) sm[c][i] = e < E && c < n ? __ldg(part + (c0 + c) * E + e) : 0.f;
            __syncthreads();
            if (j == 0) {
#pragma unroll 16
                for (int c = 0; c < n; c++) s += sm[c][i];
            }
            __syncthreads();
        }
        if (j == 0 && e < E) dst[e] += s;
    }
}

int sum_few(const float* part, long long chunks, long long E, float* dst, cudaStream_t s) {
    const long long blocks = (E + 7) / 8;
    k_sum_few<<<(unsigned)(blocks < 8192 ? blocks : 8192), 256, 0, s>>>(part, chunks, E, dst);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LBM_OK : cuda_fail(e, "k_sum_few launch");
}

int sum_chunks(const float* part, long long chunks, long long E, float* dst, cudaStream_t s) {
    const long long blocks = (E + 63) / 64;
    k_sum_chunks<<<(unsigned)(blocks < 16384 ? blocks : 16384), 64, 0, s>>>(part, chunks, E, dst);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LBM_OK : cuda_fail(e, "k_sum_chunks launch");
}

// dw += the weight gradient: any channel counts and alignment (16-byte copies
// where a tensor's channels and address allow, else value by value).
int wgrad_tc(const void* x, const void* dy, int n, int d, int h, int w, int cin, int cout, int wrap, float* dw,
             cudaStream_t s) {
    const int Wp = (w + 2 + 7) / 8 * 8;
    const WgShape sh = wg_shape(cin, cout, Wp);
    const long long nsteps = ((long long)n * (d + 2) * (h + 2) * Wp + 63) / 64;
    const long long groups = (cin + sh.cc - 1) / sh.cc, mt = (cout + sh.nt - 1) / sh.nt;
    if (!sh.nt || groups > 65535 || mt > 65535)
        return fail(LBM_ERR_ARG, "weight gradient: %d x %d channels exceed the grid", cin, cout);
    // Chunks of positions: the FP32 accumulators in TMEM truncate, about 2e-8 of a sum per K = 16 step, so the
    // chunks, their order and the order within them are part of the result's rounding: a different split moved the
    // gradients of long sums by up to 1e-4, and a network trained on them drifts away from one trained before.  A
    // chunk is one of SMs / q of the positions, q the 448-column accumulators that 27 taps of the input channels
    // would fill (and the 128-channel output tiles), or 8192 voxels outside 8 .. 256 input channels.
    long long chunks = ((long long)n * d * h * w + 8191) / 8192;
    const int cp = (cin + 15) / 16 * 16;
    if (cin >= 8 && cp <= 256) {
        const int per = 448 / cp < 27 ? 448 / cp : 27;
        chunks = sm_count() / ((27 + per - 1) / per * ((cout + TC_M - 1) / TC_M));
    }
    if (chunks < 1) chunks = 1;
    if (chunks > nsteps) chunks = nsteps;
    const long long spc = (nsteps + chunks - 1) / chunks;
    chunks = (nsteps + spc - 1) / spc;
    const long long E = 27LL * cin * cout;
    float* part = chunk_scratch((size_t)(chunks * E));
    if (!part) return fail(LBM_ERR_OOM, "weight-gradient partial sums: %lld floats", chunks * E);
    auto go = [&](auto kern) -> int {
        int rc = tc_launch_ok((const void*)kern, sh.smem, "cudaFuncSetAttribute(k_wgrad_tc)");
        if (rc) return rc;
        kern<<<dim3((unsigned)chunks, (unsigned)groups, (unsigned)mt), WG_THREADS, sh.smem, s>>>(
            static_cast<const bf16*>(x), static_cast<const bf16*>(dy), n, d, h, w, cin, cout, wrap, Wp, nsteps, spc, sh, part);
        const cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? LBM_OK : cuda_fail(e, "k_wgrad_tc launch");
    };
    const bool vx = cin % 8 == 0 && (uintptr_t)x % 16 == 0, vg = cout % 8 == 0 && (uintptr_t)dy % 16 == 0;
    const int rc = vx ? (vg ? go(k_wgrad_tc<true, true>) : go(k_wgrad_tc<true, false>))
                      : (vg ? go(k_wgrad_tc<false, true>) : go(k_wgrad_tc<false, false>));
    return rc ? rc : sum_chunks(part, chunks, E, dw, s);
}
}  // namespace nn
}  // namespace lbm

extern "C" int lbm_nn_conv3d_tc(const void* x, int n, int d, int h, int w, int cin, const void* wgt,
                                const float* bias, int cout, int relu, int wrap, void* y, float* y32, void* stream) {
    if (!x || !wgt || n < 1 || d < 1 || h < 1 || w < 1 || cin < 1 || cout < 1 || (!y && !y32) || (wrap & ~7))
        return fail(LBM_ERR_ARG, "lbm_nn_conv3d_tc: bad arguments");
    if (cin % 8 || cout % 16 || ((uintptr_t)x | (uintptr_t)wgt | (uintptr_t)y | (uintptr_t)y32) & 15)
        return fail(LBM_ERR_ARG, "lbm_nn_conv3d_tc: needs cin %% 8 == 0, cout %% 16 == 0 and 16-byte aligned operands");
    return conv3d(x, n, d, h, w, cin, wgt, bias, cout, relu, wrap, y, y32, static_cast<cudaStream_t>(stream));
}

extern "C" int lbm_nn_conv_tune(int bricks_z, int cout_tile) {
    if (bricks_z < 0 || bricks_z > 4 || cout_tile < 0 || cout_tile > 128 || cout_tile % 16 ||
        (bricks_z && cout_tile && bricks_z * cout_tile > 512))
        return fail(LBM_ERR_ARG, "lbm_nn_conv_tune: bricks_z in 0..4, cout_tile a multiple of 16 in 0..128");
    g_halo_mb = bricks_z;
    g_halo_nt = cout_tile;
    return LBM_OK;
}

extern "C" int lbm_nn_tc_timeouts(unsigned* count) {
    if (!count) return fail(LBM_ERR_ARG, "lbm_nn_tc_timeouts: NULL argument");
    cudaError_t e = cudaMemcpyFromSymbol(count, g_tc_timeouts, sizeof(unsigned));
    if (e == cudaSuccess) {
        const unsigned zero = 0;
        e = cudaMemcpyToSymbol(g_tc_timeouts, &zero, sizeof(unsigned));
    }
    return e == cudaSuccess ? LBM_OK : cuda_fail(e, "lbm_nn_tc_timeouts");
}
