// Pieces shared by the tensor-core training of both networks (train_tc.cu: the regression NeDF;
// train_cls.cu: the paper's classifier network): the tile images that the passes exchange and the
// weight-gradient kernel that reads them.
//
// Tile image: 128 batch rows of a BF16 activation or error signal of C columns as one contiguous
// block of 128 * C * 2 bytes, element (r, c) at (c / 8) * 2048 + r * 16 + (c % 8) * 2.  It is the
// shared-memory operand layout of the MMAs (8 x 16-byte core matrices, no swizzle), so one bulk copy
// moves a whole operand between shared and global memory, and the same bytes serve as
//   K-major operand, rows = M or N, columns = K: LBO (K groups) 2048, SBO (row groups) 128, K step + 4096;
//   MN-major operand, columns = M or N, rows = K: LBO (K groups) 128, SBO (column groups) 2048, K step + 256.
// Weight images ([in / 8][out / 8][8 out][8 in], out = O rows) work the same way with 16 O in the
// place of 2048.
#pragma once

#include <cuda_bf16.h>

#include "pipe_common.cuh"

namespace nedf {
namespace trn {

using namespace tc;

constexpr int kTileB = 128;                        // batch rows per tile image
constexpr uint32_t kMnA = 1u << 15, kMnB = 1u << 16;   // instruction descriptor: MN-major A / B

__host__ __device__ __forceinline__ size_t img_bytes(int cols) { return (size_t)kTileB * cols * 2; }

// shared memory -> global, tracked by the issuing thread's bulk groups
__device__ __forceinline__ void bulk_s2g(void *dst, const void *src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_addr(src)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// the sources of this thread's bulk stores have been read
__device__ __forceinline__ void bulk_s2g_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// ... and their writes are done
__device__ __forceinline__ void bulk_s2g_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// a BF16 of a ReLU output (raw bits in the low or high half of a word) is positive iff its sign bit
// is clear and it is not zero
__device__ __forceinline__ uint32_t pos_lo(uint32_t w) { return (w & 0xFFFFu) - 1u < 0x7FFFu ? 1u : 0u; }
__device__ __forceinline__ uint32_t pos_hi(uint32_t w) { return (w >> 16) - 1u < 0x7FFFu ? 1u : 0u; }
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// ---- epilogue pieces (256 threads, two per row) -----------------------------------------------------
// signs of 16 packed pairs of ReLU outputs, one bit per value
__device__ __forceinline__ uint32_t positive32(const uint32_t (&pk)[16])
{
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) m |= (pos_lo(pk[i]) << (2 * i)) | (pos_hi(pk[i]) << (2 * i + 1));
    return m;
}

// 32 accumulator columns + bias, ReLU, BF16: packed pairs, and the mask of the positive ones
__device__ __forceinline__ uint32_t forward32(const uint32_t (&v)[32], const float *bias, uint32_t (&pk)[16])
{
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const float4 b = *reinterpret_cast<const float4 *>(bias + 4 * q);
        pk[2 * q] = pack_bf16_relu(__uint_as_float(v[4 * q]) + b.x, __uint_as_float(v[4 * q + 1]) + b.y);
        pk[2 * q + 1] = pack_bf16_relu(__uint_as_float(v[4 * q + 2]) + b.z, __uint_as_float(v[4 * q + 3]) + b.w);
    }
    return positive32(pk);
}

// 32 columns of row r, from column c on, into an image
__device__ __forceinline__ void store32(uint8_t *A, int r, int c, const uint32_t (&pk)[16])
{
#pragma unroll
    for (int q = 0; q < 4; ++q)
        *reinterpret_cast<uint4 *>(A + ((c >> 3) + q) * 2048 + r * 16) = make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
}

__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 3, 256;" ::: "memory"); }

// One output tile of a weight gradient, [dW | db] = dZ^T [H | 1]: columns of dZ's image from `a` as
// the 128 rows (output features) of D, N columns of H's image from `b` as its columns (input
// features), the batch as K.  Rows below m_valid are written: row m belongs to segment s = 0 (m <
// seg) or 1 (counted from seg on); column n < n_valid goes to w_off[s] + m' * fi + n, the bias (the
// sum over the batch; `bias` jobs only) to b_off[s] + m'.
struct WgradJob {
    const uint8_t *a, *b;            // first tile's operands
    uint32_t a_stride, b_stride;     // bytes from one tile's operand to the next tile's
    uint32_t a_bytes, b_bytes;       // bytes of one tile's operands
    int N, n_valid, m_valid, seg, fi;
    bool bias;
    long long w_off[2], b_off[2];
};

// Weight gradients of every layer in one launch: blockIdx.x = job * splits + split, a split being a
// contiguous run of tiles whose sum is written as the split's own partial gradient (packed parameter
// layout).  One thread streams both operands of a 128-row tile into a ring of whole-tile stages (two
// bulk copies a stage), one thread issues the tile's eight K steps (plus the bias column's, B = a
// constant block whose first column is one), and the four warps write the accumulator once, at the end.
//
// What bounds it is the operands' way from L2 / HBM (at N = 128 64 KB a tile, about 1,000 cycles at 64
// bytes a cycle and SM, against 576 cycles of MMAs), hence whole tiles as stages (few, large copies)
// and all SMs at work: splits = SMs / jobs.
template <int STAGES, int A_MAX, int B_MAX, int TMEM_COLS, class Jobs>
__global__ void __launch_bounds__(128, 1) k_wgrad(const __grid_constant__ Jobs jobs, int splits, int n_tiles, float *partial,
                                                  long long split_stride, uint32_t *status)
{
    constexpr int STAGE = A_MAX + B_MAX;
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ uint64_t full[STAGES], empty[STAGES], done;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag;
    uint8_t *ones = smem + STAGES * STAGE;             // 16 columns x 128 rows, column 0 = 1
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int job = blockIdx.x / splits, split = blockIdx.x - job * splits;
    const WgradJob J = jobs.get(job);
    const int t0 = (int)((long long)n_tiles * split / splits), t1 = (int)((long long)n_tiles * (split + 1) / splits);
    volatile int *abort = &abort_flag;

    if (warp == 0) tmem_alloc(&tmem_base, TMEM_COLS);
    for (int i = threadIdx.x; i < 256; i += 128)
        reinterpret_cast<uint4 *>(ones)[i] = make_uint4(i < 128 ? 0x3F80u : 0u, 0u, 0u, 0u);
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    if (warp == 0 && lane == 0) {
        RingPos rp;
        int issued = 0;
        for (int t = t0; t < t1 && !*abort; ++t, rp.next(STAGES)) {
            if (!pipe_wait(&empty[rp.st], rp.ph ^ 1u, abort, status)) break;
            uint8_t *st = smem + rp.st * STAGE;
            mbar_arrive_expect_tx(&full[rp.st], J.a_bytes + J.b_bytes);
            bulk_g2s(st, J.a + (size_t)t * J.a_stride, J.a_bytes, &full[rp.st]);
            bulk_g2s(st + A_MAX, J.b + (size_t)t * J.b_stride, J.b_bytes, &full[rp.st]);
            ++issued;
        }
        // the last copies have landed before the block may end (on the normal path they have been used)
        for (int k = issued > STAGES ? issued - STAGES : 0; k < issued; ++k)
            pipe_drain(&full[k % STAGES], (uint32_t)((k / STAGES) & 1), status);
    } else if (warp == 1 && lane == 0) {
        RingPos rp;
        const uint32_t id = idesc_bf16(128, J.N) | kMnA | kMnB, id1 = idesc_bf16(128, 16) | kMnA | kMnB;
        for (int t = t0; t < t1; ++t, rp.next(STAGES)) {
            if (!pipe_wait(&full[rp.st], rp.ph, abort, status)) break;
            tc_fence_after();
            const uint32_t sa = smem_addr(smem + rp.st * STAGE);
            const uint64_t da = smem_desc(sa, 128, 2048), db = smem_desc(sa + A_MAX, 128, 2048);
            const uint64_t d1 = smem_desc(smem_addr(ones), 128, 2048);
            for (int j = 0; j < kTileB / 16; ++j) {
                const uint64_t step = (uint64_t)(j * (256 >> 4));
                const uint32_t acc = (t > t0 || j > 0) ? 1u : 0u;
                mma_bf16(tmem, da + step, db + step, id, acc);
                if (J.bias) mma_bf16(tmem + (uint32_t)J.N, da + step, d1 + step, id1, acc);
            }
            mma_commit(&empty[rp.st]);
        }
        mma_commit(&done);                             // after everything issued so far
    }
    __syncwarp();
    const bool ok = __all_sync(0xffffffffu, pipe_wait(&done, 0u, abort, status));
    if (!ok) {
        *abort = 1;
        pipe_drain(&done, 0u, status);                 // nothing in flight when TMEM goes
    }
    tc_fence_after();
    const int m = warp * 32 + lane;
    if (ok && !*abort) {
        const int s = m < J.seg ? 0 : 1, mo = s ? m - J.seg : m;
        float *w = partial + split * split_stride + J.w_off[s] + (long long)mo * J.fi;
        const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
        const bool vec = ((J.w_off[s] + (long long)mo * J.fi) & 3) == 0 && (split_stride & 3) == 0;
        for (int c = 0; c < J.N; c += 32) {
            uint32_t v[32];
            tmem_ld32(trow + (uint32_t)c, v);
            tmem_wait_ld(v);
            if (m < J.m_valid) {
#pragma unroll
                for (int i = 0; i < 32; i += 4) {
                    const int n = c + i;
                    if (vec && n + 3 < J.n_valid) {
                        *reinterpret_cast<uint4 *>(w + n) = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                    } else {
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (n + e < J.n_valid) w[n + e] = __uint_as_float(v[i + e]);
                    }
                }
            }
            __syncwarp();
        }
        if (J.bias) {
            uint32_t v[32];
            tmem_ld32(trow + (uint32_t)J.N, v);
            tmem_wait_ld(v);
            if (m < J.m_valid) partial[split * split_stride + J.b_off[s] + mo] = __uint_as_float(v[0]);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
}

template <int STAGES, int A_MAX, int B_MAX, int TMEM_COLS, class Jobs>
cudaError_t wgrad(const Jobs &jobs, int n_jobs, int splits, int n_tiles, float *partial, long long split_stride,
                  uint32_t *status, cudaStream_t st)
{
    constexpr int SMEM = STAGES * (A_MAX + B_MAX) + 4096;
    auto k = k_wgrad<STAGES, A_MAX, B_MAX, TMEM_COLS, Jobs>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    if (e != cudaSuccess) return e;
    k<<<n_jobs * splits, 128, SMEM, st>>>(jobs, splits, n_tiles, partial, split_stride, status);
    return cudaGetLastError();
}

// Splits of the batch per job: enough blocks for every SM (one block each), at most one per tile.
inline int wgrad_splits(int n_jobs, int n_tiles, int num_sms)
{
    const int s = num_sms / n_jobs;
    return s < 1 ? 1 : s > n_tiles ? n_tiles : s;
}

}  // namespace trn
}  // namespace nedf
