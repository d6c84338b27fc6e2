// Training of the paper's classifier intersection network (Section "Intersection network",
// Eq. 3-4 and the BCE loss of Eq. 6; "Training details": Adam) on the tensor cores.
//
// A batch of B labelled rays, five kernels:
//   k_cls_prep    the BF16 weight images (forward and transposed) from the packed FP32 master, and the
//                 batch's hit count;
//   k_cls_encode  the 16 encoded chord points of each ray (B x 1008, BF16) as tile images;
//   k_cls_chain   per 128-row tile: the head, 16 residual blocks and the tails, Eq. 6's loss and its
//                 gradient with respect to the logits, and the backward pass by hand (ReLU masks, the
//                 skip connection, d input = delta W), layer after layer on one SM;
//   k_wgrad       dW = delta^T input, db = column sums of delta of every layer, split over the batch
//                 (train_img.cuh);
//   k_cls_finish  the splits' sums in a fixed order and, in a training step, Adam.
// Every dense product is a tcgen05 MMA with BF16 operands and FP32 accumulation: the residual stream
// and the error signals are BF16 between products, as in the BF16 inference engine.
#include <algorithm>
#include <cmath>

#include "mlp_f32.cuh"
#include "render_launch.h"
#include "train_adam.cuh"
#include "train_img.cuh"
#include "train_launch.h"

namespace nedf {

namespace {

using namespace tc;
using trn::bulk_s2g;
using trn::bulk_s2g_wait;
using trn::bulk_s2g_wait_read;
using trn::epilogue_sync;
using trn::kTileB;
using trn::WgradJob;

constexpr int W = 256, NC = 64, NF = 128, NOUT = 1 + NC + NF, NOUT_PAD = 208, NBLK = 16;
constexpr long long kHeadW = (long long)kClsIn * W;
constexpr long long kBlock0 = kHeadW + W;
constexpr long long kLayer = (long long)W * W + W;
constexpr long long kTailA = kBlock0 + 2 * NBLK * kLayer;
constexpr long long kTailB = kTailA + (long long)(1 + NC) * (W + 1);
constexpr long long kPartial = (kClsParams + 3) & ~3ll;    // floats of one split's partial gradient

// Weight images, in the order the chain streams them: K slices of 64 inputs ([k / 8][n][8 k], N rows n):
// head (n = out, k = in, 15 slices of 64 and one of 48), W1 and W2 of each block, the tails (208 rows: tail
// A's 65, tail B's 128, 15 zero); then transposed (n = in, k = out): the tails (K = 208: three slices of
// 64 and one of 16), W2 and W1 of the blocks from the last to the first.
constexpr int kSlice = 64 * W * 2;                         // bytes of a 64-wide slice of 256 rows
constexpr int kTailSlice = 64 * NOUT_PAD * 2;
constexpr long long kImgHead = 0, kImgBody = (long long)kClsIn * W * 2, kImgLayer = (long long)W * W * 2;
constexpr long long kImgTail = kImgBody + 2 * NBLK * kImgLayer;
constexpr long long kImgTailT = kImgTail + (long long)NOUT_PAD * W * 2;
constexpr long long kImgBodyT = kImgTailT + (long long)NOUT_PAD * W * 2;
constexpr long long kImgBytes = kImgBodyT + 2 * NBLK * kImgLayer;

constexpr size_t kImgA = (size_t)kTileB * W * 2;           // tile image of 256 columns
constexpr size_t kImgX = (size_t)kTileB * kClsIn * 2;
constexpr size_t kImgG = (size_t)kTileB * NOUT_PAD * 2;

struct ClsScratch {
    uint8_t *X, *H, *T, *DZ, *DU, *DH0, *G;                // tile images: [block][tile]
    uint8_t *wimg;
    uint4 *mask;                                           // [chain block][32][256] signs of t_k, h_{k+1}
    float *hitp, *lossp, *partial;
    int tiles;
};

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

constexpr int kWgradJobs = 8 + 2 * 2 * NBLK + 2;

// The whole carve in one place: out == nullptr only counts the bytes.
size_t carve(void *base, long long B, int num_sms, ClsScratch *out)
{
    ClsScratch s{};
    const size_t tiles = (size_t)((B + kTileB - 1) / kTileB), chains = std::min<size_t>(tiles, (size_t)num_sms);
    s.tiles = (int)tiles;
    uint8_t *p = reinterpret_cast<uint8_t *>(a256(reinterpret_cast<size_t>(base)));
    uint8_t *const p0 = p;
    auto take = [&](size_t bytes) { uint8_t *q = p; p += a256(bytes); return q; };
    s.X = take(tiles * kImgX);
    s.H = take((NBLK + 1) * tiles * kImgA);
    s.T = take(NBLK * tiles * kImgA);
    s.DZ = take(NBLK * tiles * kImgA);
    s.DU = take(NBLK * tiles * kImgA);
    s.DH0 = take(tiles * kImgA);
    s.G = take(tiles * kImgG);
    s.wimg = take((size_t)kImgBytes);
    s.mask = reinterpret_cast<uint4 *>(take(chains * 2 * NBLK * 256 * sizeof(uint4)));
    s.hitp = reinterpret_cast<float *>(take((size_t)num_sms * 4));
    s.lossp = reinterpret_cast<float *>(take(chains * 4));
    s.partial = reinterpret_cast<float *>(take((size_t)trn::wgrad_splits(kWgradJobs, (int)tiles, num_sms) * kPartial * 4));
    if (out) *out = s;
    return (size_t)(p - p0) + 256;
}

// ---- weight images, hit count ------------------------------------------------------------------------
// One thread per 16-byte vector (8 k of one n), consecutive threads consecutive n: the transposed images
// read whole rows of the master, the others 32 bytes of a row per thread.
__global__ void __launch_bounds__(256) k_cls_prep(const float *w, uint8_t *img, const float *o, const float *d,
                                                  const float *hit_star, long long n_rows, long long start, long long B,
                                                  float rb, float *hitp)
{
    const long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, di = (long long)gridDim.x * blockDim.x;
    for (long long e = i0; e < kImgBytes / 16; e += di) {
        float v[8];
        const long long at = e * 16;
        if (at < kImgBody) {                                       // head
            const int n = (int)(e % W), k = (int)(e / W) * 8;
            for (int j = 0; j < 8; ++j) v[j] = w[(long long)n * kClsIn + k + j];
        } else if (at < kImgTail) {
            const long long q = (at - kImgBody) / 16;
            const int layer = (int)(q / (W * W / 8)), r = (int)(q % (W * W / 8)), n = r % W, k = r / W * 8;
            const float *m = w + kBlock0 + layer * kLayer + (long long)n * W + k;
            for (int j = 0; j < 8; ++j) v[j] = m[j];
        } else if (at < kImgTailT) {
            const int q = (int)((at - kImgTail) / 16), n = q % NOUT_PAD, k = q / NOUT_PAD * 8;
            for (int j = 0; j < 8; ++j)
                v[j] = n < 1 + NC ? w[kTailA + (long long)n * W + k + j]
                     : n < NOUT ? w[kTailB + (long long)(n - 1 - NC) * W + k + j] : 0.0f;
        } else if (at < kImgBodyT) {
            const int q = (int)((at - kImgTailT) / 16), n = q % W, k = q / W * 8;
            for (int j = 0; j < 8; ++j)
                v[j] = k + j < 1 + NC ? w[kTailA + (long long)(k + j) * W + n]
                     : k + j < NOUT ? w[kTailB + (long long)(k + j - 1 - NC) * W + n] : 0.0f;
        } else {
            const long long q = (at - kImgBodyT) / 16;
            const int layer = 2 * NBLK - 1 - (int)(q / (W * W / 8)), r = (int)(q % (W * W / 8)), n = r % W, k = r / W * 8;
            const float *m = w + kBlock0 + layer * kLayer + n;
            for (int j = 0; j < 8; ++j) v[j] = m[(long long)(k + j) * W];
        }
        reinterpret_cast<uint4 *>(img)[e] = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]),
                                                       pack_bf16(v[6], v[7]));
    }
    // hit rows of the batch (the bin terms of Eq. 6 are averaged over them)
    float hits = 0.0f;
    for (long long r = i0; r < B; r += di) {
        const long long q = (start + r) % n_rows;
        const V3 ol = v3(o[3 * q], o[3 * q + 1], o[3 * q + 2]);
        const V3 dl = normalized(v3(d[3 * q], d[3 * q + 1], d[3 * q + 2]));
        Chord ch;
        hits += bound_chord(ol, dl, rb, ch) && hit_star[q] > 0.5f ? 1.0f : 0.0f;
    }
    __shared__ float red[8];
    for (int off = 16; off; off >>= 1) hits += __shfl_xor_sync(0xffffffffu, hits, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = hits;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.0f;
        for (int k = 0; k < 8; ++k) t += red[k];
        hitp[blockIdx.x] = t;
    }
}

// ---- encoding ------------------------------------------------------------------------------------------
// Block = 32 rows x 8 of the 16 chord points (504 columns = 63 groups of 8, staged in shared memory and
// written as 512-byte runs of the tile image); thread = one coordinate of one point of one row at a time:
// [x, sin(2^k x), cos(2^k x)], k = 0..9.  Rows past the batch and rays that miss the bound are zero.
__global__ void __launch_bounds__(256) k_cls_encode(const float *o, const float *d, long long n_rows, long long start,
                                                    long long B, float rb, uint8_t *X)
{
    __shared__ __align__(16) __nv_bfloat16 st[63][32][8];
    const int r0 = blockIdx.x * 32, half = blockIdx.y;
    for (int e = threadIdx.x; e < 32 * 8 * 3; e += 256) {
        const int r = e & 31, c = (e >> 5) % 3, j = (e >> 5) / 3;
        const long long b = r0 + r;
        float x = 0.0f;
        bool kept = false;
        if (b < B) {
            const long long q = (start + b) % n_rows;
            const V3 ol = v3(o[3 * q], o[3 * q + 1], o[3 * q + 2]);
            const V3 dl = normalized(v3(d[3 * q], d[3 * q + 1], d[3 * q + 2]));
            Chord ch;
            kept = bound_chord(ol, dl, rb, ch);
            const V3 p = madd(ol, ch.te + (ch.tx - ch.te) * (float)(8 * half + j) / 15.0f, dl);
            x = c == 0 ? p.x : c == 1 ? p.y : p.z;
        }
        auto put = [&](int f, float v) {
            const int col = 63 * j + f;
            st[col >> 3][r][col & 7] = __float2bfloat16_rn(kept ? v : 0.0f);
        };
        put(c, x);
        for (int k = 0; k < 10; ++k) {
            float sn, cs;
            sincosf(ldexpf(kept ? x : 0.0f, k), &sn, &cs);
            put(3 + 3 * k + c, sn);
            put(33 + 3 * k + c, cs);
        }
    }
    __syncthreads();
    uint8_t *img = X + (size_t)(r0 / kTileB) * kImgX + (size_t)half * 63 * 2048 + (size_t)(r0 % kTileB) * 16;
    for (int v = threadIdx.x; v < 63 * 32; v += 256)
        *reinterpret_cast<uint4 *>(img + (size_t)(v >> 5) * 2048 + (v & 31) * 16) = *reinterpret_cast<const uint4 *>(st[v >> 5][v & 31]);
}

// ---- the chain -------------------------------------------------------------------------------------------
// One 128-row tile at a time per SM.  Roles: warps 0-7 epilogue (two threads a row, 128 columns each; the
// skip connection's operand stays in the thread's registers), warp 8 issues the MMAs (M = 128, N = 256)
// and sends every operand to global memory as a tile image with one bulk copy, warp 9 streams the weight
// slices through a ring of four 32 KB stages (in the head also the tile's 16 KB slices of X, into the
// quarter of the A operand with the stage's number).  A layer is 2,048 cycles of MMAs and as many of
// weights at 64 bytes a cycle from L2, then its epilogue.  As 68 GEMM launches of B / 128 blocks each a
// layer took 22-29 us at 4,096 rows, most of it the launch's own set-up, fill and strided row stores.
constexpr int kStages = 4;
constexpr int kClsChainThreads = 320;
constexpr size_t kClsChainSmem = kImgA + kStages * (size_t)kSlice + 2 * W * 4;

struct ClsChainArgs {
    float rb;
    const float *o, *d, *m_star, *hit_star;
    long long n_rows, start, B;
    const float *w;
    ClsScratch s;
    int n_hitp;
    uint32_t *status;
};

// FP32 bias n of step e: 0 the head, 1 + 2k and 2 + 2k the layers of block k, 33 the tails
__device__ __forceinline__ float cls_bias(const float *w, int e, int n)
{
    if (e == 0) return w[kHeadW + n];
    if (e <= 2 * NBLK) return w[kBlock0 + (e - 1) * kLayer + (long long)W * W + n];
    return n < 1 + NC ? w[kTailA + (long long)(1 + NC) * W + n] : n < NOUT ? w[kTailB + (long long)NF * W + (n - 1 - NC)] : 0.0f;
}

__global__ void __launch_bounds__(kClsChainThreads, 1) k_cls_chain(const __grid_constant__ ClsChainArgs a)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ uint64_t a_ready, acc_full, w_full[kStages], w_empty[kStages], a_free, fin;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag;
    __shared__ float red[8], n_hit_s;
    uint8_t *A = smem, *ring = smem + kImgA;
    float *bsm = reinterpret_cast<float *>(ring + kStages * kSlice);    // [2][256]: this step's and the next one's biases
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tiles = a.s.tiles;
    volatile int *abort = &abort_flag;

    if (warp == 8) tmem_alloc(&tmem_base, W);
    if (threadIdx.x == 0) {
        mbar_init(&a_ready, 256);
        mbar_init(&acc_full, 2);                  // the step's MMAs, and the A image's way out
        mbar_init(&a_free, 1);
        mbar_init(&fin, 1);
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&w_full[s], 1);
            mbar_init(&w_empty[s], 1);
        }
        abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        float h = 0.0f;
        for (int k = lane; k < a.n_hitp; k += 32) h += a.s.hitp[k];
        for (int off = 16; off; off >>= 1) h += __shfl_xor_sync(0xffffffffu, h, off);
        if (lane == 0) n_hit_s = fmaxf(h, 1.0f);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    if (warp == 9) {
        // ------------------------------ weight slices ---------------------------------------------
        if (lane == 0) {
            RingPos rp;
            int issued = 0;
            bool ok = true;
            uint32_t fp = 0;
            for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
                if (tile != (int)blockIdx.x) {    // the previous tile's last operand has left A
                    if (!(ok = pipe_wait(&a_free, fp, abort, a.status))) break;
                    fp ^= 1u;
                }
                const uint8_t *src = a.s.wimg;
                auto slice = [&](uint32_t bytes, const uint8_t *x, uint32_t xbytes) {
                    if (!ok || !(ok = pipe_wait(&w_empty[rp.st], rp.ph ^ 1u, abort, a.status))) return;
                    mbar_arrive_expect_tx(&w_full[rp.st], bytes + xbytes);
                    bulk_g2s(ring + rp.st * kSlice, src, bytes, &w_full[rp.st]);
                    if (xbytes) bulk_g2s(A + rp.st * 16384, x, xbytes, &w_full[rp.st]);
                    src += bytes;
                    ++issued;
                    rp.next(kStages);
                };
                const uint8_t *x = a.s.X + (size_t)tile * kImgX;
                for (int q = 0; q < 16; ++q) {
                    const int k = q < 15 ? 64 : kClsIn - 15 * 64;
                    slice((uint32_t)k * W * 2, x + q * 16384, (uint32_t)k * kTileB * 2);
                }
                for (int q = 0; q < 2 * NBLK * 4; ++q) slice(kSlice, nullptr, 0);
                for (int q = 0; q < 4; ++q) slice(kTailSlice, nullptr, 0);
                for (int q = 0; q < 4; ++q) slice(q < 3 ? kSlice : (NOUT_PAD - 192) * W * 2, nullptr, 0);
                for (int q = 0; q < 2 * NBLK * 4; ++q) slice(kSlice, nullptr, 0);
            }
            for (int k = issued > kStages ? issued - kStages : 0; k < issued; ++k)
                pipe_drain(&w_full[k % kStages], (uint32_t)((k / kStages) & 1), a.status);
        }
    } else if (warp == 8) {
        // ------------------------------ MMA issue, image stores ------------------------------------
        if (lane == 0) {
            RingPos rp;
            uint32_t ap = 0;
            bool ok = true, issued = false;
            const uint32_t sa = smem_addr(A), id = idesc_bf16(128, W), id_tail = idesc_bf16(128, NOUT_PAD);
            // one slice of ksteps K steps against A columns from byte offset aoff
            auto slice = [&](uint32_t aoff, int ksteps, uint32_t n, uint32_t idesc, bool first) {
                if (!ok || !(ok = pipe_wait(&w_full[rp.st], rp.ph, abort, a.status))) return;
                tc_fence_after();
                const uint64_t da = smem_desc(sa + aoff, 2048, 128);
                const uint64_t db = smem_desc(smem_addr(ring + rp.st * kSlice), n * 16, 128);
                for (int k = 0; k < ksteps; ++k)
                    mma_bf16(tmem, da + (uint64_t)(k * (4096 >> 4)), db + (uint64_t)k * (2 * n * 16 >> 4), idesc, !first || k > 0);
                mma_commit(&w_empty[rp.st]);
                issued = true;
                rp.next(kStages);
            };
            // a step: A's image goes out, and the product with the next slices (K columns, N rows)
            auto step = [&](uint8_t *img, uint32_t bytes, int K, uint32_t n, uint32_t idesc) {
                if (!ok || !(ok = pipe_wait(&a_ready, ap, abort, a.status))) return;
                ap ^= 1u;
                tc_fence_after();
                bulk_s2g(img, A, bytes);
                for (int k = 0; k < K; k += 64) slice((uint32_t)k * 256, min(64, K - k) / 16, n, idesc, k == 0);
                if (!ok) return;
                if (K > 0) mma_commit(&acc_full);
                else mbar_arrive(&acc_full);
                bulk_s2g_wait_read();
                mbar_arrive(&acc_full);
            };
            auto at = [&](uint8_t *p, int k, int tile) { return p + ((size_t)k * tiles + tile) * kImgA; };
            for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
                for (int q = 0; q < 16; ++q) slice((uint32_t)rp.st * 16384, q < 15 ? 4 : 3, W, id, q == 0);
                if (!ok) break;
                mma_commit(&acc_full);
                mbar_arrive(&acc_full);
                for (int k = 0; k < NBLK; ++k) {
                    step(at(a.s.H, k, tile), kImgA, W, W, id);
                    step(at(a.s.T, k, tile), kImgA, W, W, id);
                }
                step(at(a.s.H, NBLK, tile), kImgA, W, NOUT_PAD, id_tail);
                step(a.s.G + (size_t)tile * kImgG, kImgG, NOUT_PAD, W, id);
                for (int k = NBLK - 1; k >= 0; --k) {
                    step(at(a.s.DZ, k, tile), kImgA, W, W, id);
                    step(at(a.s.DU, k, tile), kImgA, W, W, id);
                }
                step(at(a.s.DH0, 0, tile), kImgA, 0, W, id);
                if (ok) mbar_arrive(&a_free);
            }
            if (issued) {
                mma_commit(&fin);
                pipe_drain(&fin, 0u, a.status);
            }
            bulk_s2g_wait();
        }
    } else {
        // ------------------------------ epilogue: two threads per row -------------------------------
        const int hf = warp >> 2, r = (warp & 3) * 32 + lane, c0 = hf * 128;
        const uint32_t tacc = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0;
        uint4 *mask = a.s.mask + (size_t)blockIdx.x * 2 * NBLK * 256 + threadIdx.x;
        const float n_hit = n_hit_s;
        uint32_t ep = 0;
        int e = 0;                                // bias row of the coming step
        float part = 0.0f, nb = 0.0f;
        auto acc_wait = [&]() {                   // accumulator complete, A free; one outcome for the 256 threads
            const bool ok = pipe_wait(&acc_full, ep, abort, a.status);
            ep ^= 1u;
            const bool dead = epilogue_any(!ok);
            if (dead) *abort = 1;
            tc_fence_after();
            return !dead;
        };
        auto a_done = [&]() {
            fence_proxy_async_smem();
            tc_fence_before();
            mbar_arrive(&a_ready);
        };
        // the bias rows are double-buffered: row e + 1 is fetched while step e runs and stored after its
        // wait (every thread is then past its reads of row e - 1, in the same buffer)
        auto bias_next = [&](int row) { bsm[(row & 1) * W + threadIdx.x] = nb; };
        uint32_t hk[4][16];                       // this thread's half row of h_k, then of dz_k
        bool alive = true;
        for (int tile = blockIdx.x; tile < tiles && alive; tile += gridDim.x) {
            nb = cls_bias(a.w, 0, threadIdx.x);
            epilogue_sync();
            bias_next(0);
            // ---- head, then two layers per block
            for (e = 0; e <= 2 * NBLK && alive; ++e) {
                nb = cls_bias(a.w, e + 1, threadIdx.x);
                if (!(alive = acc_wait())) break;
                bias_next(e + 1);
                const float *bias = bsm + (e & 1) * W + c0;
                uint4 mk;
                uint32_t *m = &mk.x;
                uint32_t v[2][32];
                tmem_ld32(tacc, v[0]);
                tmem_wait_ld(v[0]);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (q < 3) tmem_ld32(tacc + 32 * (q + 1), v[(q + 1) & 1]);
                    const uint32_t(&u)[32] = v[q & 1];
                    uint32_t pk[16];
                    if (e == 0) {                 // the head is linear
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const float2 b = *reinterpret_cast<const float2 *>(bias + 32 * q + 2 * i);
                            hk[q][i] = pk[i] = pack_bf16(__uint_as_float(u[2 * i]) + b.x, __uint_as_float(u[2 * i + 1]) + b.y);
                        }
                    } else if (e & 1) {           // t_k = ReLU(W1 h_k + b1)
                        m[q] = trn::forward32(u, bias + 32 * q, pk);
                    } else {                      // h_{k+1} = ReLU(W2 t_k + b2 + h_k)
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const float2 b = *reinterpret_cast<const float2 *>(bias + 32 * q + 2 * i);
                            float x0 = __uint_as_float(u[2 * i]) + b.x, x1 = __uint_as_float(u[2 * i + 1]) + b.y;
                            x0 += trn::bf_lo(hk[q][i]);
                            x1 += trn::bf_hi(hk[q][i]);
                            hk[q][i] = pk[i] = pack_bf16_relu(x0, x1);
                        }
                        m[q] = trn::positive32(pk);
                    }
                    trn::store32(A, r, c0 + 32 * q, pk);
                    if (q < 3) tmem_wait_ld(v[(q + 1) & 1]);
                }
                if (e > 0) mask[(size_t)(e - 1) * 256] = mk;
                a_done();
            }
            if (!alive || !(alive = acc_wait())) break;
            // ---- tails and Eq. 6: the loss and its gradient with respect to the logits (BF16: it enters the
            // products), zero beyond the 193 logits.  Segment operator S: u = (m* + 1) N_c / 2, c = floor(u),
            // f = floor((u - c) N_f), clamped.
            {
                const long long b = (long long)tile * kTileB + r;
                bool ok = false, hit = false;
                int cs = 0, fs = 0;
                if (b < a.B) {
                    const long long i = (a.start + b) % a.n_rows;
                    const V3 ol = v3(a.o[3 * i], a.o[3 * i + 1], a.o[3 * i + 2]);
                    const V3 dl = normalized(v3(a.d[3 * i], a.d[3 * i + 1], a.d[3 * i + 2]));
                    Chord ch;
                    ok = bound_chord(ol, dl, a.rb, ch);
                    hit = ok && a.hit_star[i] > 0.5f;
                    if (hit) {
                        const float u = (a.m_star[i] + 1.0f) * 0.5f * NC;
                        cs = min(max((int)floorf(u), 0), NC - 1);
                        fs = min(max((int)floorf((u - cs) * NF), 0), NF - 1);
                    }
                }
                const float *bias = bsm + ((2 * NBLK + 1) & 1) * W + c0;
                const float Bf = (float)a.B;
                for (int q = 0; q < (hf ? 3 : 4); ++q) {
                    uint32_t v[32], pk[16];
                    __syncwarp();                 // the rows' losses above diverge
                    tmem_ld32(tacc + 32 * q, v);
                    tmem_wait_ld(v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        float g2[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int col = c0 + 32 * q + 2 * i + h;
                            const float x = __uint_as_float(v[2 * i + h]) + bias[32 * q + 2 * i + h];
                            float gi = 0.0f;
                            if (ok && col < NOUT && (hit || col == 0)) {
                                const float sg = 1.0f / (1.0f + expf(-x));
                                const int one = col == 0 ? 0 : col <= NC ? 1 + cs : 1 + NC + fs;
                                const float y = col == 0 ? (hit ? 1.0f : 0.0f) : col == one ? 1.0f : 0.0f;
                                const float l = fmaxf(x, 0.0f) - x * y + log1pf(expf(-fabsf(x)));   // BCE(x, y)
                                if (col == 0) {
                                    part += 0.1f * l / Bf;
                                    gi = 0.1f * (sg - y) / Bf;
                                } else {
                                    const float bins = col <= NC ? 1.0f / NC : 1.0f / NF;      // powers of two
                                    part += l * bins / n_hit;
                                    gi = (sg - y) * bins / n_hit;
                                }
                            }
                            g2[h] = gi;
                        }
                        pk[i] = pack_bf16(g2[0], g2[1]);
                    }
                    if (hf == 0 || q < 2) {
                        trn::store32(A, r, c0 + 32 * q, pk);
                    } else {                      // columns 192 .. 207, the last of G
#pragma unroll
                        for (int g = 0; g < 2; ++g)
                            *reinterpret_cast<uint4 *>(A + (24 + g) * 2048 + r * 16) = make_uint4(pk[4 * g], pk[4 * g + 1], pk[4 * g + 2], pk[4 * g + 3]);
                    }
                }
                __syncwarp();
                a_done();
            }
            // ---- backward: dz = dh [z > 0]; du = (dz W2) [u > 0]; dh = dz + du W1 (masked by the block input
            // for the next dz; unmasked at the linear head).  Step j: 0 the tails, 1 + 2 i and 2 + 2 i the
            // layers of block 15 - i.
            for (int j = 0; j <= 2 * NBLK && alive; ++j) {
                // sign masks: dz_15 h_16 (31), du_k t_k (2 k), dz_{k-1} h_k (2 k - 1): 31 - j; the last has none
                uint4 mk = make_uint4(~0u, ~0u, ~0u, ~0u);
                if (j < 2 * NBLK) mk = mask[(size_t)(2 * NBLK - 1 - j) * 256];
                const uint32_t *m = &mk.x;
                if (!(alive = acc_wait())) break;
                uint32_t v[2][32];
                tmem_ld32(tacc, v[0]);
                tmem_wait_ld(v[0]);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (q < 3) tmem_ld32(tacc + 32 * (q + 1), v[(q + 1) & 1]);
                    const uint32_t(&u)[32] = v[q & 1];
                    uint32_t pk[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        float x0 = __uint_as_float(u[2 * i]), x1 = __uint_as_float(u[2 * i + 1]);
                        if (j > 0 && !(j & 1)) {  // dh = du W1 + dz
                            x0 += trn::bf_lo(hk[q][i]);
                            x1 += trn::bf_hi(hk[q][i]);
                        }
                        x0 = (m[q] >> (2 * i)) & 1u ? x0 : 0.0f;
                        x1 = (m[q] >> (2 * i + 1)) & 1u ? x1 : 0.0f;
                        pk[i] = pack_bf16(x0, x1);
                        if (!(j & 1)) hk[q][i] = pk[i];          // dz_k
                    }
                    trn::store32(A, r, c0 + 32 * q, pk);
                    if (q < 3) tmem_wait_ld(v[(q + 1) & 1]);
                }
                a_done();
            }
            if (alive) alive = acc_wait();        // dh_0 has left A
        }
        for (int off = 16; off; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
        if (lane == 0) red[warp] = part;
        epilogue_sync();
        if (threadIdx.x == 0) {
            float t = 0.0f;
            for (int k = 0; k < 8; ++k) t += red[k];
            a.s.lossp[blockIdx.x] = t;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 8) tmem_dealloc(tmem, W);
}

// ---- weight-gradient jobs -------------------------------------------------------------------------------
// 8 of the head (two halves of the 256 outputs x four 256-column blocks of the 1008 inputs), two of every
// body layer (halves of its outputs), two of the tails (rows 0 .. 127 and 128 .. 192 of the 193 logits).
struct ClsJobs {
    ClsScratch s;
    __device__ __forceinline__ WgradJob get(int job) const
    {
        WgradJob j;
        const size_t run = (size_t)s.tiles * kImgA;
        const int mb = job & 1;
        j.m_valid = j.seg = 128;
        j.a_stride = j.b_stride = (uint32_t)kImgA;
        j.a_bytes = 32768;
        j.b_bytes = 65536;
        j.N = j.n_valid = j.fi = W;
        j.bias = true;
        if (job < 8) {
            const int nb = job >> 1;
            j.a = s.DH0 + mb * 32768;
            j.b = s.X + nb * 65536;
            j.b_stride = (uint32_t)kImgX;
            j.N = j.n_valid = nb < 3 ? 256 : kClsIn - 768;
            j.b_bytes = (uint32_t)j.N * 256;
            j.fi = kClsIn;
            j.bias = nb == 0;
            j.w_off[0] = j.w_off[1] = (long long)mb * 128 * kClsIn + nb * 256;
            j.b_off[0] = j.b_off[1] = kHeadW + mb * 128;
        } else if (job < 8 + 4 * NBLK) {
            const int q = (job - 8) >> 1, k = q >> 1;              // body layer q: dW1 = dU^T h, dW2 = dZ^T t
            j.a = ((q & 1) ? s.DZ : s.DU) + k * run + mb * 32768;
            j.b = ((q & 1) ? s.T : s.H) + k * run;
            const long long off = kBlock0 + q * kLayer;
            j.w_off[0] = j.w_off[1] = off + (long long)mb * 128 * W;
            j.b_off[0] = j.b_off[1] = off + (long long)W * W + mb * 128;
        } else {                                                   // tails: dW = G^T h_16
            j.a = s.G + mb * 32768;
            j.a_stride = (uint32_t)kImgG;
            j.a_bytes = mb ? (uint32_t)kImgG - 32768 : 32768;
            j.b = s.H + NBLK * run;
            j.m_valid = mb ? NOUT - 128 : 128;
            j.seg = mb ? 0 : 1 + NC;
            const int skip = mb ? 128 - 1 - NC : 0;                // tail B rows before this job's first
            j.w_off[0] = kTailA;
            j.b_off[0] = kTailA + (long long)(1 + NC) * W;
            j.w_off[1] = kTailB + (long long)skip * W;
            j.b_off[1] = kTailB + (long long)NF * W + skip;
        }
        return j;
    }
};

// ---- the fixed-order sums, and Adam ----------------------------------------------------------------------
struct ClsFinishArgs {
    const float *partial, *lossp, *hitp;
    int splits, chains, n_hitp;
    float *grad, *loss;                            // grad may be null
    float *theta, *m, *v;                          // theta null: no Adam step
    float lr, c1, c2;
};

__global__ void __launch_bounds__(256) k_cls_finish(const __grid_constant__ ClsFinishArgs a)
{
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        float l = 0.0f, h = 0.0f;
        for (int c = threadIdx.x; c < a.chains; c += 32) l += a.lossp[c];
        for (int c = threadIdx.x; c < a.n_hitp; c += 32) h += a.hitp[c];
        for (int off = 16; off; off >>= 1) {
            l += __shfl_xor_sync(0xffffffffu, l, off);
            h += __shfl_xor_sync(0xffffffffu, h, off);
        }
        if (threadIdx.x == 0) {
            a.loss[0] = l;
            a.loss[1] = h;
        }
    }
    for (long long e = blockIdx.x * 256ll + threadIdx.x; e < kClsParams; e += (long long)gridDim.x * 256) {
        float g = 0.0f;
        for (int z = 0; z < a.splits; ++z) g += a.partial[(size_t)z * kPartial + e];
        if (a.grad) a.grad[e] = g;
        if (a.theta) a.theta[e] = adam_step(a.theta[e], g, a.m[e], a.v[e], a.lr, a.c1, a.c2);
    }
}

// Forward, loss, gradient and (f.theta) the Adam step of one batch.
cudaError_t run(const ClsTrainLaunch &L, const float *o, const float *d, const float *m_star, const float *hit_star,
                long long n_rows, long long start, long long B, ClsFinishArgs f)
{
    cudaStream_t st = L.stream;
    ClsScratch s;
    carve(L.scratch, B, L.num_sms, &s);
    k_cls_prep<<<L.num_sms, 256, 0, st>>>(L.master, s.wimg, o, d, hit_star, n_rows, start, B, L.rb, s.hitp);
    k_cls_encode<<<dim3(s.tiles * (kTileB / 32), 2), 256, 0, st>>>(o, d, n_rows, start, B, L.rb, s.X);
    ClsChainArgs c{};
    c.rb = L.rb;
    c.o = o; c.d = d; c.m_star = m_star; c.hit_star = hit_star;
    c.n_rows = n_rows; c.start = start; c.B = B;
    c.w = L.master; c.s = s; c.n_hitp = L.num_sms; c.status = L.status;
    cudaError_t e = cudaFuncSetAttribute(k_cls_chain, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClsChainSmem);
    if (e != cudaSuccess) return e;
    const int chains = std::min(s.tiles, L.num_sms);
    k_cls_chain<<<chains, kClsChainThreads, kClsChainSmem, st>>>(c);
    const int splits = trn::wgrad_splits(kWgradJobs, s.tiles, L.num_sms);
    e = trn::wgrad<2, 32768, 65536, 512>(ClsJobs{s}, kWgradJobs, splits, s.tiles, s.partial, kPartial, L.status, st);
    if (e != cudaSuccess) return e;
    f.partial = s.partial; f.lossp = s.lossp; f.hitp = s.hitp;
    f.splits = splits; f.chains = chains; f.n_hitp = L.num_sms;
    f.loss = L.loss;
    k_cls_finish<<<L.num_sms * 8, 256, 0, st>>>(f);
    return cudaGetLastError();
}

}  // namespace

size_t cls_train_scratch_bytes(long long batch, int num_sms) { return carve(nullptr, batch, num_sms, nullptr); }

cudaError_t launch_cls_loss_grad(const ClsTrainLaunch &L, const float *o, const float *d, const float *m_star,
                                 const float *hit_star, int n, float *grad)
{
    ClsFinishArgs f{};
    f.grad = grad;
    return run(L, o, d, m_star, hit_star, n, 0, n, f);
}

cudaError_t launch_cls_train_step(const ClsTrainLaunch &L, const float *o, const float *d, const float *m_star,
                                  const float *hit_star, long long n_rays, long long start, int batch, float *adam_m,
                                  float *adam_v, int step, float lr)
{
    ClsFinishArgs f{};
    f.theta = L.master; f.m = adam_m; f.v = adam_v;
    f.lr = lr;
    f.c1 = 1.0f - powf(0.9f, (float)step);
    f.c2 = 1.0f - powf(0.999f, (float)step);
    return run(L, o, d, m_star, hit_star, n_rays, start, batch, f);
}

}  // namespace nedf
