// Learned part on the tensor cores: BF16 NeDF training with FP32 accumulation, FP32 master weights
// and Adam (Section "Intersection network": supervision of F_Phi through Eq. 2 and Eq. 5; the
// regression form of Eq. 6; "Training details": Adam).
//
// A step on a batch of B rows, width W, L hidden layers, four kernels:
//   k_tc_prep   the BF16 weight images from the FP32 master, and the batch's hit count;
//   k_tc_chain  per 128-row tile: X0 = BF16(gamma([p_e, d])) (78 features, 2 zero pads),
//                 forward   H_{l+1} = BF16(ReLU(H_l Wb_l^T + b_l)),  l = 0 .. L-1
//                 loss      y = W_out H_L + b_out (FP32), Eq. 6 (regression form), dy,
//                           dZ_{L-1} = BF16((W_out^T dy) * [H_L > 0]), dW_out and db_out
//                 backward  dZ_{l-1} = BF16((dZ_l Wb_l) * [H_l > 0]),  l = L-1 .. 1
//               with the tile's activations in shared memory from the first layer to the last;
//   k_wgrad     [dW_l | db_l] = dZ_l^T [H_l | 1] of every layer, split over the batch (train_img.cuh);
//   k_tc_finish the splits' sums in a fixed order and, in a training step, Adam.
// Activations and error signals are BF16 operands (the error signal of a hidden layer is rounded to
// BF16 where it enters a product); every sum is FP32.  The fixed order of every sum keeps a step
// deterministic, so a resumed run repeats an uninterrupted one bit for bit.
#include <algorithm>
#include <cmath>

#include "mlp_f32.cuh"
#include "train_adam.cuh"
#include "train_img.cuh"
#include "train_launch.h"

namespace nedf {

using namespace tc;
using trn::kTileB;
using trn::bulk_s2g;
using trn::bulk_s2g_wait;
using trn::bulk_s2g_wait_read;
using trn::epilogue_sync;

constexpr int kChainThreads = 288;       // 8 epilogue warps (two threads a row), 1 issuing warp

template <int W>
struct ChainShape {
    static constexpr int WIDE = W > kNedfInPad ? W : kNedfInPad;
    static constexpr int X0 = kTileB * kNedfInPad * 2;             // image of the encoded input
    static constexpr int IMG = kTileB * W * 2;                     // image of an activation
    static constexpr int A_BYTES = kTileB * WIDE * 2;
    static constexpr int WST = W * WIDE * 2;                       // one layer's weight image
    // A operand, two weight stages, output weights [2][W] and biases, dy, the row sums' first halves
    static constexpr int FIXED = A_BYTES + 2 * WST + (2 * W + 4) * 4 + 2 * kTileB * 8;   // + biases, L x W floats
};

// offset of layer l's weights in the packed layout (W[out][in] then b[out] per layer)
__host__ __device__ __forceinline__ long long packed_off(int l, int W)
{
    return l == 0 ? 0 : (long long)kNedfIn * W + W + (long long)(l - 1) * (W * W + W);
}
// byte offset of layer l's weight image
__host__ __device__ __forceinline__ long long wimg_off(int l, int W)
{
    return l == 0 ? 0 : 2 * ((long long)W * kNedfInPad + (long long)(l - 1) * W * W);
}

// ---- scratch ----------------------------------------------------------------------------------
struct TcTrainScratch {
    uint8_t *ximg, *himg, *zimg; // images of X0, of H_1 .. H_{L-1} and of dZ_0 .. dZ_{L-1}, tile after tile
    uint8_t *wimg;               // BF16 weight images of the hidden layers
    uint2 *mask;                 // [chain block][layer][256]: the signs of each thread's columns of H_l
    float *hitp;                 // hit counts per prep block
    float *outp;                 // [chain block][2 W + 2]: dW_out, db_out
    float *lossp;                // [chain block]
    float *partial;              // [splits][partial_stride], hidden layers
};

// one split's partial gradient, in floats (rows of it keep their 16-byte alignment)
static long long partial_stride(long long n_params) { return (n_params + 3) & ~3ll; }

static size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// The whole carve in one place: base == nullptr only counts the bytes.
static size_t carve_tc(void *base, int B, int L, int W, long long n_params, int num_sms, TcTrainScratch *out)
{
    const size_t tiles = ((size_t)B + kTileB - 1) / kTileB, chains = std::min<size_t>(tiles, 2 * (size_t)num_sms);
    const size_t img = trn::img_bytes(W);
    uint8_t *p = reinterpret_cast<uint8_t *>(align256(reinterpret_cast<size_t>(base)));
    uint8_t *const p0 = p;
    auto take = [&](size_t bytes) { uint8_t *q = p; p += align256(bytes); return q; };
    TcTrainScratch s{};
    s.ximg = take(tiles * trn::img_bytes(kNedfInPad));
    s.himg = take(tiles * img * (L - 1));
    s.zimg = take(tiles * img * L);
    s.wimg = take((size_t)wimg_off(L, W));
    s.mask = reinterpret_cast<uint2 *>(take(chains * L * 256 * sizeof(uint2)));
    s.hitp = reinterpret_cast<float *>(take(4 * (size_t)num_sms));
    s.outp = reinterpret_cast<float *>(take(4 * chains * (2 * W + 2)));
    s.lossp = reinterpret_cast<float *>(take(4 * chains));
    s.partial = reinterpret_cast<float *>(take(4 * (size_t)trn::wgrad_splits(L, (int)tiles, num_sms) * partial_stride(n_params)));
    if (out) *out = s;
    return (size_t)(p - p0) + 256;
}

size_t train_tc_scratch_bytes(int batch, int hidden, int width, long long n_params, int num_sms)
{
    return carve_tc(nullptr, batch, hidden, width, n_params, num_sms, nullptr);
}

// ---- BF16 weight images from the FP32 master, and the batch's hit count ----------------------------
__global__ void __launch_bounds__(256) k_tc_prep(const float *master, uint8_t *wimg, int L, int W, const float *hit_star,
                                                 long long start, long long n, int B, float *hitp)
{
    const long long total = wimg_off(L, W) / 2;
    const long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, di = (long long)gridDim.x * blockDim.x;
    for (long long e = i0; e < total; e += di) {
        const long long n0 = (long long)W * kNedfInPad;
        const int l = e < n0 ? 0 : 1 + (int)((e - n0) / ((long long)W * W));
        const int fi = l == 0 ? kNedfIn : W;
        const long long q = e - wimg_off(l, W) / 2;      // image order: [in / 8][out][8 in]
        const int i = (int)(q / (8 * W)) * 8 + (int)(q & 7), o = (int)((q >> 3) % W);
        const float v = i < fi ? master[packed_off(l, W) + (long long)o * fi + i] : 0.0f;
        reinterpret_cast<__nv_bfloat16 *>(wimg)[e] = __float2bfloat16_rn(v);
    }
    float hits = 0.0f;
    for (long long b = i0; b < B; b += di) hits += hit_star[(start + b) % n];
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

// ---- the chain: encoding, forward, loss, backward ---------------------------------------------------
// The layers of a 128-row tile one after another on one SM, two blocks per SM taking turns on its
// tensor pipe.  Per layer the issuing thread sends the A operand to global memory as a tile image (the
// weight gradients read it), issues the layer's MMAs (M = 128 rows, N = W) and refills the weight stage
// the previous layer left; the 8 epilogue warps (thread = half a row) turn the accumulator into the next
// layer's operand.  As separate GEMM launches each layer paid its own TMEM allocation, barrier set-up,
// pipeline fill and store of 128-byte row pieces, 31 us forward and 41 us backward per layer for 5 us of
// memory traffic at 65,536 rows.  The two blocks per SM have 96 registers a thread (76 bytes spilled at W = 128).
struct ChainArgs {
    float rb;
    const float *o, *d, *m_star, *hit_star;
    long long start, n;
    int B, tiles, L, n_hitp;
    const float *master;
    TcTrainScratch s;
    uint32_t *status;
};

template <int W>
__global__ void __launch_bounds__(kChainThreads, 2) k_tc_chain(const __grid_constant__ ChainArgs a)
{
    using SH = ChainShape<W>;
    constexpr int NB = W / 64;                    // blocks of 32 columns per thread
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ uint64_t a_ready, acc_full, w_full[2], fin;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag;
    __shared__ float red[8], n_hit_s;
    uint8_t *A = smem, *ring = smem + SH::A_BYTES;
    float *wout = reinterpret_cast<float *>(ring + 2 * SH::WST);   // [2][W], b[2]
    float2 *dy = reinterpret_cast<float2 *>(wout + 2 * W + 4), *yp = dy + kTileB;
    float *bias = reinterpret_cast<float *>(yp + kTileB);          // [L][W]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, L = a.L;
    volatile int *abort = &abort_flag;

    if (warp == 8) tmem_alloc(&tmem_base, W < 128 ? 64 : 128);
    if (threadIdx.x == 0) {
        mbar_init(&a_ready, 256);
        mbar_init(&acc_full, 2);                  // the layer's MMAs, and the A image's way out
        mbar_init(&w_full[0], 1);
        mbar_init(&w_full[1], 1);
        mbar_init(&fin, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    for (int k = threadIdx.x; k < 2 * W + 2; k += kChainThreads) {
        const float v = a.master[packed_off(L, W) + k];
        wout[k] = k < 2 * W ? round_bf16(v) : v;
    }
    for (int k = threadIdx.x; k < L * W; k += kChainThreads) {
        const int l = k / W;
        bias[k] = a.master[packed_off(l, W) + (long long)(l == 0 ? kNedfIn : W) * W + (k - l * W)];
    }
    if (warp == 0) {
        float h = 0.0f;
        for (int k = lane; k < a.n_hitp; k += 32) h += a.s.hitp[k];
        for (int off = 16; off; off >>= 1) h += __shfl_xor_sync(0xffffffffu, h, off);
        if (lane == 0) n_hit_s = h;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    const int grid = gridDim.x;

    if (warp == 8) {
        // ------------------------------ MMA issue, weight loads, image stores ---------------------
        if (lane == 0) {
            const int per = 2 * L - 1;            // MMA steps per tile: L forward, L - 1 backward
            const long long total = (long long)((a.tiles - 1 - (int)blockIdx.x) / grid + 1) * per;
            const uint32_t idf = idesc_bf16(128, W), idb = idf | trn::kMnB;
            const uint32_t sa = smem_addr(A);
            long long q = 0, loaded = 0;          // MMA steps issued, weight images asked for
            int jl = 0;                           // the next load's step within its tile
            uint32_t ap = 0;
            auto load = [&]() {                   // the next step's weights into the stage of its parity
                const int l = jl < L ? jl : 2 * L - 1 - jl;
                const uint32_t bytes = (uint32_t)(wimg_off(l + 1, W) - wimg_off(l, W));
                uint64_t *bar = &w_full[loaded & 1];
                mbar_arrive_expect_tx(bar, bytes);
                bulk_g2s(ring + (loaded & 1) * SH::WST, a.s.wimg + wimg_off(l, W), bytes, bar);
                ++loaded;
                if (++jl == per) jl = 0;
            };
            load();
            if (total > 1) load();
            bool ok = true;
            for (int tile = blockIdx.x; tile < a.tiles && ok; tile += grid)
                for (int s = 0; s < 2 * L && ok; ++s, ap ^= 1u) {
                    if (!(ok = pipe_wait(&a_ready, ap, abort, a.status))) break;
                    tc_fence_after();
                    if (s == 0) bulk_s2g(a.s.ximg + (size_t)tile * SH::X0, A, SH::X0);
                    else if (s < L) bulk_s2g(a.s.himg + ((size_t)(s - 1) * a.tiles + tile) * SH::IMG, A, SH::IMG);
                    else bulk_s2g(a.s.zimg + ((size_t)(2 * L - 1 - s) * a.tiles + tile) * SH::IMG, A, SH::IMG);
                    if (s < per) {
                        // every thread's a_ready followed its wait for the previous step's MMAs, so
                        // that step's stage is free
                        if (q >= 1 && loaded < total) load();
                        if (!(ok = pipe_wait(&w_full[q & 1], (uint32_t)((q >> 1) & 1), abort, a.status))) break;
                        tc_fence_after();
                        const uint32_t sw = smem_addr(ring + (q & 1) * SH::WST);
                        const uint64_t da = smem_desc(sa, 2048, 128);
                        if (s < L) {              // B = W_l: rows out (N), K = in
                            const uint64_t db = smem_desc(sw, W * 16, 128);
                            const int nk = s == 0 ? kNedfInPad / 16 : W / 16;
                            for (int k = 0; k < nk; ++k)
                                mma_bf16(tmem, da + (uint64_t)(k * (4096 >> 4)), db + (uint64_t)(k * (2 * W * 16 >> 4)), idf, k > 0);
                        } else {                  // B = W_l^T: N = in, K = out
                            const uint64_t db = smem_desc(sw, 128, W * 16);
                            for (int k = 0; k < W / 16; ++k)
                                mma_bf16(tmem, da + (uint64_t)(k * (4096 >> 4)), db + (uint64_t)(k * (256 >> 4)), idb, k > 0);
                        }
                        mma_commit(&acc_full);
                        ++q;
                    } else {
                        mbar_arrive(&acc_full);   // dZ_0 feeds no further product
                    }
                    bulk_s2g_wait_read();
                    mbar_arrive(&acc_full);
                }
            // nothing of this block may be in flight when it ends
            for (long long k = q; k < loaded; ++k) pipe_drain(&w_full[k & 1], (uint32_t)((k >> 1) & 1), a.status);
            if (q > 0) {
                mma_commit(&fin);
                pipe_drain(&fin, 0u, a.status);
            }
            bulk_s2g_wait();
        }
    } else {
        // ------------------------------ epilogue: two threads per row ------------------------------
        const int hf = warp >> 2, r = (warp & 3) * 32 + lane, c0 = hf * (W / 2);
        const uint32_t tacc = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0;
        uint2 *mask = a.s.mask + (size_t)blockIdx.x * L * 256 + threadIdx.x;
        const float n_hit = n_hit_s;
        uint32_t ep = 0;
        // the step's accumulator is complete and A may be overwritten; one outcome for all 256 threads
        auto acc_wait = [&]() {
            const bool ok = pipe_wait(&acc_full, ep, abort, a.status);
            ep ^= 1u;
            const bool dead = epilogue_any(!ok);
            if (dead) *abort = 1;
            tc_fence_after();
            return !dead;
        };
        auto a_done = [&]() {                     // this thread's part of the next operand is written
            fence_proxy_async_smem();
            tc_fence_before();
            mbar_arrive(&a_ready);
        };
        // dW_out / db_out: thread = 8 columns (cg) and every RS-th row
        constexpr int RS = 256 / (W / 8);
        const int cg = threadIdx.x / RS, rs = threadIdx.x % RS;
        float ow[2][8] = {}, ob[2] = {0.0f, 0.0f}, part = 0.0f;
        bool alive = true;
        for (int tile = blockIdx.x; tile < a.tiles && alive; tile += grid) {
            // ---- encode: this thread's three of the row's six inputs
            const long long b = (long long)tile * kTileB + r;
            const long long i = b < a.B ? (a.start + b) % a.n : 0;
            bool kept = false;
            {
                float x[3] = {0.f, 0.f, 0.f};
                if (b < a.B) {
                    const V3 ol = v3(a.o[3 * i], a.o[3 * i + 1], a.o[3 * i + 2]);
                    const V3 dl = normalized(v3(a.d[3 * i], a.d[3 * i + 1], a.d[3 * i + 2]));
                    Chord ch;
                    kept = bound_chord(ol, dl, a.rb, ch);
                    if (kept) {
                        const V3 pe = madd(ol, ch.te, dl);
                        x[0] = hf ? dl.x : pe.x; x[1] = hf ? dl.y : pe.y; x[2] = hf ? dl.z : pe.z;
                    }
                }
                auto put = [&](int f, float v) {
                    *reinterpret_cast<__nv_bfloat16 *>(A + (f >> 3) * 2048 + r * 16 + (f & 7) * 2) = __float2bfloat16_rn(v);
                };
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    put(3 * hf + c, x[c]);
#pragma unroll 1
                    for (int k = 0; k < 6; ++k) {
                        float sn, cs;
                        sincosf(ldexpf(x[c], k), &sn, &cs);
                        put(6 + 6 * k + 3 * hf + c, sn);
                        put(42 + 6 * k + 3 * hf + c, cs);
                    }
                }
                if (hf == 0) *reinterpret_cast<uint32_t *>(A + (kNedfIn >> 3) * 2048 + r * 16 + (kNedfIn & 7) * 2) = 0u;
            }
            a_done();
            // ---- forward
            uint32_t pk[NB][16];
            uint2 mk = make_uint2(0u, 0u);
            for (int l = 0; l < L && alive; ++l) {
                if (!(alive = acc_wait())) break;
                uint32_t v[NB][32];
#pragma unroll
                for (int q = 0; q < NB; ++q) tmem_ld32(tacc + 32 * q, v[q]);
#pragma unroll
                for (int q = 0; q < NB; ++q) tmem_wait_ld(v[q]);
                mk.x = trn::forward32(v[0], bias + l * W + c0, pk[0]);
                trn::store32(A, r, c0, pk[0]);
                if (NB == 2) {
                    mk.y = trn::forward32(v[NB - 1], bias + l * W + c0 + 32, pk[NB - 1]);
                    trn::store32(A, r, c0 + 32, pk[NB - 1]);
                }
                if (l + 1 < L) {
                    mask[(size_t)l * 256] = mk;   // of H_{l+1}
                    a_done();
                }
            }
            if (!alive) break;
            // ---- output layer (FP32, BF16 weights): the row's sum runs over the first half's columns,
            // then over the second half's, which takes the loss
            float y0 = wout[2 * W], y1 = wout[2 * W + 1];
            auto fold = [&]() {
#pragma unroll
                for (int q = 0; q < NB; ++q)
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const int k = c0 + 32 * q + 2 * e;
                        const float2 w0 = *reinterpret_cast<const float2 *>(wout + k);
                        const float2 w1 = *reinterpret_cast<const float2 *>(wout + W + k);
                        const float h0 = trn::bf_lo(pk[q][e]), h1 = trn::bf_hi(pk[q][e]);
                        y0 = fmaf(w0.x, h0, fmaf(w0.y, h1, y0));
                        y1 = fmaf(w1.x, h0, fmaf(w1.y, h1, y1));
                    }
            };
            if (hf == 0) {
                fold();
                yp[r] = make_float2(y0, y1);
            }
            epilogue_sync();
            if (hf == 1) {
                y0 = yp[r].x;
                y1 = yp[r].y;
                fold();
                float dm = 0.0f, da = 0.0f;
                if (kept) {
                    const float al = a.hit_star[i];
                    const float bce = fmaxf(y1, 0.0f) - al * y1 + log1pf(expf(-fabsf(y1)));
                    part += 0.1f * bce / (float)a.B;
                    if (al > 0.5f) {
                        const float e = y0 - a.m_star[i];
                        part += e * e / n_hit;
                        dm = 2.0f * e / n_hit;
                    }
                    da = 0.1f * (1.0f / (1.0f + expf(-y1)) - al) / (float)a.B;
                }
                dy[r] = make_float2(dm, da);
            }
            epilogue_sync();
            // ---- dW_out, db_out of this tile (H_L is in A), then dZ_{L-1} over it
#pragma unroll 4
            for (int j = 0; j < kTileB / RS; ++j) {
                const int rr = rs + j * RS;
                const uint4 h = *reinterpret_cast<const uint4 *>(A + cg * 2048 + rr * 16);
                const float2 g = dy[rr];
                const uint32_t hw[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    ow[0][2 * e] = fmaf(g.x, trn::bf_lo(hw[e]), ow[0][2 * e]);
                    ow[0][2 * e + 1] = fmaf(g.x, trn::bf_hi(hw[e]), ow[0][2 * e + 1]);
                    ow[1][2 * e] = fmaf(g.y, trn::bf_lo(hw[e]), ow[1][2 * e]);
                    ow[1][2 * e + 1] = fmaf(g.y, trn::bf_hi(hw[e]), ow[1][2 * e + 1]);
                }
                if (cg == 0) { ob[0] += g.x; ob[1] += g.y; }
            }
            const float2 g = dy[r];
#pragma unroll
            for (int q = 0; q < NB; ++q)
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const int k = c0 + 32 * q + 2 * e;
                    const float2 w0 = *reinterpret_cast<const float2 *>(wout + k);
                    const float2 w1 = *reinterpret_cast<const float2 *>(wout + W + k);
                    const float g0 = trn::pos_lo(pk[q][e]) ? w0.x * g.x + w1.x * g.y : 0.0f;
                    const float g1 = trn::pos_hi(pk[q][e]) ? w0.y * g.x + w1.y * g.y : 0.0f;
                    pk[q][e] = pack_bf16(g0, g1);
                }
            epilogue_sync();                      // every read of H_L is done
#pragma unroll
            for (int q = 0; q < NB; ++q) trn::store32(A, r, c0 + 32 * q, pk[q]);
            a_done();
            // ---- backward
            for (int l = L - 1; l >= 1 && alive; --l) {
                const uint2 pm = mask[(size_t)(l - 1) * 256];   // of H_l
                if (!(alive = acc_wait())) break;
                uint32_t v[NB][32];
#pragma unroll
                for (int q = 0; q < NB; ++q) tmem_ld32(tacc + 32 * q, v[q]);
#pragma unroll
                for (int q = 0; q < NB; ++q) tmem_wait_ld(v[q]);
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    const uint32_t m = q ? pm.y : pm.x;
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        pk[q][e] = pack_bf16((m >> (2 * e)) & 1u ? __uint_as_float(v[q][2 * e]) : 0.0f,
                                             (m >> (2 * e + 1)) & 1u ? __uint_as_float(v[q][2 * e + 1]) : 0.0f);
                    trn::store32(A, r, c0 + 32 * q, pk[q]);
                }
                a_done();
            }
            if (alive) alive = acc_wait();        // dZ_0 has left A
        }
        // ---- the block's sums
#pragma unroll
        for (int o = 0; o < 2; ++o) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                for (int off = RS / 2; off; off >>= 1) ow[o][e] += __shfl_xor_sync(0xffffffffu, ow[o][e], off);
                if (rs == 0) a.s.outp[(size_t)blockIdx.x * (2 * W + 2) + o * W + cg * 8 + e] = ow[o][e];
            }
            for (int off = RS / 2; off; off >>= 1) ob[o] += __shfl_xor_sync(0xffffffffu, ob[o], off);
            if (threadIdx.x == 0) a.s.outp[(size_t)blockIdx.x * (2 * W + 2) + 2 * W + o] = ob[o];
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
    if (warp == 8) tmem_dealloc(tmem, W < 128 ? 64 : 128);
}

// ---- weight-gradient jobs: one per hidden layer -----------------------------------------------------
struct TcJobs {
    TcTrainScratch s;
    int W, tiles;
    __device__ __forceinline__ trn::WgradJob get(int l) const
    {
        const int fi = l == 0 ? kNedfIn : W, fip = l == 0 ? kNedfInPad : W;
        const size_t img = trn::img_bytes(W);
        trn::WgradJob j;
        j.a = s.zimg + (size_t)l * tiles * img;
        j.b = l == 0 ? s.ximg : s.himg + (size_t)(l - 1) * tiles * img;
        j.a_stride = j.a_bytes = (uint32_t)img;
        j.b_stride = j.b_bytes = (uint32_t)trn::img_bytes(fip);
        j.N = fip; j.n_valid = fi; j.m_valid = W; j.seg = W; j.fi = fi; j.bias = true;
        j.w_off[0] = j.w_off[1] = packed_off(l, W);
        j.b_off[0] = j.b_off[1] = packed_off(l, W) + (long long)fi * W;
        return j;
    }
};

// ---- the fixed-order sums, and Adam -----------------------------------------------------------------
struct FinishArgs {
    TcTrainScratch s;
    int splits, chains, n_hitp, L, W, hidden_blocks;
    long long stride;                              // floats from one split's partial to the next
    float *grad;                                   // or null
    float *loss;
    float *master, *kernel_w, *m, *v;              // master null: no Adam step
    float lr, c1, c2;
};

__global__ void __launch_bounds__(256) k_tc_finish(const __grid_constant__ FinishArgs a)
{
    const long long n_hid = packed_off(a.L, a.W);
    long long i = -1;
    float g = 0.0f;
    if ((int)blockIdx.x < a.hidden_blocks) {       // a thread per hidden weight, splits in order
        i = blockIdx.x * 256ll + threadIdx.x;
        if (i >= n_hid) return;
#pragma unroll 8
        for (int z = 0; z < a.splits; ++z) g += a.s.partial[(size_t)z * a.stride + i];
    } else {                                       // a warp per output-layer weight
        const int lane = threadIdx.x & 31, n_out = 2 * a.W + 2;
        const int k = ((int)blockIdx.x - a.hidden_blocks) * 8 + (threadIdx.x >> 5);
        if (k < n_out) {
            for (int c = lane; c < a.chains; c += 32) g += a.s.outp[(size_t)c * n_out + k];
            i = lane == 0 ? n_hid + k : -1;
        } else if (k == n_out) {                   // one warp more: the loss
            float h = 0.0f;
            for (int c = lane; c < a.chains; c += 32) g += a.s.lossp[c];
            for (int c = lane; c < a.n_hitp; c += 32) h += a.s.hitp[c];
            for (int off = 16; off; off >>= 1) h += __shfl_xor_sync(0xffffffffu, h, off);
            if (lane == 0) a.loss[1] = h;
        }
        for (int off = 16; off; off >>= 1) g += __shfl_xor_sync(0xffffffffu, g, off);
        if (k == n_out && lane == 0) a.loss[0] = g;
        if (i < 0) return;
    }
    if (a.grad) a.grad[i] = g;
    if (a.master) {
        const float th = adam_step(a.master[i], g, a.m[i], a.v[i], a.lr, a.c1, a.c2);
        a.master[i] = th;
        a.kernel_w[kernel_index(i, a.L, a.W)] = th;
    }
}

// ---- one forward / backward pass ----------------------------------------------------------------
template <int W>
static cudaError_t run_tc(const TrainLaunch &L, const float *o, const float *d, const float *m_star,
                          const float *hit_star, long long start, long long n, int B, FinishArgs f)
{
    cudaStream_t st = L.stream;
    const int nl = L.hidden, tiles = (B + kTileB - 1) / kTileB;
    TcTrainScratch s;
    carve_tc(L.scratch, B, nl, W, L.n_params, L.num_sms, &s);
    k_tc_prep<<<L.num_sms, 256, 0, st>>>(L.master, s.wimg, nl, W, hit_star, start, n, B, s.hitp);
    ChainArgs c{};
    c.rb = L.rb;
    c.o = o; c.d = d; c.m_star = m_star; c.hit_star = hit_star;
    c.start = start; c.n = n; c.B = B; c.tiles = tiles; c.L = nl; c.n_hitp = L.num_sms;
    c.master = L.master; c.s = s; c.status = L.status;
    const int sm = ChainShape<W>::FIXED + nl * W * 4;
    cudaError_t e = cudaFuncSetAttribute(k_tc_chain<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    if (e != cudaSuccess) return e;
    const int chains = std::min(tiles, 2 * L.num_sms);
    k_tc_chain<W><<<chains, kChainThreads, sm, st>>>(c);
    const int splits = trn::wgrad_splits(nl, tiles, L.num_sms);
    // stages of 32 KB + 32 KB (W = 64: its 16 KB of dZ and what follows it in the stage fill the M = 128
    // rows; the rows past W are not written)
    e = trn::wgrad<3, 32768, 32768, 256>(TcJobs{s, W, tiles}, nl, splits, tiles, s.partial,
                                        partial_stride(L.n_params), L.status, st);
    if (e != cudaSuccess) return e;
    f.s = s;
    f.splits = splits; f.chains = chains; f.n_hitp = L.num_sms; f.L = nl; f.W = W; f.stride = partial_stride(L.n_params);
    f.loss = L.loss;
    f.hidden_blocks = (int)((packed_off(nl, W) + 255) / 256);
    k_tc_finish<<<f.hidden_blocks + (2 * W + 2 + 1 + 7) / 8, 256, 0, st>>>(f);
    return cudaGetLastError();
}

static cudaError_t tc_fwd_bwd(const TrainLaunch &L, const float *o, const float *d, const float *m_star,
                              const float *hit_star, long long start, long long n, int B, const FinishArgs &f)
{
    switch (L.width) {
    case 64: return run_tc<64>(L, o, d, m_star, hit_star, start, n, B, f);
    case 128: return run_tc<128>(L, o, d, m_star, hit_star, start, n, B, f);
    default: return cudaErrorInvalidValue;
    }
}

bool train_tc_supported(int width, int hidden) { return (width == 64 || width == 128) && hidden >= 1 && hidden <= 16; }

cudaError_t launch_loss_grad_tc(const TrainLaunch &L, const float *o, const float *d, const float *m_star,
                                const float *hit_star, int n, float *grad)
{
    FinishArgs f{};
    f.grad = grad;
    return tc_fwd_bwd(L, o, d, m_star, hit_star, 0, n, n, f);
}

cudaError_t launch_train_step_tc(const TrainLaunch &L, const float *o, const float *d, const float *m_star,
                                 const float *hit_star, long long n_rays, long long start, int batch, float *adam_m,
                                 float *adam_v, int step, float lr)
{
    FinishArgs f{};
    f.master = L.master; f.kernel_w = L.kernel_w; f.m = adam_m; f.v = adam_v;
    f.lr = lr;
    f.c1 = (float)(1.0 - std::pow(0.9, step));
    f.c2 = (float)(1.0 - std::pow(0.999, step));
    return tc_fwd_bwd(L, o, d, m_star, hit_star, start, n_rays, batch, f);
}

}  // namespace nedf
