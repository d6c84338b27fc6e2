// Pieces of the tensor-core MLP engines shared by the one-SM engines (render_pipe.cu) and the
// SM-pair NeRF engine (render_pair.cu): tile shapes, the weight-blob offsets, the input encodings,
// the A-operand row stores and the layer epilogues (TMEM -> ReLU / rounding -> next A operand, or
// the output-layer fold).
#pragma once

#include "pipe_common.cuh"

namespace nedf {

using namespace tc;

// The NeDF's operands (78 inputs padded to 80) as 128-row halves; F8: hidden layers after the first in E4M3
// (first layer BF16; output layer on CUDA cores).
template <int N, bool F8>
struct PipeShape {
    static constexpr int K0 = kNedfInPad;                            // input width of layer 0
    // BF16: the bias of every layer is folded into its MMAs: two constant-one input columns times
    // the bias split into BF16 high and low parts.  Layer 0 has them inside its input padding;
    // hidden layers read them from a 16-column block at ONES, after every column a layer writes.
    // F8: layer 0 as in BF16; later biases are added (with the layer's scale) in the epilogue.
    static constexpr int ONES = K0 > N ? K0 : N;
    static constexpr int A_ROW = F8 ? (2 * K0 > N ? 2 * K0 : N) : 2 * (ONES + kKC);   // A bytes per row
    static constexpr int CHUNK = N * 32;                             // N x 16 BF16 or N x 32 E4M3
    static constexpr size_t A_BYTES = (size_t)kHalf * A_ROW;
};

// ---- weight blobs: per layer, chunks of 32 bytes of input per output row, each chunk N rows in the
// core-matrix layout (SBO 256 bytes).  Layer 0 (BF16) has K0 / 16 chunks with the bias in input
// columns K_in, K_in + 1 (high and low BF16 parts).  A BF16 hidden layer has N / 16 chunks plus
// one bias chunk (columns 0, 1); an E4M3 hidden layer has N / 32 chunks of W / s_l.  Then the fp32
// block: [w_out n_out x N (BF16 values)][b_out], and for E4M3 at pipe_f8_bias_off
// [bias L x N (row 0 unused)][s_l, L values (s_0 unused)].
__host__ __device__ inline size_t pipe_layer_off(int K0, int N, int l, bool f8)
{
    return l == 0 ? 0 : (size_t)K0 * N * 2 + (size_t)(l - 1) * (f8 ? (size_t)N * N : (size_t)(N + kKC) * N * 2);
}
__host__ __device__ inline size_t pipe_w_bytes(int K0, int N, int L, bool f8) { return pipe_layer_off(K0, N, L, f8); }
__host__ __device__ inline size_t pipe_f8_bias_off(int N, int n_out) { return ((size_t)n_out * N + n_out + 3) & ~(size_t)3; }
__host__ __device__ inline size_t pipe_f32_floats(int N, int L, int n_out, bool f8)
{
    const size_t b = pipe_f8_bias_off(N, n_out);
    return f8 ? (b + (size_t)L * N + L + 3) & ~(size_t)3 : b;
}
// ---- encodings into a BF16 A row (identity, sine blocks, cosine blocks; 2^k frequencies from the
// double-angle identities applied to sincos(x)) ---------------------------------------------------
template <int NIN, int F>
__device__ __forceinline__ void pipe_encode(const float *x, float *out)
{
#pragma unroll
    for (int c = 0; c < NIN; ++c) out[c] = x[c];
#pragma unroll
    for (int c = 0; c < NIN; ++c) {
        float s, co;
        sincosf(x[c], &s, &co);
#pragma unroll
        for (int k = 0; k < F; ++k) {
            out[NIN + k * NIN + c] = s;
            out[NIN + F * NIN + k * NIN + c] = co;
            float s2 = 2.0f * s * co;
            float c2 = (co - s) * (co + s);
            s = s2;
            co = c2;
        }
    }
}


// The same layout for E4M3 activations: 16 columns per 16-byte slice, slice stride 2048; one
// K = 32 MMA step again reads two slices (4 KB).
__device__ __forceinline__ uint32_t a_offset8(int r, int k)
{
    return (uint32_t)((k >> 4) * 2048 + (r >> 3) * 128 + (r & 7) * 16 + (k & 15));
}

// The encoded row as packed BF16 pairs: inputs, then the two constant-one columns the layer-0 bias is
// folded into, then zeros, K columns in all.
template <int K>
__device__ __forceinline__ void pipe_pack_row(const float *f, int n_valid, uint32_t (&pk)[K / 2])
{
#pragma unroll
    for (int k = 0; k < K; k += 2) {
        const float v0 = k < n_valid ? f[k] : (k < n_valid + 2 ? 1.0f : 0.0f);
        const float v1 = k + 1 < n_valid ? f[k + 1] : (k + 1 < n_valid + 2 ? 1.0f : 0.0f);
        pk[k / 2] = pack_bf16(v0, v1);
    }
}
// KG: bytes between 8-column groups (2048 for a 128-row half; 4096 for the 256 rows of a swapped
// NeDF tile, whose B operand spans both halves)
template <int K, int KG = 2048>
__device__ __forceinline__ void pipe_store_packed(uint8_t *A, int r, const uint32_t (&pk)[K / 2])
{
#pragma unroll
    for (int c = 0; c < K / 8; ++c)
        *reinterpret_cast<uint4 *>(A + (uint32_t)(c * KG + (r >> 3) * 128 + (r & 7) * 16)) =
            make_uint4(pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
}
template <int K, int KG = 2048>
__device__ __forceinline__ void pipe_store_row(uint8_t *A, int r, const float *f, int n_valid)
{
    uint32_t pk[K / 2];
    pipe_pack_row<K>(f, n_valid, pk);
    pipe_store_packed<K, KG>(A, r, pk);
}
// pipe_encode packed as it goes (NIN even: the inputs two by two, so every pair of neighbouring features
// comes together), with the constant-one columns and the padding: the same values without the K floats.
template <int NIN, int F, int K>
__device__ __forceinline__ void pipe_encode_packed(float *x, uint32_t (&pk)[K / 2])
{
    static_assert(NIN % 2 == 0, "pairs of inputs");
    constexpr int n = NIN * (2 * F + 1);
#pragma unroll
    for (int c = 0; c < NIN; c += 2) {
        float s0, c0, s1, c1;
        sincosf(x[c], &s0, &c0);
        sincosf(x[c + 1], &s1, &c1);
        pk[c / 2] = pack_bf16(x[c], x[c + 1]);
#pragma unroll
        for (int k = 0; k < F; ++k) {
            pk[(NIN + k * NIN + c) / 2] = pack_bf16(s0, s1);
            pk[(NIN + F * NIN + k * NIN + c) / 2] = pack_bf16(c0, c1);
            const float d0 = 2.0f * s0 * c0, e0 = (c0 - s0) * (c0 + s0), d1 = 2.0f * s1 * c1, e1 = (c1 - s1) * (c1 + s1);
            s0 = d0; c0 = e0; s1 = d1; c1 = e1;
        }
        // one pair of inputs after another (three at once would take 60 registers more)
#pragma unroll
        for (int k = 0; k < 2 * F; ++k) asm volatile("" : "+r"(pk[(NIN + k * NIN + c) / 2]));
        if (c + 2 < NIN) asm volatile("" : "+f"(x[c + 2]), "+f"(x[c + 3]));
    }
#pragma unroll
    for (int k = n; k < K; k += 2) pk[k / 2] = k == n ? pack_bf16(1.0f, 1.0f) : 0u;
}

// A quarter of the NeRF's input row (90 features, two ones, four zeros) as packed BF16 pairs.  Position
// features: x, sin(2^k x) (k = 0..9, coordinate fastest) are columns 0..32, cos(2^k x) 33..62, the direction's
// first coordinate is column 63; `high` picks columns 32..63 over 0..31.  The values are pipe_encode's.
__device__ __forceinline__ void nerf_encode_position(const float *x, bool high, uint32_t (&pk)[16])
{
    float f[32];                                      // columns 32 high ..
    float s[3], c[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        sincosf(x[i], &s[i], &c[i]);
        if (!high) f[i] = x[i];
    }
    if (high) f[31] = x[3];
#pragma unroll
    for (int k = 0; k < 10; ++k) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int cs = 3 + 3 * k + i, cc = 33 + 3 * k + i - 32;
            if (cs < 32) { if (!high) f[cs] = s[i]; }
            else if (high) f[cs - 32] = s[i];
            if (high) f[cc] = c[i];
            const float s2 = 2.0f * s[i] * c[i], c2 = (c[i] - s[i]) * (c[i] + s[i]);
            s[i] = s2;
            c[i] = c2;
        }
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) pk[k] = pack_bf16(f[2 * k], f[2 * k + 1]);
}
// Columns 64..95: the direction's other coordinates, sin and cos of it (4 frequencies), ones and zeros.
__device__ __forceinline__ void nerf_encode_direction(const float *d, uint32_t (&pk)[16])
{
    float f[kNerfInPad - 63];
    pipe_encode<3, 4>(d, f);
    f[27] = f[28] = 1.0f;
    f[29] = f[30] = f[31] = f[32] = 0.0f;
#pragma unroll
    for (int k = 0; k < 16; ++k) pk[k] = pack_bf16(f[2 * k + 1], f[2 * k + 2]);
}

// ReLU and BF16 of C accumulator columns of this thread's row (the bias is already in them),
// stored as A columns [c0, c0 + C) of row r.
template <int C>
__device__ __forceinline__ void epi_convert(const uint32_t (&v)[C], uint8_t *A, int r, int c0)
{
#pragma unroll
    for (int q = 0; q < C / 8; ++q) {
        const uint32_t *u = v + 8 * q;
        uint4 pk;
        pk.x = pack_bf16_relu(__uint_as_float(u[0]), __uint_as_float(u[1]));
        pk.y = pack_bf16_relu(__uint_as_float(u[2]), __uint_as_float(u[3]));
        pk.z = pack_bf16_relu(__uint_as_float(u[4]), __uint_as_float(u[5]));
        pk.w = pack_bf16_relu(__uint_as_float(u[6]), __uint_as_float(u[7]));
        *reinterpret_cast<uint4 *>(A + a_offset(r, c0 + 8 * q)) = pk;
    }
}

// Four accumulator columns as x = acc (AFF false: bias already in it) or acc * s + bias (AFF; bias 16-byte
// aligned): one load of four biases and two packed FMAs (s2 = (s, s)).  The E4M3 engines' steps are
// bound by the issue slots of their epilogues (4096-instance E4M3 frame
// 29.1 -> 28.5 ms against scalar FMAs with scalar bias loads).
template <bool AFF>
__device__ __forceinline__ void epi_affine4(const uint32_t *u, const float *bias, uint64_t s2, float (&x)[4])
{
    if (AFF) {
        const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(bias);
        split2(fma2(pair2(u[0], u[1]), s2, b.x), x[0], x[1]);
        split2(fma2(pair2(u[2], u[3]), s2, b.y), x[2], x[3]);
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = __uint_as_float(u[e]);
    }
}

// E4M3 activations of C columns: ReLU and E4M3, stored as A columns [c0, c0 + C) of row r.
template <bool AFF, int C>
__device__ __forceinline__ void epi_convert8(const uint32_t (&v)[C], const float *bias, float s, uint8_t *A, int r, int c0)
{
    const uint64_t s2 = pair2(s, s);
    uint32_t w[C / 4];
#pragma unroll
    for (int q = 0; q < C / 4; ++q) {
        float x[4];
        epi_affine4<AFF>(v + 4 * q, bias + 4 * q, s2, x);
        w[q] = pack_e4m3_relu(x[0], x[1]) | (pack_e4m3_relu(x[2], x[3]) << 16);
    }
#pragma unroll
    for (int q = 0; q < C / 16; ++q)
        *reinterpret_cast<uint4 *>(A + a_offset8(r, c0 + 16 * q)) = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
}

// Last hidden layer: ReLU and BF16 rounding of 32 columns, folded into the NOUT outputs (w_out
// rows of length N; 16-byte aligned at every multiple of 4 columns).  The weights are read four
// columns per load; the FMAs run in column order, so the sums are those of a column-by-column loop.
template <int NOUT, int N, int C = 32>
__device__ __forceinline__ void epi_output(const uint32_t (&v)[C], const float *wout, float *out)
{
#pragma unroll
    for (int jj = 0; jj < C; jj += 4) {
        float4 w[NOUT];
#pragma unroll
        for (int o = 0; o < NOUT; ++o) w[o] = *reinterpret_cast<const float4 *>(wout + o * N + jj);
        const uint32_t p0 = pack_bf16_relu(__uint_as_float(v[jj]), __uint_as_float(v[jj + 1]));
        const uint32_t p1 = pack_bf16_relu(__uint_as_float(v[jj + 2]), __uint_as_float(v[jj + 3]));
        const float h0 = __uint_as_float(p0 << 16), h1 = __uint_as_float(p0 & 0xFFFF0000u);
        const float h2 = __uint_as_float(p1 << 16), h3 = __uint_as_float(p1 & 0xFFFF0000u);
#pragma unroll
        for (int o = 0; o < NOUT; ++o) {
            out[o] = fmaf(h1, w[o].y, fmaf(h0, w[o].x, out[o]));
            out[o] = fmaf(h3, w[o].w, fmaf(h2, w[o].z, out[o]));
        }
    }
}

// The same with E4M3 rounding of the last hidden activation (bias and weights four columns per
// load).
template <int NOUT, int N, bool AFF, int C = 32>
__device__ __forceinline__ void epi_output8(const uint32_t (&v)[C], const float *bias, float s, const float *wout, float *out)
{
    const uint64_t s2 = pair2(s, s);
#pragma unroll
    for (int jj = 0; jj < C; jj += 4) {
        float4 w[NOUT];
#pragma unroll
        for (int o = 0; o < NOUT; ++o) w[o] = *reinterpret_cast<const float4 *>(wout + o * N + jj);
        float x[4];
        epi_affine4<AFF>(v + jj, bias + jj, s2, x);
        float h0, h1, h2, h3;
        unpack_e4m3(pack_e4m3_relu(x[0], x[1]), h0, h1);
        unpack_e4m3(pack_e4m3_relu(x[2], x[3]), h2, h3);
#pragma unroll
        for (int o = 0; o < NOUT; ++o) {
            out[o] = fmaf(h1, w[o].y, fmaf(h0, w[o].x, out[o]));
            out[o] = fmaf(h3, w[o].w, fmaf(h2, w[o].z, out[o]));
        }
    }
}

// One layer's epilogue over the N accumulator columns of this thread's row, TMEM loads
// double-buffered (block b + 1 loads while block b is converted).  LAST: fold into the outputs;
// otherwise write the next layer's A operand (BF16, or E4M3 when F8).
template <int N, int NOUT, bool F8, bool AFF, bool LAST>
__device__ __forceinline__ void epi_layer(uint32_t tmem_row, uint8_t *Ag, int r, const float *bias, float s,
                                          const float *wout, float *out)
{
    uint32_t va[32], vb[32];
    tmem_ld32(tmem_row, va);
    tmem_wait_ld(va);
#pragma unroll 1
    for (int c0 = 0; c0 < N; c0 += 64) {
        tmem_ld32(tmem_row + c0 + 32, vb);
        if (LAST) {
            if (F8) epi_output8<NOUT, N, AFF>(va, bias + c0, s, wout + c0, out);
            else epi_output<NOUT, N>(va, wout + c0, out);
        } else {
            if (F8) epi_convert8<AFF>(va, bias + c0, s, Ag, r, c0);
            else epi_convert(va, Ag, r, c0);
        }
        tmem_wait_ld(vb);
        if (c0 + 64 < N) tmem_ld32(tmem_row + c0 + 64, va);
        if (LAST) {
            if (F8) epi_output8<NOUT, N, AFF>(vb, bias + c0 + 32, s, wout + c0 + 32, out);
            else epi_output<NOUT, N>(vb, wout + c0 + 32, out);
        } else {
            if (F8) epi_convert8<AFF>(vb, bias + c0 + 32, s, Ag, r, c0 + 32);
            else epi_convert(vb, Ag, r, c0 + 32);
        }
        if (c0 + 64 < N) tmem_wait_ld(va);
    }
}

// The BF16 last layer's fold, 16 TMEM columns at a time: a quarter of the registers of epi_layer (the
// NeDF engine holds the next tile's packed inputs meanwhile; its other warps hide the loads).
template <int N, int NOUT>
__device__ __forceinline__ void epi_fold(uint32_t tmem_row, const float *wout, float *out)
{
#pragma unroll 1
    for (int c0 = 0; c0 < N; c0 += 16) {
        uint32_t v[16];
        tmem_ld16(tmem_row + c0, v);
        tmem_wait_ld(v);
        epi_output<NOUT, N, 16>(v, wout + c0, out);
    }
}

// 32 rows of one feature (ReLU, BF16): four 16-byte vectors of eight rows, 128 bytes apart.
__device__ __forceinline__ void epi_rows8(const uint32_t (&v)[32], uint8_t *dst)
{
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const uint32_t *u = v + 8 * b;
        uint4 pk;
        pk.x = pack_bf16_relu(__uint_as_float(u[0]), __uint_as_float(u[1]));
        pk.y = pack_bf16_relu(__uint_as_float(u[2]), __uint_as_float(u[3]));
        pk.z = pack_bf16_relu(__uint_as_float(u[4]), __uint_as_float(u[5]));
        pk.w = pack_bf16_relu(__uint_as_float(u[6]), __uint_as_float(u[7]));
        *reinterpret_cast<uint4 *>(dst + b * 128) = pk;
    }
}

// Epilogue of a swapped NeDF layer (D = W H^T: TMEM lane = output feature f, column = tile row):
// the 128 columns from tcol are rows row0 .. row0 + 127.  Each value is ReLU'd, rounded to BF16 and
// stored as the next layer's B operand, MN-major: 16-feature chunk f / 16 at 8 KB steps, 8-feature
// group at 4 KB, feature f % 8 at 16 bytes, rows contiguous in 16-byte vectors of eight (128 bytes
// per 8-row group).  TMEM loads double-buffered as in epi_layer.
__device__ __forceinline__ void epi_swapped(uint32_t tcol, uint8_t *H, int f, int row0)
{
    uint8_t *dst = H + (f >> 4) * 8192 + ((f >> 3) & 1) * 4096 + (f & 7) * 16 + (row0 >> 3) * 128;
    uint32_t va[32], vb[32];
    tmem_ld32(tcol, va);
    tmem_wait_ld(va);
#pragma unroll 1
    for (int c0 = 0; c0 < 128; c0 += 64) {
        tmem_ld32(tcol + c0 + 32, vb);
        epi_rows8(va, dst + (c0 >> 3) * 128);
        tmem_wait_ld(vb);
        if (c0 + 64 < 128) tmem_ld32(tcol + c0 + 64, va);
        epi_rows8(vb, dst + ((c0 + 32) >> 3) * 128);
        if (c0 + 64 < 128) tmem_wait_ld(va);
    }
}
}  // namespace nedf
