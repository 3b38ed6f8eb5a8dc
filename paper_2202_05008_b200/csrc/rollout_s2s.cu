// Sequence-to-sequence addition task with an LSTM encoder-decoder policy (paper Section 3,
// "Seq2Seq Learning"): a single-step task whose fitness is minus the mean cross-entropy of the
// answer digits over a batch of queries that every member sees.
//
// Conventions: tokens '0'..'9' -> 0..9, '+' -> 10, '=' -> 11; the encoder reads "a+b" (2 nd + 1
// tokens), the decoder is fed '=' and then the true answer digits and must produce the nd + 1
// digits of the sum; gate order (input, forget, cell, output); flat parameters enc.Wx[4h][12],
// enc.Wh[4h][h], enc.b[4h], dec.*, out.W[12][h], out.b[12].  A cell's pre-activation is one
// contraction [Wh | Wx | b] . [h; onehot(token); 1] with bf16 operands and fp32 accumulation; the
// read-out out.W . h likewise.
//
//   k_s2s_simple  CUDA cores, one block per (member, 16 queries): the plain version, which also writes logits.
//   k_s2s_mma     h = 32, 64, 96: warp-level tensor-core products, weights and cell state in registers.
//   k_s2s_tc      tcgen05, one block per (member, 128 queries), one block per SM.  The member's
//                 [4h = 512] x [K = 144] weight tile (bf16, 144 KB) stays in shared memory for a
//                 whole phase (encoder, then decoder); the B operand is the hidden state of the 128
//                 queries plus their one-hot token and a constant 1, so one chain of 9 MMAs per gate
//                 produces the complete pre-activation in TMEM (2 halves x 4 gates x 64 columns =
//                 all 512 columns).  The queries are two halves of 64 whose steps alternate: while
//                 the epilogue warps of one half apply the gate non-linearities (thread = hidden
//                 unit = TMEM lane, cell state in registers) and write the new hidden state straight
//                 back into the B operand, the tensor cores work on the other half.  The rows of the
//                 sigmoid gates are halved when staged, so every non-linearity is one tanh of the
//                 special-function unit; that unit (5 tanh per cell and step) is what bounds the
//                 kernel, not the tensor cores.  The decoder's read-out runs on the CUDA cores from
//                 the B operand while the next step's MMAs are in flight: as warp-level products a generation of
//                 1,024 members x 128 queries takes 641 us instead of 655, but these cut their sums off
//                 where additions round (logits of 128 positive terms: relative error 3.4e-7 RMS, all of one sign,
//                 against 0.7e-7 without bias).  The logits are kept and
//                 the cross-entropy is taken once per item.  The next cell's weights are prefetched
//                 into L2 while the current phase computes.  Every wait is bounded.
#include "internal.h"
#include "async.cuh"
#include "noise.cuh"
#include "umma.cuh"
#include "fp32x2.cuh"

namespace evo {

constexpr int kVocab = 12;
constexpr int kTokPlus = 10, kTokEq = 11;
constexpr int kS2sMaxDigits = 4;
constexpr int kS2sMaxTe = 2 * kS2sMaxDigits + 1, kS2sMaxTd = kS2sMaxDigits + 1;

__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// Query i of a generation: a, b uniform on [0, 10^nd) from the first two words of stream 6.
__device__ __forceinline__ void s2s_query(const PhiloxKey& key, uint32_t generation, uint32_t i, uint32_t nd,
                                          uint8_t* enc, uint8_t* dec, uint8_t* tgt)
{
    uint32_t range = 1;
    for (uint32_t k = 0; k < nd; ++k) range *= 10u;
    const uint4 w = philox4x32_10(i, 0u, generation, 6u, key);
    const uint32_t a = __umulhi(w.x, range), b = __umulhi(w.y, range), sum = a + b;
    uint32_t div = range / 10u;
    for (uint32_t k = 0; k < nd; ++k, div /= 10u) {
        enc[k] = static_cast<uint8_t>((a / div) % 10u);
        enc[nd + 1 + k] = static_cast<uint8_t>((b / div) % 10u);
    }
    enc[nd] = kTokPlus;
    div = range;
    for (uint32_t k = 0; k <= nd; ++k, div /= 10u) tgt[k] = static_cast<uint8_t>((sum / div) % 10u);
    dec[0] = kTokEq;
    for (uint32_t k = 1; k <= nd; ++k) dec[k] = tgt[k - 1];
}

__device__ __forceinline__ float sigmoid_acc(float x) { return 1.0f / (1.0f + expf(-x)); }

// cross-entropy of one position from its 12 logits
__device__ __forceinline__ float token_loss(const float* lg, int target)
{
    float mx = lg[0];
#pragma unroll
    for (int o = 1; o < kVocab; ++o) mx = fmaxf(mx, lg[o]);
    float se = 0.f;
#pragma unroll
    for (int o = 0; o < kVocab; ++o) se += expf(lg[o] - mx);
    return (mx + logf(se)) - lg[target];
}

struct S2sArgs {
    const float* theta; uint32_t ldD, P;
    uint32_t h, nd, B;
    uint32_t k0, k1;
    const DeviceStatus* status;  // holds the generation counter
    float* partial;              // [P][n_chunks] sums of token losses
    uint32_t n_chunks;
    uint32_t per_chunk;          // k_s2s_tc: queries per item
    float* logits;               // nullable: [P][B][nd+1][12] (simple kernel only)
};

// ------------------------------------------------------------------------------------------
// CUDA-core version: thread = hidden unit, 16 queries per block, weights read through the caches.
// ------------------------------------------------------------------------------------------
constexpr int kSimpleQ = 16;

__global__ void __launch_bounds__(128)
k_s2s_simple(const S2sArgs a)
{
    __shared__ __align__(16) float hs[kSimpleQ][128];           // bf16-rounded hidden state
    __shared__ float lg[kSimpleQ][kVocab];
    __shared__ uint8_t enc[kSimpleQ][kS2sMaxTe], dec[kSimpleQ][kS2sMaxTd], tgt[kSimpleQ][kS2sMaxTd];
    __shared__ float loss_s[kSimpleQ];
    const uint32_t h = a.h, r = threadIdx.x, member = blockIdx.x, q0 = blockIdx.y * kSimpleQ;
    const uint32_t nq = min(static_cast<uint32_t>(kSimpleQ), a.B - q0);
    const uint32_t Te = 2 * a.nd + 1, Td = a.nd + 1;
    const PhiloxKey key = philox_key(a.k0, a.k1);
    if (r < kSimpleQ) {
        s2s_query(key, a.status->generation, q0 + min(r, nq - 1u), a.nd, enc[r], dec[r], tgt[r]);
        loss_s[r] = 0.f;
    }
    for (uint32_t s = 0; s < kSimpleQ; ++s) hs[s][r] = 0.f;
    float c[kSimpleQ];
#pragma unroll
    for (int s = 0; s < kSimpleQ; ++s) c[s] = 0.f;
    const float* p = a.theta + static_cast<size_t>(member) * a.ldD;
    const size_t cell = static_cast<size_t>(4) * h * kVocab + static_cast<size_t>(4) * h * h + 4u * h;
    const float* oW = p + 2 * cell;
    const float* ob = oW + static_cast<size_t>(kVocab) * h;
    __syncthreads();

    for (uint32_t t = 0; t < Te + Td; ++t) {
        const bool decoding = t >= Te;
        const float* Wx = p + (decoding ? cell : 0);
        const float* Wh = Wx + static_cast<size_t>(4) * h * kVocab;
        const float* bb = Wh + static_cast<size_t>(4) * h * h;
        float acc[4][kSimpleQ];
#pragma unroll
        for (int g = 0; g < 4; ++g)
#pragma unroll
            for (int s = 0; s < kSimpleQ; ++s) acc[g][s] = 0.f;
        if (r < h) {
            for (uint32_t k = 0; k < h; k += 4) {
                float4 w[4];
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    w[g] = __ldg(reinterpret_cast<const float4*>(Wh + (static_cast<size_t>(g) * h + r) * h + k));
                    w[g].x = bf16_round(w[g].x); w[g].y = bf16_round(w[g].y);
                    w[g].z = bf16_round(w[g].z); w[g].w = bf16_round(w[g].w);
                }
#pragma unroll
                for (int s = 0; s < kSimpleQ; ++s) {
                    const float4 x = *reinterpret_cast<const float4*>(&hs[s][k]);
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        acc[g][s] = fmaf(w[g].x, x.x, acc[g][s]);
                        acc[g][s] = fmaf(w[g].y, x.y, acc[g][s]);
                        acc[g][s] = fmaf(w[g].z, x.z, acc[g][s]);
                        acc[g][s] = fmaf(w[g].w, x.w, acc[g][s]);
                    }
                }
            }
        }
        __syncthreads();                                       // every thread is done reading hs
        if (r < h) {
            float bias[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) bias[g] = bf16_round(bb[g * h + r]);
#pragma unroll
            for (int s = 0; s < kSimpleQ; ++s) {
                const uint32_t tok = decoding ? dec[s][t - Te] : enc[s][t];
                float pre[4];
#pragma unroll
                for (int g = 0; g < 4; ++g)
                    pre[g] = acc[g][s] + bf16_round(Wx[(static_cast<size_t>(g) * h + r) * kVocab + tok]) + bias[g];
                const float ig = sigmoid_acc(pre[0]), fg = sigmoid_acc(pre[1]);
                const float gg = tanhf(pre[2]), og = sigmoid_acc(pre[3]);
                c[s] = fmaf(fg, c[s], ig * gg);
                hs[s][r] = bf16_round(og * tanhf(c[s]));
            }
        }
        __syncthreads();
        if (decoding) {
            for (uint32_t idx = r; idx < kSimpleQ * kVocab; idx += blockDim.x) {
                const uint32_t s = idx / kVocab, o = idx % kVocab;
                float v = 0.f;
                for (uint32_t k = 0; k < h; ++k) v = fmaf(bf16_round(oW[o * h + k]), hs[s][k], v);
                lg[s][o] = v + ob[o];
                if (a.logits && s < nq)
                    a.logits[((static_cast<size_t>(member) * a.B + q0 + s) * Td + (t - Te)) * kVocab + o] = lg[s][o];
            }
            __syncthreads();
            if (r < nq) loss_s[r] += token_loss(lg[r], tgt[r][t - Te]);
            __syncthreads();
        }
    }
    if (r == 0) {
        float total = 0.f;
        for (uint32_t s = 0; s < nq; ++s) total += loss_s[s];
        a.partial[static_cast<size_t>(member) * a.n_chunks + blockIdx.y] = total;
    }
}

// LANES per member.  One: the sums of its chunks in order.  Four: every fourth sum each, then the lanes as a tree, for the sums of k_s2s_mma (one
// per 8 queries) where they are more than four.
template <int LANES>
__global__ void k_s2s_finalize(const float* __restrict__ partial, uint32_t P, uint32_t n_chunks, float inv_count,
                               float* __restrict__ fitness)
{
    dep_wait();
    dep_trigger();
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x, m = i / LANES, lane = i % LANES;
    float s = 0.f;
    if (m < P)
        for (uint32_t t = lane; t < n_chunks; t += LANES) s += partial[static_cast<size_t>(m) * n_chunks + t];
#pragma unroll
    for (int off = LANES / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (m < P && lane == 0u) fitness[m] = -s * inv_count;
}

// ------------------------------------------------------------------------------------------
// Narrow cells (h = 32, 64, 96) on warp-level tensor-core products.  A block takes (member, up to 8 TILES queries) at a time; a warp owns 8
// hidden units with all four of their gates, rows (input | forget) and (cell | output) of two 16-row operand tiles that
// it keeps in registers for a whole phase, so a lane's accumulators are the four pre-activations of its
// (unit, two queries) and the cell state never leaves its registers.  The hidden state travels through shared memory
// as the B operand [query][h; onehot(token); 1], two buffers, one barrier per step.
//
// The gates in fp32: sigma(x) = 1 / (1 + 2^(-x log2 e)), tanh(x) = 2 sigma(2 x) - 1.  The special-function unit, which takes 8
// clocks per warp for an exponential and 16 for a reciprocal, bounds the kernel, so a cell's four gates share one
// reciprocal and two cells share that of tanh(c): 64 clocks per cell and step.  The CUDA-core version took one
// fp32 multiply-add per weight and query on top: h = 64, 2 digits, 300 members x 100 queries: 765 us, here 67 us.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_bf16_first(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1), "f"(0.f));
}

// 2^(-x log2 e), held below 2^30 so that a product of four (1 + e) stays finite
__device__ __forceinline__ float gate_exp(float x)
{
    float e;
    asm("{\n\t.reg .f32 t;\n\tmul.f32 t, %1, 0fBFB8AA3B;\n\tmin.NaN.f32 t, t, 0f41F00000;\n\tex2.approx.ftz.f32 %0, t;\n\t}" : "=f"(e) : "f"(x));
    return e;
}
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// One LSTM cell's state from its pre-activations (that of the cell gate doubled); returns the output gate.
__device__ __forceinline__ float lstm_cell(float pi, float pf, float pg2, float po, float& c)
{
    const float a = gate_exp(pi) + 1.0f, b = gate_exp(pf) + 1.0f, d = gate_exp(po) + 1.0f, e = gate_exp(pg2) + 1.0f;
    const float ab = a * b, de = d * e, r = rcp_approx(ab * de);
    const float rab = r * de, rde = r * ab;
    c = fmaf(rab * a, c, rab * b * fmaf(2.0f, rde * d, -1.0f));
    return rde * e;
}
// tanh of two cell states (|c| is at most the number of steps, so nothing overflows)
__device__ __forceinline__ void tanh_two(float c0, float c1, float& t0, float& t1)
{
    float e0, e1;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(c0 * -2.885390082f));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(c1 * -2.885390082f));
    const float a = e0 + 1.0f, b = e1 + 1.0f, r = rcp_approx(a * b);
    t0 = fmaf(2.0f, r * b, -1.0f);
    t1 = fmaf(2.0f, r * a, -1.0f);
}

// A block has `chunk` n-tiles of a member, or (RUNS) a run of the n-tiles of all members, which are dealt out evenly to the blocks and
// worked off in pieces of one member and up to TILES tiles.  s2s_split.h chooses.
template <int H, int TILES, bool RUNS>
__global__ void __launch_bounds__(4 * H, H == 32 ? 6 : H == 64 ? 2 : 1)
k_s2s_mma(const S2sArgs a, uint32_t chunk)
{
    constexpr int KH = H / 16, KT = KH + 1, kWarps = H / 8, kQ = 8 * TILES, kOwn = (TILES + kWarps - 1) / kWarps;
    constexpr uint32_t kPitch = (H + 16) * 2 + 16;               // bytes per query of the operand: rows of 8 queries fall in distinct banks
    __shared__ __align__(16) unsigned char bop[2 * kQ * kPitch + 32];      // two buffers (the last row's last k-tile is read with the 16 bytes behind it)
    __shared__ __align__(16) uint4 out_w[KH * 32];               // read-out weights in operand order
    __shared__ float out_b[16];
    __shared__ uint8_t enc[kQ][kS2sMaxTe], dec[kQ][kS2sMaxTd], tgt[kQ][kS2sMaxTd];

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, g = lane >> 2, t4 = lane & 3;
    const uint32_t Te = 2 * a.nd + 1, Td = a.nd + 1, T = Te + Td;
    const PhiloxKey key = philox_key(a.k0, a.k1);
    dep_wait();
    dep_trigger();
    constexpr size_t cell = static_cast<size_t>(4) * H * kVocab + static_cast<size_t>(4) * H * H + 4u * H;
    uint32_t member = blockIdx.x, tile0 = blockIdx.y * chunk, nt = min(chunk, a.n_chunks - tile0);     // first n-tile and n-tiles of the piece
    uint32_t at = 0, run_end = 0;                                // this block's run, in tiles of all members
    if (RUNS) {
        const uint64_t all = static_cast<uint64_t>(a.P) * a.n_chunks;
        at = static_cast<uint32_t>(all * blockIdx.x / gridDim.x);
        run_end = static_cast<uint32_t>(all * (blockIdx.x + 1u) / gridDim.x);
    }
    do {
        if (RUNS) {
            member = at / a.n_chunks; tile0 = at % a.n_chunks;
            const uint32_t left = min(run_end - at, a.n_chunks - tile0), pieces = (left + TILES - 1u) / TILES;
            nt = (left + pieces - 1u) / pieces;
        }
        const uint32_t q0 = tile0 * 8u, nq = min(nt * 8u, a.B - q0);
        const float* p = a.theta + static_cast<size_t>(member) * a.ldD;
        if (RUNS) __syncthreads();                                   // the piece before is done with shared memory

        float loss[kOwn];                                            // of the n-tiles that this warp reads out
#pragma unroll
        for (int i = 0; i < kOwn; ++i) loss[i] = 0.f;
        if (tid < kQ) s2s_query(key, a.status->generation, q0 + min(static_cast<uint32_t>(tid), nq - 1u), a.nd, enc[tid], dec[tid], tgt[tid]);
        for (uint32_t i = tid; i < sizeof(bop) / 16u; i += 4 * H) reinterpret_cast<uint4*>(bop)[i] = make_uint4(0u, 0u, 0u, 0u);
        {
            const float* oW = p + 2 * cell;
            for (int i = tid; i < KH * 32; i += 4 * H) {
                const int k = (i >> 5) * 16 + 2 * (i & 3), r = (i & 31) >> 2;
                uint32_t v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {                    // rows r, r + 8; inputs k, k + 1 and k + 8, k + 9
                    const int row = r + 8 * (j & 1), col = k + 8 * (j >> 1);
                    v[j] = row < kVocab ? pack_bf16(__ldg(oW + row * H + col), __ldg(oW + row * H + col + 1)) : 0u;
                }
                out_w[i] = make_uint4(v[0], v[1], v[2], v[3]);
            }
            if (tid < 16) out_b[tid] = tid < kVocab ? __ldg(oW + kVocab * H + tid) : 0.f;
        }
        __syncthreads();
        auto write_token = [&](uint32_t buf, uint32_t n, uint32_t tok) {
            uint32_t w[8];
            const uint32_t one = (tok & 1u) ? 0x3F800000u : 0x00003F80u;      // bf16 1.0 in the upper / lower half
#pragma unroll
            for (uint32_t i = 0; i < 8u; ++i) w[i] = (i == (tok >> 1)) ? one : 0u;
            w[6] |= 0x00003F80u;                                      // input 12: the constant 1 of the bias
            uint4* dst = reinterpret_cast<uint4*>(bop + buf * (kQ * kPitch) + n * kPitch + H * 2);
            dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
            dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
        };
        if (tid < kQ) write_token(0u, tid, enc[tid][0]);

        float c[TILES][2];
#pragma unroll
        for (int j = 0; j < TILES; ++j) c[j][0] = c[j][1] = 0.f;
        const uint32_t bop0 = smem_u32(bop), ld_row = (lane & 7) * kPitch + 16u * (lane >> 3), st_row = lane * kPitch + 16u * warp;
        const int u = 8 * warp + g;                                   // this lane's hidden unit

        for (uint32_t phase = 0; phase < 2u; ++phase) {
            const float* Wx = p + (phase ? cell : 0);
            const float* Wh = Wx + static_cast<size_t>(4) * H * kVocab;
            const float* bb = Wh + static_cast<size_t>(4) * H * H;
            uint4 w[2][KT];
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int k = 0; k < KT; ++k) {
                    uint32_t v[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int gate = 2 * m + (j & 1), row = gate * H + u, col = 2 * t4 + 8 * (j >> 1);
                        const float s = gate == 2 ? 2.0f : 1.0f;      // the cell gate is doubled (exact in bf16)
                        if (k < KH) {
                            const float2 x = __ldg(reinterpret_cast<const float2*>(Wh + static_cast<size_t>(row) * H + 16 * k + col));
                            v[j] = pack_bf16(s * x.x, s * x.y);
                        } else {
                            const float x = col < kVocab ? __ldg(Wx + row * kVocab + col) : col == kVocab ? __ldg(bb + row) : 0.f;
                            const float y = col < kVocab ? __ldg(Wx + row * kVocab + col + 1) : 0.f;
                            v[j] = pack_bf16(s * x, s * y);
                        }
                    }
                    w[m][k] = make_uint4(v[0], v[1], v[2], v[3]);
                }
            __syncthreads();
            for (uint32_t t = phase ? Te : 0u; t < (phase ? T : Te); ++t) {
                const uint32_t src = bop0 + (t & 1u) * (kQ * kPitch), dst = bop0 + ((t + 1u) & 1u) * (kQ * kPitch);
#pragma unroll
                for (int j4 = 0; j4 < TILES; j4 += 4) {
                    if (static_cast<uint32_t>(j4) < nt) {
                        uint32_t hp[4];
#pragma unroll
                        for (int jj = 0; jj < 4; ++jj) {
                            const int j = j4 + jj;
                            hp[jj] = 0u;
                            if (j < TILES && static_cast<uint32_t>(j) < nt) {
                                float x[4], y[4];                     // (input, forget) and (cell, output) of two queries
                                const uint32_t row = src + j * 8u * kPitch + ld_row;
#pragma unroll
                                for (int k = 0; k < KT; k += 2) {
                                    uint32_t b0, b1, b2, b3;
                                    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                                                 : "=r"(b0), "=r"(b1), "=r"(b2), "=r"(b3) : "r"(row + 32u * k));
                                    if (k == 0) { mma_bf16_first(x, w[0][0], b0, b1); mma_bf16_first(y, w[1][0], b0, b1); }
                                    else { mma_bf16(x, w[0][k], b0, b1); mma_bf16(y, w[1][k], b0, b1); }
                                    if (k + 1 < KT) { mma_bf16(x, w[0][k + 1 < KT ? k + 1 : k], b2, b3); mma_bf16(y, w[1][k + 1 < KT ? k + 1 : k], b2, b3); }
                                }
                                const float o0 = lstm_cell(x[0], x[2], y[0], y[2], c[j % TILES][0]);
                                const float o1 = lstm_cell(x[1], x[3], y[1], y[3], c[j % TILES][1]);
                                float t0, t1;
                                tanh_two(c[j % TILES][0], c[j % TILES][1], t0, t1);
                                hp[jj] = pack_bf16(o0 * t0, o1 * t1);
                            }
                        }
                        if (j4 + 4 <= TILES)
                            asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};"
                                         :: "r"(dst + j4 * 8u * kPitch + st_row), "r"(hp[0]), "r"(hp[1]), "r"(hp[2]), "r"(hp[3]) : "memory");
                        else                                          // (rows of lanes 16 to 31 are not used)
                            asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1,%2};"
                                         :: "r"(dst + j4 * 8u * kPitch + st_row), "r"(hp[0]), "r"(hp[1]) : "memory");
                    }
                }
                if (t + 1u < T && tid < kQ) write_token((t + 1u) & 1u, tid, t + 1u < Te ? enc[tid][t + 1u] : dec[tid][t + 1u - Te]);
                __syncthreads();
                if (t >= Te) {
                    // read-out and cross-entropy of this position, an n-tile per warp; the next step's products need the same buffer
#pragma unroll
                    for (int own = 0; own < kOwn; ++own) {
                        const uint32_t j = warp + own * kWarps;
                        if (j >= nt) break;
                        float l[4];
                        const uint32_t row = dst + j * 8u * kPitch + ld_row;
#pragma unroll
                        for (int k = 0; k < KH; k += 2) {
                            uint32_t b0, b1, b2, b3;
                            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                                         : "=r"(b0), "=r"(b1), "=r"(b2), "=r"(b3) : "r"(row + 32u * k));
                            if (k == 0) mma_bf16_first(l, out_w[lane], b0, b1);
                            else mma_bf16(l, out_w[k * 32 + lane], b0, b1);
                            mma_bf16(l, out_w[k * 32 + 32 + lane], b2, b3);
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i) {                 // query 2 t4 + i: token g and, for g < 4, token g + 8
                            const uint32_t n = j * 8u + 2u * t4 + i;
                            const int target = tgt[n][t - Te];
                            const float l0 = l[i] + out_b[g], l1 = g < kVocab - 8 ? l[2 + i] + out_b[g + 8] : -INFINITY;
                            float mx = fmaxf(l0, l1), hit = target == g ? l0 : target == g + 8 ? l1 : 0.f;
#pragma unroll
                            for (int off = 4; off < 32; off <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
                            float se = expf(l0 - mx) + (g < kVocab - 8 ? expf(l1 - mx) : 0.f);
#pragma unroll
                            for (int off = 4; off < 32; off <<= 1) {
                                se += __shfl_xor_sync(0xffffffffu, se, off);
                                hit += __shfl_xor_sync(0xffffffffu, hit, off);
                            }
                            if (g == 0 && n < nq) loss[own] += (mx + logf(se)) - hit;
                        }
                    }
                }
            }
            __syncthreads();
        }
        // a sum per n-tile, whichever block had it: the form of the launch (a shard may take another) changes no bit of the fitness
#pragma unroll
        for (int own = 0; own < kOwn; ++own) {
            const uint32_t j = warp + own * kWarps;
            loss[own] += __shfl_xor_sync(0xffffffffu, loss[own], 1);
            loss[own] += __shfl_xor_sync(0xffffffffu, loss[own], 2);
            if (lane == 0 && j < nt) a.partial[static_cast<size_t>(member) * a.n_chunks + tile0 + j] = loss[own];
        }
        at += nt;
    } while (RUNS && at < run_end);
}

// ------------------------------------------------------------------------------------------
// tensor-core version (h = 128)
// ------------------------------------------------------------------------------------------
constexpr int kTcH = 128;
constexpr int kTcQ = 128;                                  // queries per block: two halves of 64
constexpr int kTcSub = 1;                                  // warps per TMEM lane quarter and half: each takes 64 / kTcSub queries
constexpr int kTcHalfThreads = 128 * kTcSub;
constexpr int kTcEpiThreads = 2 * kTcHalfThreads;          // half 0's warps first, then half 1's
constexpr int kTcCols = 64 / kTcSub;                       // queries per epilogue thread
constexpr int kTcOutPerThread = kVocab * 64 / kTcHalfThreads;   // read-out: tokens per thread
constexpr int kTcThreads = kTcEpiThreads + 32;             // + the MMA warp
constexpr int kTcKBlocks = 18;                             // K = 128 (h) + 16 (one-hot, 1, padding) in groups of 8
constexpr uint32_t kTcALbo = 64 * 128 + 16;                // 64 row groups of 8 x 16 bytes between K groups, +16 bytes
                                                           // (bank spread of the staging stores)
constexpr uint32_t kTcBLbo = 16 * 128 + 16;                // 16 row groups, +16 bytes so that the 2-byte stores
                                                           // of a warp (4 K groups) fall in distinct banks
constexpr uint32_t kTcABytes = kTcKBlocks * kTcALbo;       // 147,744
constexpr uint32_t kTcBBytes = kTcKBlocks * kTcBLbo;       // 37,152
constexpr uint32_t kTcCellFloats = 4 * kTcH * kVocab + 4 * kTcH * kTcH + 4 * kTcH;   // one LSTM cell

struct __align__(128) S2sSmem {
    unsigned char A[kTcABytes];                            // [Wh | Wx | b | 0] as core matrices
    unsigned char Bop[kTcBBytes];                          // [h; onehot; 1; 0] of the 128 queries
    float oW[16][kVocab][8];                               // read-out weights [K group][token][k], bf16-rounded
    float ob[kVocab];
    float lg[kS2sMaxTd][kTcQ][kVocab];                     // logits of every answer position
    uint8_t enc[kTcQ][kS2sMaxTe + 1], dec[kTcQ][kS2sMaxTd + 1], tgt[kTcQ][kS2sMaxTd + 1];
    float loss_w[kTcThreads / 32];
    uint64_t full[2];                                      // the gates of a half are in TMEM
    uint64_t hready[2];                                    // a half's B operand holds the next step's input
    uint32_t tmem_slot;
    volatile int abort;
};

__device__ __forceinline__ float tanh_sfu(float x)
{
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(p));
    return p != 0;
}
// asks the L2 to fetch `bytes` (multiple of 16) starting at a 16-byte aligned address
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(__cvta_generic_to_global(p)), "r"(bytes) : "memory");
}

// One cell's weights -> A operand (all threads of the block).  The rows of the input, forget and
// output gates are halved (exact in bf16) so that their sigma(x) = 0.5 tanh(x / 2) + 0.5 needs no
// scaling of the accumulator.  TIMES_ZERO: the sum of the thread's recurrent weights times zero (else 0), which is NaN where one is infinite.
template <bool TIMES_ZERO>
__device__ __forceinline__ float s2s_stage_weights(S2sSmem& S, const float* __restrict__ cellp, uint32_t tid)
{
    uint32_t zero = 0u;
    const float* Wx = cellp;
    const float* Wh = Wx + 4 * kTcH * kVocab;
    const float* bb = Wh + 4 * kTcH * kTcH;
    // Wh: 64 groups of 8 rows x 128 k.  A warp reads a whole row with one fully coalesced 128-bit
    // load per lane (lane l gets k = 4l .. 4l+3), 8 rows per group, two groups at a time.  A
    // 16-byte row of a core matrix (8 k) is the data of an even/odd lane pair, so the pair swaps
    // halves: the even lane ends with rows 0-3 of its K group, the odd lane with rows 4-7, and each
    // stores them as 128-bit words (the K-group pitch is padded by 16 bytes so that the four K
    // groups of a quarter-warp fall in distinct banks).
    const uint32_t warp = tid >> 5, lane = tid & 31u;
    const bool odd = lane & 1u;
    constexpr uint32_t kWarps = kTcThreads / 32, G = 2;
#pragma unroll 1
    for (uint32_t mg0 = warp * G; mg0 < 64u; mg0 += kWarps * G) {
        float4 v[G][8];
#pragma unroll
        for (uint32_t g = 0; g < G; ++g)
#pragma unroll
            for (uint32_t r = 0; r < 8u; ++r) {
                const uint32_t mg = min(mg0 + g, 63u);
                v[g][r] = __ldg(reinterpret_cast<const float4*>(Wh + (mg * 8u + r) * kTcH) + lane);
            }
#pragma unroll
        for (uint32_t g = 0; g < G; ++g) {
            const uint32_t mg = mg0 + g;
            if (mg < 64u) {
                const float sc = ((mg >> 4) == 2u) ? 1.0f : 0.5f;       // 16 row groups per gate
                uint32_t w0[8], w1[8];
#pragma unroll
                for (uint32_t r = 0; r < 8u; ++r) {
                    w0[r] = pack_bf16(sc * v[g][r].x, sc * v[g][r].y);
                    w1[r] = pack_bf16(sc * v[g][r].z, sc * v[g][r].w);
                    if constexpr (TIMES_ZERO)
                        asm("fma.rn.bf16x2 %0, %1, %3, %0;\n\tfma.rn.bf16x2 %0, %2, %3, %0;" : "+r"(zero) : "r"(w0[r]), "r"(w1[r]), "r"(0u));
                }
                unsigned char* dst = S.A + (lane >> 1) * kTcALbo + mg * 128u + (odd ? 64u : 0u);
#pragma unroll
                for (uint32_t i = 0; i < 4u; ++i) {
                    const uint32_t got0 = __shfl_xor_sync(0xffffffffu, odd ? w0[i] : w0[i + 4], 1);
                    const uint32_t got1 = __shfl_xor_sync(0xffffffffu, odd ? w1[i] : w1[i + 4], 1);
                    const uint32_t keep0 = odd ? w0[i + 4] : w0[i], keep1 = odd ? w1[i + 4] : w1[i];
                    // the even lane's words are k 0-3 of the K group, the odd lane's k 4-7
                    *reinterpret_cast<uint4*>(dst + i * 16u) =
                        odd ? make_uint4(got0, got1, keep0, keep1) : make_uint4(keep0, keep1, got0, got1);
                }
            }
        }
    }
    // K groups 16, 17: Wx[m][0..7] | Wx[m][8..11], b[m], 0, 0, 0
    for (uint32_t m = tid; m < 512u; m += kTcThreads) {
        const float4* wx = reinterpret_cast<const float4*>(Wx + m * kVocab);        // 48-byte rows
        const float4 w0 = __ldg(wx), w1 = __ldg(wx + 1), w2 = __ldg(wx + 2);
        const float sc = ((m >> 7) == 2u) ? 1.0f : 0.5f;
        const float bias = sc * __ldg(bb + m);
        *reinterpret_cast<uint4*>(S.A + 16u * kTcALbo + (m >> 3) * 128u + (m & 7u) * 16u) =
            make_uint4(pack_bf16(sc * w0.x, sc * w0.y), pack_bf16(sc * w0.z, sc * w0.w),
                       pack_bf16(sc * w1.x, sc * w1.y), pack_bf16(sc * w1.z, sc * w1.w));
        *reinterpret_cast<uint4*>(S.A + 17u * kTcALbo + (m >> 3) * 128u + (m & 7u) * 16u) =
            make_uint4(pack_bf16(sc * w2.x, sc * w2.y), pack_bf16(sc * w2.z, sc * w2.w), pack_bf16(bias, 0.f), 0u);
    }
    return __uint_as_float(zero << 16) + __uint_as_float(zero & 0xFFFF0000u);
}

// one-hot (+ constant 1) rows of query n for the coming step
__device__ __forceinline__ void s2s_write_onehot(S2sSmem& S, uint32_t n, uint32_t tok)
{
    uint32_t w[8];
    const uint32_t one = (tok & 1u) ? 0x3F800000u : 0x00003F80u;  // bf16 1.0 in the upper / lower half
#pragma unroll
    for (uint32_t i = 0; i < 8u; ++i) w[i] = (i == (tok >> 1)) ? one : 0u;
    w[6] |= 0x00003F80u;                                          // k = 12: the constant input of the bias
    *reinterpret_cast<uint4*>(S.Bop + 16u * kTcBLbo + n * 16u) = make_uint4(w[0], w[1], w[2], w[3]);
    *reinterpret_cast<uint4*>(S.Bop + 17u * kTcBLbo + n * 16u) = make_uint4(w[4], w[5], w[6], w[7]);
}

// barrier over the four epilogue warps of one half
__device__ __forceinline__ void half_barrier(uint32_t half)
{
    if (half) asm volatile("bar.sync 2, %0;" :: "n"(kTcHalfThreads) : "memory");
    else      asm volatile("bar.sync 1, %0;" :: "n"(kTcHalfThreads) : "memory");
}

// kPadded: items are worked off as 128 queries whatever they hold, and the loops do not ask (128 queries, 1,036 members, 3 digits: 456 us; kPartial
// takes 465.  148 members: 66 us, kPartial with 120 queries 69, with 112 64).  kFull: they hold 128, and nothing asks (454 us).
enum class Items { kPartial, kPadded, kFull };
template <Items KIND>
__global__ void __launch_bounds__(kTcThreads, 1)
k_s2s_tc(const S2sArgs a, DeviceStatus* status)
{
    constexpr bool FULL = KIND != Items::kPartial;
    extern __shared__ __align__(128) unsigned char s2s_smem_raw[];
    S2sSmem& S = *reinterpret_cast<S2sSmem*>(s2s_smem_raw);
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31u;
    const uint32_t Te = 2 * a.nd + 1, Td = a.nd + 1, T = Te + Td;
    const uint32_t n_items = a.P * a.n_chunks;
    const PhiloxKey key = philox_key(a.k0, a.k1);

    if (tid == 0) {
        mbar_init(smem_u32(&S.full[0]), 1); mbar_init(smem_u32(&S.full[1]), 1);
        mbar_init(smem_u32(&S.hready[0]), kTcHalfThreads / 32); mbar_init(smem_u32(&S.hready[1]), kTcHalfThreads / 32);
        S.abort = 0;
        mbar_init_fence();
    }
    __syncwarp();
    if (warp == 0) tmem_alloc(smem_u32(&S.tmem_slot), 512);
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_slot;

    uint32_t n_wait = 0u, n_wait1 = 0u;        // completed waits: full[half] (epilogue) / hready[0], hready[1] (MMA warp)
    const bool is_mma = warp >= kTcEpiThreads / 32;
    const uint32_t half = (tid / kTcHalfThreads) & 1u;          // epilogue warps: which 64 queries
    const uint32_t sub = (tid % kTcHalfThreads) >> 7;           // ... and which kTcCols of them
    const uint32_t r = tid & 127u;             // epilogue thread: hidden unit = TMEM lane
    uint32_t staged_chunk = 0xFFFFFFFFu;

    for (uint32_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        const uint32_t member = item / a.n_chunks, chunk = item % a.n_chunks;
        const uint32_t q0 = chunk * (FULL ? kTcQ : a.per_chunk);
        const uint32_t nq = FULL ? kTcQ : min(a.per_chunk, a.B - q0);
        // The halves share the queries evenly, to eights, and what holds none is left out: a half, eight queries of it, a warp's read-out.
        // Every item was worked off as 128 queries before.  1,036 members, 3 digits: 40 queries 455 -> 330 us, 64 455 -> 347, 100 456 -> 450,
        // 130 (two items of 65 instead of 128 and 2) 849 -> 677, 300 1,272 -> 1,216.
        const uint32_t nq0 = FULL ? 64u : min(nq, (nq + 15u) / 16u * 8u), n_halves = FULL || nq > nq0 ? 2u : 1u, nq_half = half ? nq - nq0 : nq0;
        const float* p = a.theta + static_cast<size_t>(member) * a.ldD;

        // ---- per-item setup: queries, zero state, read-out weights, encoder weights ------------
        if (chunk != staged_chunk) {
            if (tid < kTcQ) {                                     // the query of row `tid`; rows that hold none repeat the last one
                uint32_t q = tid;
                if (KIND == Items::kPadded) q = min(q, a.B - 1u - q0);
                if (KIND == Items::kPartial) q = min(q < 64u ? q : nq0 + q - 64u, nq - 1u);
                s2s_query(key, a.status->generation, q0 + q, a.nd, S.enc[tid], S.dec[tid], S.tgt[tid]);
            }
            staged_chunk = chunk;
        }
        if (is_mma) {                                            // the decoder's weights will be wanted next
            const char* next = reinterpret_cast<const char*>(p + kTcCellFloats);
            constexpr uint32_t piece = kTcCellFloats * 4u / 32u;       // 9,024 bytes per lane
            prefetch_l2(next + lane * piece, piece);
        }
        if constexpr (FULL)
            for (uint32_t i = tid; i < 16u * kTcBLbo / 16u; i += kTcThreads) reinterpret_cast<uint4*>(S.Bop)[i] = make_uint4(0u, 0u, 0u, 0u);
        for (uint32_t i = tid; i < kVocab * 16u; i += kTcThreads) {       // (token, K group) -> 8 weights
            const uint32_t o = i >> 4, kb = i & 15u;
            const float4* src = reinterpret_cast<const float4*>(p + 2u * kTcCellFloats + o * kTcH + kb * 8u);
            const float4 w0 = __ldg(src), w1 = __ldg(src + 1);
            float* dst = S.oW[kb][o];
            dst[0] = bf16_round(w0.x); dst[1] = bf16_round(w0.y); dst[2] = bf16_round(w0.z); dst[3] = bf16_round(w0.w);
            dst[4] = bf16_round(w1.x); dst[5] = bf16_round(w1.y); dst[6] = bf16_round(w1.z); dst[7] = bf16_round(w1.w);
        }
        if (tid < kVocab) S.ob[tid] = p[2u * kTcCellFloats + kVocab * kTcH + tid];
        // kPartial: the first step leaves the zero state out, but an infinite weight times zero is NaN, and a step later so is every unit
        float loss = s2s_stage_weights<!FULL>(S, p, tid);
        __syncthreads();                                        // tokens are there
        if (tid < kTcQ) s2s_write_onehot(S, tid, S.enc[tid][0]);
        fence_async_smem();
        __syncthreads();

        float c[kTcCols];
#pragma unroll
        for (int i = 0; i < kTcCols; ++i) c[i] = 0.f;

        for (uint32_t phase = 0; phase < 2u; ++phase) {
            const uint32_t t0 = phase ? Te : 0u, t1 = phase ? T : Te;
            if (phase) {
                // every MMA of the encoder has been waited for by an epilogue warp: A may be replaced
                __syncthreads();
                s2s_stage_weights<false>(S, p + kTcCellFloats, tid);
                fence_async_smem();
                __syncthreads();
                if (is_mma && item + gridDim.x < n_items) {     // the next item's encoder cell
                    const uint32_t nm = (item + gridDim.x) / a.n_chunks;
                    const char* next = reinterpret_cast<const char*>(a.theta + static_cast<size_t>(nm) * a.ldD);
                    constexpr uint32_t piece = kTcCellFloats * 4u / 32u;
                    prefetch_l2(next + lane * piece, piece);
                }
            }
            if (is_mma) {
                // ================= MMA warp (the whole warp walks the loop, one lane issues) ===========
                // The halves alternate, so that one half's MMAs run while the other half's gates are
                // being applied.
                constexpr uint32_t idesc = umma_idesc_bf16(128, 64);
                const uint32_t a_base = smem_u32(S.A), b_base = smem_u32(S.Bop);
                for (uint32_t t = t0; t < t1; ++t) {
#pragma unroll
                    for (uint32_t x = 0; x < 2u; ++x) {
                        if (x >= n_halves) break;
                        if (t > 0) {                             // step 0 reads the tokens that the setup wrote
                            uint32_t& n = x ? n_wait1 : n_wait;
                            wait_or_abort(&S.abort, &S.hready[x], n & 1u, status);
                            ++n;
                        }
                        tc_fence_after();
                        if (elect_one()) {
                            auto issue = [&](uint32_t g, uint32_t kk, uint32_t accumulate) {
                                const uint64_t ad = umma_smem_desc(a_base + 2u * kk * kTcALbo + g * 16u * 128u, kTcALbo, 128u);
                                const uint64_t bd = umma_smem_desc(b_base + 2u * kk * kTcBLbo + x * 8u * 128u, kTcBLbo, 128u);
                                umma_bf16(tmem + x * 256u + g * 64u, ad, bd, idesc, accumulate);
                            };
                            if (!FULL && t == 0u) {              // the start state is zero: token and bias only (the last K-step)
#pragma unroll
                                for (uint32_t g = 0; g < 4u; ++g) issue(g, kTcKBlocks / 2 - 1, 0u);
                            } else {
#pragma unroll
                                for (uint32_t g = 0; g < 4u; ++g)
#pragma unroll
                                    for (uint32_t kk = 0; kk < kTcKBlocks / 2; ++kk) issue(g, kk, kk);
                            }
                            umma_commit(smem_u32(&S.full[x]));
                        }
                        __syncwarp();
                    }
                }
            } else if (half < n_halves) {
                // ================= epilogue warps ======================================================
                const uint32_t tq = tmem + (static_cast<uint32_t>((warp & 3u) * 32u) << 16) + half * 256u + sub * kTcCols;
                for (uint32_t t = t0; t < t1; ++t) {
                    wait_or_abort(&S.abort, &S.full[half], n_wait & 1u, status);
                    ++n_wait;
                    tc_fence_after();
                    // chunks of 8 queries; the loads of the next chunk are in flight while this one
                    // is worked on (two register sets)
                    uint32_t g0[2][8], g1[2][8], g2[2][8], g3[2][8];
                    tmem_ld8_issue(tq + 0u * 64u, g0[0]); tmem_ld8_issue(tq + 1u * 64u, g1[0]);
                    tmem_ld8_issue(tq + 2u * 64u, g2[0]); tmem_ld8_issue(tq + 3u * 64u, g3[0]);
                    tmem_ld8x4_fence(g0[0], g1[0], g2[0], g3[0]);
#pragma unroll
                    for (uint32_t ch = 0; ch < kTcCols / 8u; ++ch) {
                        const uint32_t cur = ch & 1u, nxt = cur ^ 1u;
                        if (ch + 1u < kTcCols / 8u) {
                            tmem_ld8_issue(tq + 0u * 64u + (ch + 1u) * 8u, g0[nxt]);
                            tmem_ld8_issue(tq + 1u * 64u + (ch + 1u) * 8u, g1[nxt]);
                            tmem_ld8_issue(tq + 2u * 64u + (ch + 1u) * 8u, g2[nxt]);
                            tmem_ld8_issue(tq + 3u * 64u + (ch + 1u) * 8u, g3[nxt]);
                        }
                        // hidden unit r of query n sits at K group r/8, row n, element r%8
                        unsigned char* dst = S.Bop + (r >> 3) * kTcBLbo + (half * 64u + sub * kTcCols + ch * 8u) * 16u + (r & 7u) * 2u;
#pragma unroll
                        for (int j = 0; j < 8; j += 2) {
                            // the accumulators of the i, f, o gates already hold x / 2
                            float2 hv;
                            {
                                const float ig = fmaf(0.5f, tanh_sfu(__uint_as_float(g0[cur][j])), 0.5f);
                                const float fg = fmaf(0.5f, tanh_sfu(__uint_as_float(g1[cur][j])), 0.5f);
                                const float cg = tanh_sfu(__uint_as_float(g2[cur][j]));
                                const float og = fmaf(0.5f, tanh_sfu(__uint_as_float(g3[cur][j])), 0.5f);
                                float& c0 = c[ch * 8 + j];
                                c0 = fmaf(fg, c0, ig * cg);
                                hv.x = og * tanh_sfu(c0);
                            }
                            {
                                const float ig = fmaf(0.5f, tanh_sfu(__uint_as_float(g0[cur][j + 1])), 0.5f);
                                const float fg = fmaf(0.5f, tanh_sfu(__uint_as_float(g1[cur][j + 1])), 0.5f);
                                const float cg = tanh_sfu(__uint_as_float(g2[cur][j + 1]));
                                const float og = fmaf(0.5f, tanh_sfu(__uint_as_float(g3[cur][j + 1])), 0.5f);
                                float& c1 = c[ch * 8 + j + 1];
                                c1 = fmaf(fg, c1, ig * cg);
                                hv.y = og * tanh_sfu(c1);
                            }
                            const uint32_t hb = pack_bf16(hv.x, hv.y);
                            *reinterpret_cast<uint16_t*>(dst + j * 16) = static_cast<uint16_t>(hb & 0xFFFFu);
                            *reinterpret_cast<uint16_t*>(dst + j * 16 + 16) = static_cast<uint16_t>(hb >> 16);
                        }
                        if (ch + 1u < kTcCols / 8u) tmem_ld8x4_fence(g0[nxt], g1[nxt], g2[nxt], g3[nxt]);
                        if (!FULL && sub * kTcCols + (ch + 1u) * 8u >= nq_half) break;
                    }
                    // the coming step's token (none after the last step)
                    if (t + 1u < T && sub == 0u && r < 64u) {
                        const uint32_t n = half * 64u + r;
                        s2s_write_onehot(S, n, (t + 1u < Te) ? S.enc[n][t + 1u] : S.dec[n][t + 1u - Te]);
                    }
                    fence_async_smem();
                    tc_fence_before();
                    if (t >= Te) {
                        // read-out on the CUDA cores from the state just written (all warps of the
                        // half must have written it), while the tensor cores work on the next step
                        half_barrier(half);
                        if (t + 1u < T && lane == 0) mbar_arrive(smem_u32(&S.hready[half]));
                        const uint32_t s = tid & 63u, o0 = ((tid % kTcHalfThreads) >> 6) * kTcOutPerThread;
                        const uint32_t kb_end = FULL || (s & 32u) < nq_half ? 16u : 0u;             // (logits of no query are not looked at)
                        float2 acc[kTcOutPerThread];
#pragma unroll
                        for (int o = 0; o < kTcOutPerThread; ++o) acc[o] = make_float2(0.f, 0.f);
                        const unsigned char* hrow = S.Bop + (half * 64u + s) * 16u;
#pragma unroll 4
                        for (uint32_t kb = 0; kb < kb_end; ++kb) {
                            const uint4 hv = *reinterpret_cast<const uint4*>(hrow + kb * kTcBLbo);
                            const uint32_t hw[4] = { hv.x, hv.y, hv.z, hv.w };
                            float2 x[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                x[i] = make_float2(__uint_as_float(hw[i] << 16), __uint_as_float(hw[i] & 0xFFFF0000u));
#pragma unroll
                            for (int o = 0; o < kTcOutPerThread; ++o) {
                                const float4 w0 = *reinterpret_cast<const float4*>(&S.oW[kb][o0 + o][0]);
                                const float4 w1 = *reinterpret_cast<const float4*>(&S.oW[kb][o0 + o][4]);
                                ffma2(acc[o], make_float2(w0.x, w0.y), x[0]);
                                ffma2(acc[o], make_float2(w0.z, w0.w), x[1]);
                                ffma2(acc[o], make_float2(w1.x, w1.y), x[2]);
                                ffma2(acc[o], make_float2(w1.z, w1.w), x[3]);
                            }
                        }
#pragma unroll
                        for (int o = 0; o < kTcOutPerThread; ++o) S.lg[t - Te][half * 64u + s][o0 + o] = (acc[o].x + acc[o].y) + S.ob[o0 + o];
                        // the next epilogue overwrites the state: everyone must be done reading it
                        half_barrier(half);
                    } else {
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&S.hready[half]));
                    }
                }
            }
        }
        // ---- the item's loss: cross-entropy of every (position, query), summed in a fixed order ----
        __syncthreads();
        for (uint32_t idx = tid; idx < Td * kTcQ; idx += kTcThreads) {
            const uint32_t pos = idx / kTcQ, q = idx % kTcQ;
            const uint32_t row = q < nq0 ? q : 64u + q - nq0;
            if (q < nq && (KIND != Items::kPadded || q0 + q < a.B)) loss += token_loss(S.lg[pos][row], S.tgt[row][pos]);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
        if (lane == 0) S.loss_w[warp] = loss;
        __syncthreads();
        if (tid == 0) {
            float total = 0.f;
            for (int w = 0; w < kTcThreads / 32; ++w) total += S.loss_w[w];
            a.partial[static_cast<size_t>(member) * a.n_chunks + chunk] = total;
        }
        __syncthreads();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------
uint32_t s2s_param_count(uint32_t h)
{
    return 2u * (4u * h * kVocab + 4u * h * h + 4u * h) + kVocab * h + kVocab;
}

bool s2s_supported(uint32_t h, uint32_t nd, uint32_t B)
{
    return h >= 32 && h <= 128 && h % 32 == 0 && nd >= 1 && nd <= kS2sMaxDigits && B >= 1;
}

static cudaError_t launch_s2s_mma(cudaStream_t st, const S2sArgs& a, const S2sSplit& split)
{
    if (split.chunk == 0u)
        return launch_dependent(a.h == 64u ? k_s2s_mma<64, kS2sRunTiles64, true> : k_s2s_mma<96, kS2sRunTiles96, true>, dim3(split.places),
                                dim3(4u * a.h), 0, st, a, 0u);
    return launch_dependent(a.h == 32u ? k_s2s_mma<32, 8, false> : a.h == 64u ? k_s2s_mma<64, 8, false> : k_s2s_mma<96, 8, false>,
                            dim3(a.P, split.chunks), dim3(4u * a.h), 0, st, a, split.chunk);
}

size_t s2s_scratch_bytes(uint32_t P, uint32_t B)
{
    return static_cast<size_t>(P) * ((B + 7u) / 8u) * sizeof(float);          // the finest split any kernel uses
}

int launch_rollout_s2s(cudaStream_t st, const float* theta, uint32_t ldD, uint32_t P, uint32_t h, uint32_t nd,
                       uint32_t B, uint32_t k0, uint32_t k1, uint32_t kernel_choice, const S2sSplit& split,
                       void* scratch, float* fitness, float* logits, DeviceStatus* status)
{
    const bool want_tc = kernel_choice != EVO_ROLLOUT_GENERIC;
    if (want_tc && (h != kTcH || logits)) {
        if (kernel_choice == EVO_ROLLOUT_TILED) return -2;       // asked for explicitly, not available
    }
    const bool tc = want_tc && h == kTcH && !logits, mma = want_tc && h != kTcH && !logits;
    S2sArgs a;
    a.theta = theta; a.ldD = ldD; a.P = P; a.h = h; a.nd = nd; a.B = B;
    a.k0 = k0; a.k1 = k1; a.status = status;
    a.partial = static_cast<float*>(scratch);
    a.n_chunks = mma ? (B + 7u) / 8u : (B + kSimpleQ - 1u) / kSimpleQ;
    a.per_chunk = kSimpleQ;
    a.logits = logits;
    if (tc) {
        static int sm_count = 0;
        if (sm_count == 0) {
            int dev = 0;
            if (cudaGetDevice(&dev) != cudaSuccess) return -1;
            if (cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
        }
        a.n_chunks = split.chunks;
        a.per_chunk = split.chunk;
        auto kernel = split.chunk != kTcQ ? k_s2s_tc<Items::kPartial> : B % kTcQ == 0u ? k_s2s_tc<Items::kFull> : k_s2s_tc<Items::kPadded>;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(sizeof(S2sSmem))) != cudaSuccess) return -1;
        const uint32_t items = P * a.n_chunks;
        const uint32_t grid = items < static_cast<uint32_t>(sm_count) ? items : static_cast<uint32_t>(sm_count);
        kernel<<<grid, kTcThreads, sizeof(S2sSmem), st>>>(a, status);
    } else if (mma) {
        if (launch_s2s_mma(st, a, split) != cudaSuccess) return -1;
    } else {
        dim3 grid(P, a.n_chunks);
        k_s2s_simple<<<grid, 128, 0, st>>>(a);
    }
    if (cudaGetLastError() != cudaSuccess) return -1;
    const float inv = 1.0f / (static_cast<float>(B) * static_cast<float>(nd + 1));
    const bool four = mma && a.n_chunks > 4u;
    const uint32_t members = four ? 64u : 256u;                   // per block of 256 threads
    if (launch_dependent(four ? k_s2s_finalize<4> : k_s2s_finalize<1>, dim3((P + members - 1u) / members), dim3(256), 0, st, a.partial, P,
                         a.n_chunks, inv, fitness) != cudaSuccess)
        return -1;
    return 2;
}

}  // namespace evo
