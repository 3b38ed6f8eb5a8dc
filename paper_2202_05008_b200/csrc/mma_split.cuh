// Warp-level tensor-core products with fp32 accuracy for the control roll-outs.
//
// A weight is two fp16 numbers, w = hi + lo / 2048 with hi = fp16(w), lo = fp16(2048 (w - hi)): 22 mantissa bits
// (the factor keeps the small parts out of the subnormal range); an activation is hi + lo.  Products of fp16
// numbers are exact and sums are kept in fp32.  The products run as mma.sync m16n8k16: the 16x16 weight
// tile is an operand in REGISTERS (or one 128-bit shared-memory load per lane), which is what these
// roll-outs need: a member has its own weights and only 4 or 8 columns of activations, so an MMA is paced
// by its weight operand.  tcgen05 fetches 4 KB of weights from tensor or shared memory per 128x16 tile and
// step (21-32 clocks for 8 columns) and its result is read 340 clocks later at the earliest; mma.sync takes
// the same 128x16x8 product from registers in 16 clocks of the four sub-cores (8.1 clocks per m16n8k16 and
// sub-core, measured) and the result is there after 22 (28 for another pipe).
//
// tanh.  A layer's weights and biases are taken times f = 2 log2(e) when they are loaded, so its sums are p = f x and
//     tanh x = (e - 1) / (e + 1),  e = 2^p:
// e - 1 is exact where e is near 1, so a small tanh keeps its relative accuracy as far as the exponential has it.  It
// travels times 2^13: the low part of an activation is then in fp16's normal range down to 2^-16 of the largest.  (Carrying
// r = 1 / (1 + 2^p) instead, with the layers rewritten for it, saves a few instructions, but r is near 1/2 for small
// activations: the products then cancel, and the states were 2 to 5 times as far from the 64-bit ones.)
//
// Activations of a layer lie in shared memory as the B operand, [column][unit] fp16, a column = one episode and
// part.  Two packings of the columns of an n-tile (8 columns) are used:
//   pairs  (4 episodes): column 2e = hi, 2e + 1 = -lo of episode e: a lane of the accumulator then holds both
//          products of its episode side by side; all four cross terms, two MMAs per tile
//   planes (8 episodes): one n-tile of the hi parts and one of the -lo parts: hi*hi, hi*lo and lo*hi, three
//          MMAs per tile for twice the episodes (lo*lo is below 2^-22 of the product)
// A lane's values of 16 units, v[]: pairs: units g, g + 8 of episode t; planes: unit g of episodes 2t and 2t + 1,
// then unit g + 8 of the two (g = lane / 4, t = lane % 4).
#pragma once
#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "internal.h"

namespace evo {
namespace ms {

// c[0], c[1]: row g, columns 2t, 2t + 1; c[2], c[3]: row g + 8 (g = lane / 4, t = lane % 4)
__device__ __forceinline__ void mma_k16(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// the same from zero sums (no register has to be cleared for it)
__device__ __forceinline__ void mma_k16_first(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1), "f"(0.f));
}

// 8x8 fp16 matrices from shared memory, row addresses from lanes 0-7, 8-15, ...
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
// accumulator fragments (rows = units) to shared memory as [column][unit]
__device__ __forceinline__ void stsm_x2_t(uint32_t addr, uint32_t r0, uint32_t r1)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1,%2};" :: "r"(addr), "r"(r0), "r"(r1) : "memory");
}

__device__ __forceinline__ void stsm_x4_t(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};"
                 :: "r"(addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3) : "memory");
}
// an 8x8 fp16 matrix held by a warp, transposed: accumulator layout -> B operand layout
__device__ __forceinline__ uint32_t transpose8(uint32_t x)
{
    uint32_t r;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(x));
    return r;
}

constexpr float kF = 2.885390082f;                           // 2 log2(e)
// What a factor f lacks: the fp32 f is short by 1.3e-8, and the tensor core cuts its sums off, which leaves a result 3e-8 short
// on average.  (Both are systematic, and a roll-out adds them up: without, the states of 28-64-64-64-8 shrink by 4e-8 per step
// and the fitness is off by 5e-7; with, by less than 1e-8 per step, and by 2e-7.)
constexpr float kRest = 1.3e-8f + 3.0e-8f;
constexpr float kAct = 8192.0f, kActInv = 1.0f / 8192.0f;    // scale of the activations (a start state of 5.8, the largest normal, fits fp16)
constexpr float kLo = 2048.0f, kLoInv = 1.0f / 2048.0f;      // scale of the weights' low parts

// a and b, a in the low half: hi parts in one word, the negated low parts in the other
__device__ __forceinline__ void split_two(float a, float b, uint32_t& hi, uint32_t& neg_lo)
{
    float x, y;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(b), "f"(a));
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\tsub.rn.f32.f16 %0, l, %3;\n\tsub.rn.f32.f16 %1, h, %4;\n\t}"
        : "=f"(x), "=f"(y) : "r"(hi), "f"(a), "f"(b));
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(neg_lo) : "f"(y), "f"(x));
}

// Weights beyond the fp16 range: a unit that has any keeps its weights times 2^-n, which brings f w of the largest below it, and
// its sums are multiplied back.  What the other weights lose is then below 2^-22 of the largest, as it is in the unit's
// sum; other units, and the biases, are not touched.  The kernels look at a member's largest weight first: nearly always there is
// nothing to scale, and a step then does without the units' factors.  Infinities count, and are taken, as the largest finite
// number (the tanh behind them saturates); NaN stays NaN.
__device__ __forceinline__ uint32_t magnitude(float w)                    // bit pattern
{
    const uint32_t m = __float_as_uint(w) & 0x7FFFFFFFu;
    return m > 0x7F800000u ? 0u : min(m, 0x7F7FFFFFu);
}
__device__ __forceinline__ int scale_exponent(uint32_t peak)              // n: 0 for weights below 8,192
{
    return max(static_cast<int>(peak >> 23) - (127 + 12), 0);
}
__device__ __forceinline__ float scale_down(int n) { return __uint_as_float(static_cast<uint32_t>(127 - n) << 23); }
__device__ __forceinline__ float scale_up(int n) { return __uint_as_float(static_cast<uint32_t>(127 + n) << 23) * kActInv; }      // and the activations' scale
__device__ __forceinline__ float finite(float w)
{
    asm("max.NaN.f32 %0, %0, %1;\n\tmin.NaN.f32 %0, %0, %2;" : "+f"(w) : "f"(-3.402823466e38f), "f"(3.402823466e38f));
    return w;
}
// f x; a finite x stays finite
__device__ __forceinline__ float times_f(float x) { return isinf(x) ? x : finite(kF * x); }
// k wa and k wb, a in the low half, with kRest and the roundings of the products in the low parts
__device__ __forceinline__ void split_weights(float wa, float wb, float k, uint32_t& hi, uint32_t& lo)
{
    const float a = wa * k, b = wb * k, k2 = k * kRest;
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    const float ra = fmaf(wa, k2, fmaf(wa, k, -a)), rb = fmaf(wb, k2, fmaf(wb, k, -b));
    const __half2 l = __floats2half2_rn(((a - f.x) + ra) * kLo, ((b - f.y) + rb) * kLo);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

// This lane's part of a 16x16 tile at (row0, col0) of a row-major [no][ni] matrix: w[i] = columns 2t and 2t + 1 (i < 2) or
// 2t + 8 and 2t + 9 of row g (i even) or g + 8; zeros outside the matrix.  `pairs`: ni is even and W 8-byte aligned.
__device__ __forceinline__ void read_tile(const float* W, int ni, int no, int row0, int col0, int lane, bool pairs, float2 (&w)[4])
{
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int row = row0 + g + 8 * (i & 1), col = col0 + 2 * t + 8 * (i >> 1);
        const float* p = W + static_cast<size_t>(row) * ni + col;
        w[i] = make_float2(0.f, 0.f);
        if (pairs) {
            if (row < no && col < ni) w[i] = *reinterpret_cast<const float2*>(p);
        } else {
            if (row < no && col < ni) w[i].x = p[0];
            if (row < no && col + 1 < ni) w[i].y = p[1];
        }
    }
}
// Exponents of rows g and g + 8 of the `kt` tiles from row0 on, of the matrix times `times`.
__device__ __forceinline__ void row_exponents(const float* W, int ni, int no, int row0, int kt, int lane, int& n0, int& n1, float times = 1.0f)
{
    uint32_t m0 = 0, m1 = 0;
    for (int k = 0; k < kt; ++k) {
        float2 w[4];
        read_tile(W, ni, no, row0, 16 * k, lane, false, w);
        m0 = max(max(m0, max(magnitude(times * w[0].x), magnitude(times * w[0].y))), max(magnitude(times * w[2].x), magnitude(times * w[2].y)));
        m1 = max(max(m1, max(magnitude(times * w[1].x), magnitude(times * w[1].y))), max(magnitude(times * w[3].x), magnitude(times * w[3].y)));
    }
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
        m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, off));
        m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, off));
    }
    n0 = scale_exponent(m0);
    n1 = scale_exponent(m1);
}
// A tile times f (and `times`) as the A operand; n0, n1: the exponents of rows g and g + 8.
__device__ __forceinline__ void load_tile(const float* W, int ni, int no, int row0, int col0, int lane, int n0, int n1,
                                          uint4& hi, uint4& lo, bool pairs = false, float times = 1.0f)
{
    float2 w[4];
    read_tile(W, ni, no, row0, col0, lane, pairs, w);
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        split_weights(finite(times * w[i].x), finite(times * w[i].y), kF * scale_down(i & 1 ? n1 : n0), h[i], l[i]);
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// The tanh-linear task's dynamics x' = tanh(A x + s B a) as operand tiles: tile i of six, three (two of A, one of B) for each 16 rows,
// and the exponents of its rows where anything is scaled.  Entries of B stay below 2.1 (normals over sqrt(8)), so s does
// not have to be looked at more closely below 2,048.
__device__ __forceinline__ bool scales_dynamics(float action_scale) { return !(fabsf(action_scale) < 2048.0f); }
__device__ __forceinline__ void load_dynamics(const float* task_const, float action_scale, int i, int lane, bool scaled, int& n0, int& n1,
                                              uint4& hi, uint4& lo)
{
    const float* A = task_const;
    const float* B = task_const + kTlNx * kTlNx;
    const int row0 = 16 * (i / 3);
    n0 = n1 = 0;
    if (scaled) {
        int b0, b1;
        row_exponents(A, kTlNx, kTlNx, row0, 2, lane, n0, n1);
        row_exponents(B, kTlNa, kTlNx, row0, 1, lane, b0, b1, action_scale);
        n0 = max(n0, b0); n1 = max(n1, b1);
    }
    if (i % 3 < 2) load_tile(A, kTlNx, kTlNx, row0, 16 * (i % 3), lane, n0, n1, hi, lo);
    else load_tile(B, kTlNa, kTlNx, row0, 0, lane, n0, n1, hi, lo, false, action_scale);
}

__device__ __forceinline__ float ex2_fast(float p)
{
    float e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(p));
    return e;
}
__device__ __forceinline__ float rcp_fast(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// kAct tanh(p / f).  p is held below 40, where the tanh is 1 to fp32 long since, so that e stays finite.
__device__ __forceinline__ float hold(float p)
{
    asm("min.NaN.f32 %0, %0, 0f42200000;" : "+f"(p));
    return p;
}
__device__ __forceinline__ float tanh_one(float p)
{
    const float e = ex2_fast(hold(p));
    return fmaf(kAct, e, -kAct) * rcp_fast(e + 1.0f);
}
// Two of them with one reciprocal, 1/a = b / (a b): the special-function unit takes 8 clocks per warp for an exponential and 16
// for a reciprocal.  Two more multiplications, each with its rounding.
__device__ __forceinline__ void tanh_two(float& p, float& q)
{
    const float e = ex2_fast(hold(p)), d = ex2_fast(hold(q));
    const float a = e + 1.0f, b = d + 1.0f;
    const float r = rcp_fast(a * b);
    p = fmaf(kAct, e, -kAct) * b * r;
    q = fmaf(kAct, d, -kAct) * a * r;
}
// With the Taylor polynomial to x^9 below |x| = 0.3, where what it leaves out is below 6e-8 of x.  For k_rollout_mlp_deep and
// k_rollout_mlp_mma, which also take policies with layers so narrow that their sums do not hide the exponential's error near 1.  State error
// against that of tanhf on the fp32 pipe, after 1 / 20 / 200 steps: 28-20-8 without it 1.05 / 1.05 / 1.18, with it 0.95 / 0.82 / 0.92;
// 28-64-10-10-8 without 1.04 / 1.12 / 1.16; 28-64-64-64-8 without 0.91 / 0.84 / 0.86.  In k_rollout_mlp_deep after 5 / 20 / 60 steps: 28-40-8
// without 0.95 / 1.09 / 1.09, 28-48-8 0.96 / 1.01 / 1.01, 28-56-8 0.93 / 0.96 / 0.98, 28-40-40-40-8 0.94 / 1.05 / 1.03, 28-56-56-56-8 0.89 / 0.94 / 0.93,
// all with it 0.74 to 0.82.  It costs there 4 to 12 % (28-64-64-64-8, 512 members, 200 steps 222 -> 244 us; 128 members 143 -> 148), so a
// policy has it whose narrowest hidden layer is below 49 units.
__device__ __forceinline__ float tanh_fine(float p)
{
    constexpr double f = 2.885390081777927, g = 1.0 / (f * f);                // z = p^2 = x^2 / g
    const float z = p * p, k = p * static_cast<float>(8192.0 / f);
    float c = fmaf(z, static_cast<float>(62.0 / 2835.0 * g * g * g * g), static_cast<float>(-17.0 / 315.0 * g * g * g));
    c = fmaf(c, z, static_cast<float>(2.0 / 15.0 * g * g));
    c = fmaf(c, z, static_cast<float>(-1.0 / 3.0 * g));
    c = fmaf(c, z * k, k);
    const float h = tanh_one(p);
    return fabsf(p) < static_cast<float>(0.3 * f) ? c : h;
}

// Activations of an episode packing: columns of the operand, values per lane, sums of 16 units.
template <int EB> struct Units;

template <> struct Units<4> {
    static constexpr int kRows = 8, kValues = 2;
    static __device__ __forceinline__ int episode(int, int t) { return t; }        // of value i in a lane
    float h[4], l[4];
    // b: the 16 inputs of the tile
    __device__ __forceinline__ void first(const uint4& wh, const uint4& wl, const uint32_t* b)
    {
        mma_k16_first(h, wh, b[0], b[1]);
        mma_k16_first(l, wl, b[0], b[1]);
    }
    __device__ __forceinline__ void add(const uint4& wh, const uint4& wl, const uint32_t* b)
    {
        mma_k16(h, wh, b[0], b[1]);
        mma_k16(l, wl, b[0], b[1]);
    }
    // p of units g and g + 8: their scale_up, f times their biases.  The small products are added up first.
    __device__ __forceinline__ void sums(float up0, float up1, float b0, float b1, float* v) const
    {
        v[0] = fmaf(up0, h[0], fmaf(up0, fmaf(kLoInv, l[0] - l[1], -h[1]), b0));
        v[1] = fmaf(up1, h[2], fmaf(up1, fmaf(kLoInv, l[2] - l[3], -h[3]), b1));
    }
    // eight outputs (hi parts of their weights in rows 0-7 of the tile, low parts in rows 8-15): output g
    static __device__ __forceinline__ void eight(const uint4& w, const uint32_t* b, float up, float bias, float* v)
    {
        float c[4];
        mma_k16_first(c, w, b[0], b[1]);
        v[0] = fmaf(up, c[0], fmaf(up, fmaf(kLoInv, c[2] - c[3], -c[1]), bias));
    }
    // address of this lane's row for store() and load(): 16 units from byte 32 k on
    static __device__ __forceinline__ uint32_t row(uint32_t base, uint32_t pitch, int lane)
    {
        return base + (lane & 7) * pitch + 16u * (lane >> 3);
    }
    static constexpr int kLoadTiles = 2;                          // 16-unit tiles per load
    static __device__ __forceinline__ void load(uint32_t row, uint32_t (*b)[4])
    {
        ldsm_x4(row, b[0][0], b[0][1], b[1][0], b[1][1]);
    }
    static __device__ __forceinline__ void split(const float* v, uint32_t* w)
    {
        uint32_t hi, lo;
        split_two(v[0], v[1], hi, lo);
        w[0] = __byte_perm(hi, lo, 0x5410);
        w[1] = __byte_perm(hi, lo, 0x7632);
    }
    static __device__ __forceinline__ void store(uint32_t row, const float* v)
    {
        uint32_t w[2];
        split(v, w);
        stsm_x2_t(row, w[0], w[1]);
    }
    static __device__ __forceinline__ void transpose(const float* v, uint32_t* b)   // own 16 units as the B operand
    {
        uint32_t w[2];
        split(v, w);
        b[0] = transpose8(w[0]); b[1] = transpose8(w[1]);
    }
};

template <> struct Units<8> {
    static constexpr int kRows = 16, kValues = 4;
    static __device__ __forceinline__ int episode(int i, int t) { return 2 * t + (i & 1); }
    float hh[4], hl[4], lh[4];
    __device__ __forceinline__ void first(const uint4& wh, const uint4& wl, const uint32_t* b)
    {
        mma_k16_first(hh, wh, b[0], b[1]);
        mma_k16_first(hl, wh, b[2], b[3]);
        mma_k16_first(lh, wl, b[0], b[1]);
    }
    __device__ __forceinline__ void add(const uint4& wh, const uint4& wl, const uint32_t* b)   // b[2], b[3]: the low parts
    {
        mma_k16(hh, wh, b[0], b[1]);
        mma_k16(hl, wh, b[2], b[3]);
        mma_k16(lh, wl, b[0], b[1]);
    }
    __device__ __forceinline__ void sums(float up0, float up1, float b0, float b1, float* v) const
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float up = i < 2 ? up0 : up1;
            v[i] = fmaf(up, hh[i], fmaf(up, fmaf(kLoInv, lh[i], -hl[i]), i < 2 ? b0 : b1));
        }
    }
    static __device__ __forceinline__ void eight(const uint4& w, const uint32_t* b, float up, float bias, float* v)
    {
        float c[4], d[4];
        mma_k16_first(c, w, b[0], b[1]);
        mma_k16_first(d, w, b[2], b[3]);
        v[0] = fmaf(up, c[0], fmaf(up, fmaf(kLoInv, c[2], -d[0]), bias));
        v[1] = fmaf(up, c[1], fmaf(up, fmaf(kLoInv, c[3], -d[1]), bias));
    }
    static __device__ __forceinline__ uint32_t row(uint32_t base, uint32_t pitch, int lane)
    {
        return base + ((lane & 7) + 8 * (lane >> 4)) * pitch + 16u * ((lane >> 3) & 1);
    }
    static constexpr int kLoadTiles = 1;
    static __device__ __forceinline__ void load(uint32_t row, uint32_t (*b)[4]) { ldsm_x4(row, b[0][0], b[0][1], b[0][2], b[0][3]); }
    static __device__ __forceinline__ void split(const float* v, uint32_t* w)
    {
        split_two(v[0], v[1], w[0], w[2]);
        split_two(v[2], v[3], w[1], w[3]);
    }
    static __device__ __forceinline__ void store(uint32_t row, const float* v)
    {
        uint32_t w[4];
        split(v, w);
        stsm_x4_t(row, w[0], w[1], w[2], w[3]);
    }
    static __device__ __forceinline__ void transpose(const float* v, uint32_t* b)
    {
        uint32_t w[4];
        split(v, w);
#pragma unroll
        for (int i = 0; i < 4; ++i) b[i] = transpose8(w[i]);
    }
};

enum class Tanh { kOwn, kShared, kFine };                // a reciprocal each, one for two, with the polynomial

template <int EB, Tanh KIND> __device__ __forceinline__ void tanh_units(float* v)
{
#pragma unroll
    for (int i = 0; i < Units<EB>::kValues; i += 2) {
        if (KIND == Tanh::kShared) tanh_two(v[i], v[i + 1]);
        else if (KIND == Tanh::kFine) { v[i] = tanh_fine(v[i]); v[i + 1] = tanh_fine(v[i + 1]); }
        else { v[i] = tanh_one(v[i]); v[i + 1] = tanh_one(v[i + 1]); }
    }
}

}  // namespace ms
}  // namespace evo
