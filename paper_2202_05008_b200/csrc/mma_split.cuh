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
// tanh.  tanh(x) = 1 - 2 r, r = 1 / (1 + 2^p), p = 2 log2(e) x.  The activation that travels is r (between 0 and 1, so
// its low part needs no scaling), and the layers are rewritten once, when the weights are loaded, to give p from r:
//     p = f (b + sum_k w_k) + sum_k (-2 f w_k) r_k        f = 2 log2(e)
// so a tanh is an exponential, an addition and a reciprocal.  r is as accurate as the 1 - 2 r it stands for.
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
__device__ __forceinline__ void ldsm_x2(uint32_t addr, uint32_t& r0, uint32_t& r1)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}
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

// Weights beyond the fp16 range: a member that has any keeps all of its weights and biases times a power of two that
// brings -2 f w of the largest finite one below it; p is multiplied back.  `peak` = the bit pattern of that
// magnitude.  Infinities are taken as that magnitude (the tanh behind is saturated); NaN stays NaN.
struct Scale {
    float down, up, limit;
    __device__ __forceinline__ explicit Scale(uint32_t peak)
    {
        const int e = static_cast<int>(peak >> 23) - 127, d = e <= 12 ? 0 : e - 12;
        down = __uint_as_float(static_cast<uint32_t>(127 - d) << 23);
        up = __uint_as_float(static_cast<uint32_t>(127 + d) << 23);
        limit = __uint_as_float(max(peak, 0x46000000u));                 // 8,192 or the peak
    }
    __device__ __forceinline__ float weight(float w) const
    {
        asm("max.NaN.f32 %0, %0, %1;\n\tmin.NaN.f32 %0, %0, %2;" : "+f"(w) : "f"(-limit), "f"(limit));
        return w;
    }
};
__device__ __forceinline__ uint32_t finite_magnitude(float w)
{
    const uint32_t m = __float_as_uint(w) & 0x7FFFFFFFu;
    return m < 0x7F800000u ? m : 0u;
}
__device__ __forceinline__ void split_weights(float a, float b, uint32_t& hi, uint32_t& lo)
{
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn((a - f.x) * kLo, (b - f.y) * kLo);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

// This lane's part of the 16x16 weight tile at (row0, col0) of a row-major [no][ni] matrix, times `factor`, as the A
// operand; zeros outside the matrix.  `pairs`: ni is even and W 8-byte aligned.
__device__ __forceinline__ void load_tile(const float* W, int ni, int no, int row0, int col0, int lane, const Scale& sc,
                                          float factor, uint4& hi, uint4& lo, bool pairs = false)
{
    const int g = lane >> 2, t = lane & 3;
    const float k = factor * sc.down;
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {                       // rows g, g + 8; columns 2t, then 2t + 8
        const int row = row0 + g + 8 * (i & 1), col = col0 + 2 * t + 8 * (i >> 1);
        const float* p = W + static_cast<size_t>(row) * ni + col;
        float2 w = make_float2(0.f, 0.f);
        if (pairs) {
            if (row < no && col < ni) w = *reinterpret_cast<const float2*>(p);
        } else {
            if (row < no && col < ni) w.x = p[0];
            if (row < no && col + 1 < ni) w.y = p[1];
        }
        split_weights(sc.weight(w.x) * k, sc.weight(w.y) * k, h[i], l[i]);
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// f (bias + sum of a row's weights) of `unit`; the four lanes of a group add a quarter of the row each
__device__ __forceinline__ float folded_bias(const float* W, const float* B, int ni, int no, int unit, int lane, const Scale& sc)
{
    float s = 0.f;
    if (unit < no) {
        if ((lane & 3) == 0) s = B[unit];
        for (int k = lane & 3; k < ni; k += 4) s += sc.weight(W[static_cast<size_t>(unit) * ni + k]);
    }
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    return kF * s;
}

// r = 1 / (1 + 2^p).  The special-function unit takes 8 clocks per warp for an exponential and 16 for a reciprocal, so two
// values share one: 1/a = b / (a b).  p is held below 60 there so that the product stays finite (r is 0 to fp32 from
// 2^-24 on: 1 - 2 r rounds to 1).
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
__device__ __forceinline__ float logistic2(float p) { return rcp_fast(ex2_fast(p) + 1.0f); }
__device__ __forceinline__ void logistic2(float& p, float& q)
{
    asm("min.NaN.f32 %0, %0, 0f42700000;\n\tmin.NaN.f32 %1, %1, 0f42700000;" : "+f"(p), "+f"(q));
    const float a = ex2_fast(p) + 1.0f, b = ex2_fast(q) + 1.0f;
    const float r = rcp_fast(a * b);
    p = r * b;
    q = r * a;
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
    // up = Scale::up, up_lo = up / 2048, b0 and b1: biases of units g and g + 8
    __device__ __forceinline__ void sums(float up, float up_lo, float b0, float b1, float* v) const
    {
        v[0] = fmaf(up_lo, l[0] - l[1], fmaf(up, h[0] - h[1], b0));
        v[1] = fmaf(up_lo, l[2] - l[3], fmaf(up, h[2] - h[3], b1));
    }
    // eight outputs (hi parts of their weights in rows 0-7 of the tile, low parts in rows 8-15): output g
    static __device__ __forceinline__ void eight(const uint4& w, const uint32_t* b, float up, float up_lo, float bias, float* v)
    {
        float c[4];
        mma_k16_first(c, w, b[0], b[1]);
        v[0] = fmaf(up_lo, c[2] - c[3], fmaf(up, c[0] - c[1], bias));
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
    __device__ __forceinline__ void sums(float up, float up_lo, float b0, float b1, float* v) const
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = fmaf(up_lo, lh[i], fmaf(up, hh[i] - hl[i], i < 2 ? b0 : b1));
    }
    static __device__ __forceinline__ void eight(const uint4& w, const uint32_t* b, float up, float up_lo, float bias, float* v)
    {
        float c[4], d[4];
        mma_k16_first(c, w, b[0], b[1]);
        mma_k16_first(d, w, b[2], b[3]);
        v[0] = fmaf(up_lo, c[2], fmaf(up, c[0] - d[0], bias));
        v[1] = fmaf(up_lo, c[3], fmaf(up, c[1] - d[1], bias));
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

template <int EB> __device__ __forceinline__ void logistic_units(float* v)
{
#pragma unroll
    for (int i = 0; i < Units<EB>::kValues; i += 2) logistic2(v[i], v[i + 1]);
}

}  // namespace ms
}  // namespace evo
