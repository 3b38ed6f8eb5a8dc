// Warp-level tensor-core products with fp32 accuracy for the control roll-outs.
//
// A weight is two fp16 numbers, w = hi + lo with hi = fp16(w), lo = fp16(w - hi) (22 mantissa bits), an
// activation likewise; products of fp16 numbers are exact and sums are kept in fp32.  The products run
// as mma.sync m16n8k16: the 16x16 weight tile is an operand in REGISTERS (or one 128-bit shared-memory
// load per lane), which is what these roll-outs need: a member has its own weights and only 4 or 8
// columns of activations, so an MMA is paced by its weight operand.  tcgen05 fetches 4 KB of
// weights from tensor or shared memory per 128x16 tile and step (21-32 clocks for 8 columns) and its result is
// read 340 clocks later at the earliest; mma.sync takes the same 128x16x8 product from registers in 16
// clocks of the four sub-cores (8.1 clocks per m16n8k16 and sub-core, measured) and the
// result is there after 21.
//
// Activations of a layer lie in shared memory as the B operand, [column][unit] fp16, a column = one episode and
// part.  Two packings of the columns of an n-tile (8 columns) are used:
//   pairs:  column 2e = hi, 2e + 1 = lo of episode e (4 episodes): a lane of the accumulator then holds both
//           products of its episode side by side; all four cross terms, two MMAs per tile
//   planes: one n-tile of the hi parts and one of the lo parts of 8 episodes: hi*hi, hi*lo and lo*hi, three MMAs
//           per tile for twice the episodes (lo*lo is below 2^-24 of the product)
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

// 8x8 fp16 matrices from shared memory, row addresses from lanes 0-7, 8-15, ...
__device__ __forceinline__ void ldsm_x2(uint32_t addr, uint32_t& r0, uint32_t& r1)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr) : "memory");
}
// accumulator fragments (rows = units) to shared memory as [column][unit]
__device__ __forceinline__ void stsm_x2_t(uint32_t addr, uint32_t r0, uint32_t r1)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1,%2};" :: "r"(addr), "r"(r0), "r"(r1) : "memory");
}

// x = hi + lo, hi in the low half of the word
__device__ __forceinline__ uint32_t split_pair(float x)
{
    const float hi = __half2float(__float2half_rn(x));
    uint32_t d;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(x - hi), "f"(hi));
    return d;
}

// hi and lo parts of two weights (magnitudes beyond the fp16 range are taken as the largest fp16 number:
// the tanh behind such a weight is saturated; NaN stays NaN)
__device__ __forceinline__ void split_weights(float a, float b, uint32_t& hi, uint32_t& lo)
{
    asm("max.NaN.f32 %0, %0, 0fC77FE000;\n\tmin.NaN.f32 %0, %0, 0f477FE000;" : "+f"(a));
    asm("max.NaN.f32 %0, %0, 0fC77FE000;\n\tmin.NaN.f32 %0, %0, 0f477FE000;" : "+f"(b));
    const __half2 h = __floats2half2_rn(a, b);
    const float2 hf = __half22float2(h);
    const __half2 l = __floats2half2_rn(a - hf.x, b - hf.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

// This lane's part of the 16x16 weight tile at (row0, col0) of a row-major [no][ni] matrix, as the A operand;
// zeros outside the matrix.
__device__ __forceinline__ void load_tile(const float* __restrict__ W, int ni, int no, int row0, int col0, int lane,
                                          uint4& hi, uint4& lo)
{
    const int g = lane >> 2, t = lane & 3;
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {                       // rows g, g + 8; columns 2t, then 2t + 8
        const int row = row0 + g + 8 * (i & 1), col = col0 + 2 * t + 8 * (i >> 1);
        const float* p = W + static_cast<size_t>(row) * ni + col;
        const float a = (row < no && col < ni) ? __ldg(p) : 0.f, b = (row < no && col + 1 < ni) ? __ldg(p + 1) : 0.f;
        split_weights(a, b, h[i], l[i]);
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// tanh(x) = 1 - 2 / (e^2x + 1) on the special-function unit, which takes 8 clocks per warp for an exponential and
// 16 for a reciprocal: the values share one reciprocal, 1/a0 = a1 / (a0 a1) and so on (absolute error about
// 3e-7).  e^2x is held below 2^30 so that the product of four stays finite (tanh is 1 to fp32 long before).
__device__ __forceinline__ float exp2x(float x)
{
    float e;
    asm("{\n\t.reg .f32 t;\n\tmul.f32 t, %1, 0f4038AA3B;\n\tmin.NaN.f32 t, t, 0f41F00000;\n\tex2.approx.ftz.f32 %0, t;\n\t}" : "=f"(e) : "f"(x));
    return e;
}
__device__ __forceinline__ float rcp_fast(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float tanh1(float x) { return fmaf(-2.0f, rcp_fast(exp2x(x) + 1.0f), 1.0f); }
__device__ __forceinline__ void tanh2(float& x, float& y)
{
    const float a = exp2x(x) + 1.0f, b = exp2x(y) + 1.0f;
    const float r = rcp_fast(a * b);
    x = fmaf(-2.0f, r * b, 1.0f);
    y = fmaf(-2.0f, r * a, 1.0f);
}
__device__ __forceinline__ void tanh4(float& x, float& y, float& z, float& w)
{
    const float a = exp2x(x) + 1.0f, b = exp2x(y) + 1.0f, c = exp2x(z) + 1.0f, d = exp2x(w) + 1.0f;
    const float ab = a * b, cd = c * d, r = rcp_fast(ab * cd);
    const float rab = r * cd, rcd = r * ab;
    x = fmaf(-2.0f, rab * b, 1.0f);
    y = fmaf(-2.0f, rab * a, 1.0f);
    z = fmaf(-2.0f, rcd * d, 1.0f);
    w = fmaf(-2.0f, rcd * c, 1.0f);
}

}  // namespace ms
}  // namespace evo
