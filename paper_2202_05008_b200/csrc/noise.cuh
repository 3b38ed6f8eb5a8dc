// Counter-based random numbers on the device: Philox4x32-10 (Salmon et al., SC'11), 24-bit
// uniforms and a Box-Muller transform whose every floating-point step is a single IEEE
// round-to-nearest fp32 operation (explicit *_rn intrinsics: the compiler may neither fuse
// nor approximate them), so that the same counters give the same bits on any conforming
// machine.  Used by ask (ES noise), by the regenerated-noise gradient and by task resets
// (the centrally generated roll-out seeds of the paper's Section 2).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace evo {

// The key with its schedule: round r uses (k0 + r W0, k1 + r W1), W = the Weyl increments.  The ten
// pairs are computed once where the key is made (on the host for the solver kernels, whose key is a
// launch parameter: the round keys then come straight out of the constant bank and the generator
// spends no instruction on the schedule).
struct PhiloxKey { uint32_t r[20]; };

__host__ __device__ __forceinline__ PhiloxKey philox_key(uint32_t k0, uint32_t k1)
{
    PhiloxKey k;
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        k.r[2 * i] = k0 + static_cast<uint32_t>(i) * 0x9E3779B9u;
        k.r[2 * i + 1] = k1 + static_cast<uint32_t>(i) * 0xBB67AE85u;
    }
    return k;
}

// counter = (item, row, generation, stream); FIRST: rounds that have been done
template <int FIRST = 0>
__device__ __forceinline__ uint4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                               const PhiloxKey& key)
{
#pragma unroll
    for (int r = FIRST; r < 10; ++r) {
        const uint64_t p0 = static_cast<uint64_t>(0xD2511F53u) * c0;      // one wide multiply each
        const uint64_t p1 = static_cast<uint64_t>(0xCD9E8D57u) * c2;
        const uint32_t hi0 = static_cast<uint32_t>(p0 >> 32), lo0 = static_cast<uint32_t>(p0);
        const uint32_t hi1 = static_cast<uint32_t>(p1 >> 32), lo1 = static_cast<uint32_t>(p1);
        c0 = hi1 ^ c1 ^ key.r[2 * r];
        c1 = lo1;
        c2 = hi0 ^ c3 ^ key.r[2 * r + 1];
        c3 = lo0;
    }
    return make_uint4(c0, c1, c2, c3);
}

// The generator for many rows of one (item, generation, stream): of the first three rounds' six products four do not depend on the
// row.  What is left of those rounds are two products and four exclusive ors with these words.
struct PhiloxItem { uint32_t a, b, c, d, e; };

__device__ __forceinline__ PhiloxItem philox_item(uint32_t item, uint32_t generation, uint32_t stream, const PhiloxKey& key)
{
    const uint64_t p0 = static_cast<uint64_t>(0xD2511F53u) * item, p1 = static_cast<uint64_t>(0xCD9E8D57u) * generation;
    const uint64_t q1 = static_cast<uint64_t>(0xCD9E8D57u) * (static_cast<uint32_t>(p0 >> 32) ^ stream ^ key.r[1]);
    const uint64_t s0 = static_cast<uint64_t>(0xD2511F53u) * (static_cast<uint32_t>(q1 >> 32) ^ static_cast<uint32_t>(p1) ^ key.r[2]);
    PhiloxItem x;
    x.a = static_cast<uint32_t>(p1 >> 32) ^ key.r[0];
    x.b = static_cast<uint32_t>(p0) ^ key.r[3];
    x.c = static_cast<uint32_t>(q1) ^ key.r[4];
    x.d = static_cast<uint32_t>(s0 >> 32) ^ key.r[5];
    x.e = static_cast<uint32_t>(s0);
    return x;
}
__device__ __forceinline__ uint4 philox4x32_10(const PhiloxItem& x, uint32_t row, const PhiloxKey& key)
{
    const uint64_t p = static_cast<uint64_t>(0xD2511F53u) * (x.a ^ row);
    const uint64_t q = static_cast<uint64_t>(0xCD9E8D57u) * (static_cast<uint32_t>(p >> 32) ^ x.b);
    return philox4x32_10<3>(static_cast<uint32_t>(q >> 32) ^ x.c, static_cast<uint32_t>(q), static_cast<uint32_t>(p) ^ x.d, x.e, key);
}

__device__ __forceinline__ float uniform_open(uint32_t r)   // (0, 1]
{
    return __fmul_rn(__uint2float_rn((r >> 8) + 1u), 5.9604644775390625e-08f);
}
__device__ __forceinline__ float uniform_half(uint32_t r)   // [0, 1)
{
    return __fmul_rn(__uint2float_rn(r >> 8), 5.9604644775390625e-08f);
}

// Two fp32 numbers in one 64-bit register: one instruction, two correctly rounded operations (add / mul / fma .rn.f32x2
// round each half like the scalar instruction).
typedef unsigned long long fp2;
__device__ __forceinline__ fp2 fp2_make(float a, float b)
{
    fp2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ fp2 fp2_both(float a) { return fp2_make(a, a); }
__device__ __forceinline__ fp2 fp2_both_bits(uint32_t a) { return fp2_both(__uint_as_float(a)); }
__device__ __forceinline__ void fp2_split(fp2 x, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x)); }
__device__ __forceinline__ fp2 fp2_add(fp2 a, fp2 b) { fp2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ fp2 fp2_mul(fp2 a, fp2 b) { fp2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ fp2 fp2_fma(fp2 a, fp2 b, fp2 c) { fp2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }

constexpr float kRoundMagic = 12582912.0f;       // 1.5 * 2^23: adding it rounds to an integer (ties to even) in the low bits

// ln(k 2^-24) for two integers k in [1, 2^24]: k = m 2^e with m in [sqrt(1/2), sqrt(2)), f = m - 1,
// ln m = f - f^2/2 + f^3 P(f), P of degree 7 (its coefficients are part of the definition of the
// generator).  Relative accuracy holds up to k = 2^24 (u = 1), and there is no division.  e and m come out of the bits of
// float(k) (exact): what lies above the bits of sqrt(1/2) counts whole octaves.
__device__ __forceinline__ fp2 ln_of_u24(uint32_t ka, uint32_t kb)
{
    const uint32_t ba = __float_as_uint(__uint2float_rn(ka)), bb = __float_as_uint(__uint2float_rn(kb));
    const uint32_t xa = ba - 0x3F3504F3u, xb = bb - 0x3F3504F3u;
    const fp2 m = fp2_make(__uint_as_float(ba - (xa & 0xFF800000u)), __uint_as_float(bb - (xb & 0xFF800000u)));
    const fp2 e = fp2_add(fp2_make(__uint_as_float(0x4B400000u + (xa >> 23)), __uint_as_float(0x4B400000u + (xb >> 23))),
                          fp2_both(-(kRoundMagic + 24.0f)));               // exact: small integers
    const fp2 f = fp2_add(m, fp2_both(-1.0f));
    const fp2 z = fp2_mul(f, f);
    fp2 p = fp2_both_bits(0xBDA5EB80u);
    p = fp2_fma(p, f, fp2_both_bits(0x3E022C8Du));
    p = fp2_fma(p, f, fp2_both_bits(0xBE04D5F2u));
    p = fp2_fma(p, f, fp2_both_bits(0x3E116E25u));
    p = fp2_fma(p, f, fp2_both_bits(0xBE2A6AA7u));
    p = fp2_fma(p, f, fp2_both_bits(0x3E4CD0A6u));
    p = fp2_fma(p, f, fp2_both_bits(0xBE800064u));
    p = fp2_fma(p, f, fp2_both_bits(0x3EAAAAA9u));
    const fp2 t = fp2_mul(f, z);
    const fp2 r = fp2_fma(t, p, fp2_mul(fp2_both(-0.5f), z));
    return fp2_fma(e, fp2_both_bits(0x3F317218u), fp2_add(f, r));
}

// Correctly rounded square roots of two numbers that are 0 or in the normal range: from an approximate reciprocal root y,
// g = x y, and the residual of g taken with one rounding, g + (x - g^2) y / 2 (P. Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", 1990).  That this rounds correctly for every argument the generator
// can produce (2^24 of them) is checked exhaustively by a test.  The floor under the root's argument keeps y finite at 0.
__device__ __forceinline__ fp2 sqrt_rn2(fp2 x)
{
    float a, b, ya, yb;
    fp2_split(x, a, b);
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ya) : "f"(fmaxf(a, 1e-30f)));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yb) : "f"(fmaxf(b, 1e-30f)));
    const fp2 y = fp2_make(ya, yb), g = fp2_mul(x, y), ng = fp2_mul(x, fp2_make(-ya, -yb));
    return fp2_fma(fp2_fma(ng, g, x), fp2_mul(fp2_both(0.5f), y), g);
}

// (cos, sin)(2 pi v) for two v = j 2^-24, j in [0, 2^24): quarter-turn reduction, Taylor polynomials
// (sin to x^9, cos to x^10) on [-pi/4, pi/4].
__device__ __forceinline__ void cossin_of_v24(uint32_t ja, uint32_t jb, float (&c)[2], float (&s)[2])
{
    const fp2 w = fp2_mul(fp2_make(__uint2float_rn(ja), __uint2float_rn(jb)), fp2_both(2.384185791015625e-07f));   // 4 v = j 2^-22, exact
    const fp2 k = fp2_add(w, fp2_both(kRoundMagic));            // nearest, ties to even
    const fp2 t = fp2_fma(fp2_add(k, fp2_both(-kRoundMagic)), fp2_both(-1.0f), w);       // exact
    const fp2 x = fp2_mul(t, fp2_both_bits(0x3FC90FDBu));       // pi/2
    const fp2 z = fp2_mul(x, x);

    fp2 sp = fp2_both_bits(0x3638EF1Du);                        //  1/9!
    sp = fp2_fma(sp, z, fp2_both_bits(0xB9500D01u));            // -1/7!
    sp = fp2_fma(sp, z, fp2_both_bits(0x3C088889u));            //  1/5!
    sp = fp2_fma(sp, z, fp2_both_bits(0xBE2AAAABu));            // -1/3!
    sp = fp2_fma(sp, z, fp2_both(1.0f));
    const fp2 sn = fp2_mul(x, sp);

    fp2 cp = fp2_both_bits(0xB493F27Eu);                        // -1/10!
    cp = fp2_fma(cp, z, fp2_both_bits(0x37D00D01u));            //  1/8!
    cp = fp2_fma(cp, z, fp2_both_bits(0xBAB60B61u));            // -1/6!
    cp = fp2_fma(cp, z, fp2_both_bits(0x3D2AAAABu));            //  1/4!
    cp = fp2_fma(cp, z, fp2_both(-0.5f));
    const fp2 cs = fp2_fma(cp, z, fp2_both(1.0f));

    float sv[2], cv[2], kv[2];
    fp2_split(sn, sv[0], sv[1]);
    fp2_split(cs, cv[0], cv[1]);
    fp2_split(k, kv[0], kv[1]);
#pragma unroll
    for (int i = 0; i < 2; ++i) {                               // the two low bits of k: the quarter turn
        const uint32_t q = __float_as_uint(kv[i]);
        const float a = (q & 1u) ? sv[i] : cv[i];               // |cos| source
        const float b = (q & 1u) ? cv[i] : sv[i];               // |sin| source
        c[i] = __uint_as_float(__float_as_uint(a) ^ (((q + 1u) << 30) & 0x80000000u));
        s[i] = __uint_as_float(__float_as_uint(b) ^ ((q << 30) & 0x80000000u));
    }
}

// Box-Muller: (r.x, r.y) -> (z.x, z.y), (r.z, r.w) -> (z.z, z.w);
// radius = sqrt(-2 ln u), u = ((r_even >> 8) + 1) 2^-24; angle = 2 pi (r_odd >> 8) 2^-24.
// Both transforms of a quad in packed arithmetic.  Instruction issue bounded the generator; asking for 8 GB of parameters takes
// 165 instructions per four normals now where two scalar transforms took 231, and the multiply pipe bounds it (a wide
// multiply of the counters holds it for 4 clocks, a packed operation for 2).  1,000,003 columns x 1,000 pairs,
// recomputed noise: ask 2.01 -> 1.67 ms; 131,072 x 8,192, stored noise (12.9 GB written): 2.17 -> 1.81 ms.  Then four of the counters'
// products per column instead of per row (PhiloxItem), and four packed operations instead of eight for the two members: a generation
// of the former, ask and tell, 3,133 -> 3,093 us.  Slower: the upper halves of the products from the idle fp64 pipe,
// by multiply-adds rounded towards zero beside 2^84 (two, four, seven of the last rounds: 3,168, 3,242, 3,317 us).
__device__ __forceinline__ float4 normal4(uint4 r)
{
    float ra, rb, c[2], s[2];
    fp2_split(sqrt_rn2(fp2_mul(fp2_both(-2.0f), ln_of_u24((r.x >> 8) + 1u, (r.z >> 8) + 1u))), ra, rb);
    cossin_of_v24(r.y >> 8, r.w >> 8, c, s);
    return make_float4(__fmul_rn(ra, c[0]), __fmul_rn(ra, s[0]), __fmul_rn(rb, c[1]), __fmul_rn(rb, s[1]));
}

__device__ __forceinline__ float4 stream_normal4(const PhiloxKey& key, uint32_t stream, uint32_t generation,
                                                 uint32_t row, uint32_t item)
{
    return normal4(philox4x32_10(item, row, generation, stream, key));
}

}  // namespace evo
