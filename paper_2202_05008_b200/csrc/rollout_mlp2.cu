// Control roll-outs of policies with two hidden layers of up to 128 units, on warp-level tensor-core products
// (mma_split.cuh) with the weights in REGISTERS for all T steps.
//
//   k_rollout_mlp2      block = (member, EB episodes).  A warp keeps RT tiles of 16 rows of both hidden layers (the
//                       second as up to 8 k-tiles) and the action layer's columns of its own units, so the
//                       action layer needs no pass through shared memory: a warp turns its hidden units into
//                       an operand (transpose8) or a dot product and only partial sums meet.
//   k_rollout_cart_solo one warp = (member, 4 episodes), at most 16 hidden units: the step has no barrier and
//                       no shared memory at all; every lane steps the task of its episode.
//
// What bounds them.  Many members per SM: the MMA pipe (2 or 3 MMAs of 8.1 clocks per 16x16 tile and sub-core) and
// the issue slots; few: the serial chain of a step, three barriers long.
//
// Paper: Section 2 (roll-out loop, central seeds), Section 4 (get_actions over the population with parameters as
// data; stateless task step; identical initial observations).
#include "internal.h"
#include "async.cuh"
#include "mma_split.cuh"
#include "noise.cuh"
#include "tasks.cuh"

#include <type_traits>

namespace evo {
namespace {

using namespace ms;

constexpr uint32_t kXPitch = 32 * 2 + 16;           // bytes per column of the state operand [x 28 | 0 4]
constexpr uint32_t kDynTiles = 6;                   // [A | B] in operand tiles: two of 16 rows x three of 16 inputs

// `floats` (a multiple of four) of the member's parameters into shared memory with one bulk copy; false after a time-out (in every thread): the
// return is then reported as NaN, and the copy gets one more bounded chance to land before the block leaves.
__device__ __forceinline__ bool fetch_row(const RolloutMlpArgs& a, DeviceStatus* status, uint64_t* bar, int* ok, float* stage,
                                          const float* src, uint32_t floats, uint32_t member, uint32_t eb)
{
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(bar), 1);
        mbar_init_fence();
        if (!(status->debug_flags & EVO_DEBUG_DROP_COMPLETION))
            bulk_copy_g2s(smem_u32(stage), src, floats * 4u, smem_u32(bar));
        *ok = mbar_wait_bounded(smem_u32(bar), 0u, &status->wait_cycles_log2) ? 1 : 0;
        if (!*ok) {
            atomicOr(&status->sticky, 1u << EVO_ERR_TIMEOUT);
            mbar_wait_bounded(smem_u32(bar), 0u, &status->wait_cycles_log2);
            store_return(a, status, member, eb, __int_as_float(0x7FC00000));
        }
    }
    __syncthreads();
    return *ok != 0;
}

// KT: 16-unit tiles of the first hidden layer (rounded up to 1, 2, 3, 4, 6 or 8); RT: row tiles per warp.  With one row tile
// a warp has all of its weights in registers, the shortest chain, but a wide member then takes eight warps of 128
// registers and two members fill an SM.  RT = 2: four warps, the low parts of the second layer in shared memory,
// three members per SM.  28-128-128-8, 4 episodes, per step of one / two / three resident members: RT = 1 0.76 / 0.97 us
// (three do not fit), RT = 2 0.81 / 1.07 / 1.26 us; 28-96-40-8, 250 members: RT = 1 0.63 us, RT = 2 0.80 us.
// RA, RB: row tiles per warp of the first and of the second layer, at least one of them RT.  A layer of at most half as many tiles as the other has
// one per warp, and those of the other are dealt out in turn; four such members fit an SM.  (With two neighbouring tiles per warp in both, half
// of the warps had nothing to do in the narrow layer: 28-90-40-8, 600 members x 4 episodes, 50 steps 171 -> 112 us; 28-40-90-8 164 -> 111;
// 28-115-51-8, 3,470 x 4 923 -> 715; 5-120-60-1, 500 x 8 234 -> 143; 5-40-110-1, 372 x 8 114 -> 107.)  Where both layers have two a warp takes
// neighbours: dealt out in turn, 28-128-128-8, 4,096 x 4 takes 1,426 instead of 1,331 us.  Cart-pole policies with RB = 2 have registers for
// three members: with four 5-40-110-1, 372 x 8 takes 119.
template <int EB, bool CART, int KT, int RA, int RB>
__global__ void __launch_bounds__(RA + RB == 2 && KT > 4 ? 256 : 128, RA + RB == 4 || (CART && RB == 2) ? 3 : RA + RB == 3 ? 4 : KT > 4 ? 2 : 4)
k_rollout_mlp2(const RolloutMlpArgs a, DeviceStatus* status)
{
    using U = Units<EB>;
    constexpr int RT = RA > RB ? RA : RB;
    constexpr int NV = U::kValues, NH = NV / 2;                      // NH: values of one unit in a lane
    // The special-function unit is what several cart-pole members on an SM wait for (5-64-64-1, 256 members: 778 us with shared
    // reciprocals, 797 without), the issue slots what tanh-linear ones do (28-128-128-8, 4,096: 12.06 and 11.64 ms).
    constexpr Tanh kTanh = CART ? Tanh::kShared : Tanh::kOwn;
    constexpr int MW = RT == 1 && KT > 4 ? 8 : 4;                    // warps at most
    constexpr uint32_t kPitch = (KT + 1) / 2 * 64 + 16;              // bytes per column of the hidden operand (read two tiles at a time)
    // first the parameters (RT = 2: of the first layer only), then (RT = 2) the low parts of the second layer, [warp][tile][k]
    extern __shared__ __align__(128) float stage[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ int copy_ok;
    __shared__ uint32_t peak;
    __shared__ __align__(16) unsigned char h1[U::kRows * kPitch];
    __shared__ __align__(16) float obs[CART ? 5 : 1][EB];            // cart-pole: observation
    __shared__ __align__(16) float part_c[CART ? MW : 1][8 * EB];    // ... shares of the action layer, [warp][g][episode]
    __shared__ __align__(16) unsigned char xop[CART ? 16 : 2 * U::kRows * kXPitch];      // tanh-linear: state, two buffers
    __shared__ __align__(16) float part_t[CART ? 1 : MW][CART ? 1 : 32 * NH];            // ... shares of the action layer
    __shared__ uint4 dyn[CART ? 1 : kDynTiles * 64];                 // ... task matrices in operand order
    __shared__ float x0s[CART ? 1 : kTlNx][EB];                      // ... start states
    __shared__ float rets[2][EB];
    __shared__ float ups[2 * 16 * MW * RT + 8 + (CART ? 0 : 32)];    // scale_up of the units of both hidden layers, the actions, the states

    // (the shuffle tells the compiler that the warp number is the same in all lanes)
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int nw = static_cast<int>(blockDim.x >> 5);
    const uint32_t member = blockIdx.x, eb = blockIdx.y, e0 = eb * EB;
    const int nE = min(static_cast<uint32_t>(EB), a.E - e0);
    const int n1 = static_cast<int>(a.sizes[1]), n2 = static_cast<int>(a.sizes[2]);
    const int nin = CART ? 5 : static_cast<int>(kTlNx), nout = CART ? 1 : static_cast<int>(kTlNa);
    const int mt1 = (n1 + 15) >> 4, mt2 = (n2 + 15) >> 4;
    const int tile0 = RA + RB == 4 ? 2 * warp : warp, apart = RA + RB == 4 ? 1 : nw;                      // the warp's row tiles
    auto tile_of = [&](int r) { return tile0 + r * apart; };
    const uint32_t traced = a.trace ? a.trace_T : 0u;
    const PhiloxKey key = philox_key(a.k0, a.k1);
    // The first warp (cart-pole) or two (tanh-linear) also step the task.  (Another warp in each of the blocks that share an SM was
    // measured and is slower: 5-64-64-1, 256 members, 1.10 us a step against 0.82.)
    const bool tw = warp < (CART ? 1 : 2);

    if (tid == 0) peak = 0u;
    dep_wait();
    const float* row = a.theta + static_cast<size_t>(member) * a.ldD;
    const int w2_at = n1 * nin + n1;
    if (!fetch_row(a, status, &bar, &copy_ok, stage, row, RT == 1 ? a.ldD : static_cast<uint32_t>((w2_at + 3) & ~3), member, eb)) return;
    const uint32_t generation = status->generation;
    {
        // (of the parameters only: what a caller's matrix has in its padding columns is nobody's)
        uint32_t most = 0;
        const float* all = RT == 1 ? stage : row;
        const uint32_t n_params = static_cast<uint32_t>(w2_at + (n1 + 1) * n2 + (n2 + 1) * nout);
        for (uint32_t i = tid; i < n_params / 4u; i += blockDim.x) {
            const float4 w = reinterpret_cast<const float4*>(all)[i];
            most = max(max(most, max(magnitude(w.x), magnitude(w.y))), max(magnitude(w.z), magnitude(w.w)));
        }
        if (tid < static_cast<int>(n_params & 3u)) most = max(most, magnitude(all[(n_params & ~3u) + tid]));
        most = __reduce_max_sync(0xffffffffu, most);
        if (lane == 0) atomicMax(&peak, most);
        for (uint32_t i = tid; i < sizeof(h1) / 4u; i += blockDim.x) reinterpret_cast<uint32_t*>(h1)[i] = 0u;
        if (CART) for (uint32_t i = tid; i < sizeof(part_c) / 4u; i += blockDim.x) (&part_c[0][0])[i] = 0.f;
        else for (uint32_t i = tid; i < sizeof(part_t) / 4u; i += blockDim.x) (&part_t[0][0])[i] = 0.f;
        __syncthreads();
    }
    const int most = scale_exponent(peak);
    const bool scaled = most != 0 || (!CART && scales_dynamics(a.action_scale));

    // ---- weights into registers, times f (see mma_split.cuh) ---------------------------------------
    const float* W1 = stage;
    const float* B1 = W1 + n1 * nin;
    const float* W2 = (RT == 1 ? stage : row) + w2_at;
    const float* B2 = W2 + n2 * n1;
    const float* W3 = B2 + n2;
    const float* B3 = W3 + nout * n2;
    const bool pairs = ((n1 | w2_at) & 1) == 0;                      // the second layer's rows can be read two weights at a time
    uint4 w2h[RB][KT], w2l[RT == 1 ? KT : 1];
    uint4 w1h[CART ? 1 : RA][2], w1l[CART ? 1 : RA][2], w3[CART ? 1 : RB];           // w3: the action layer's own inputs (see Units::eight)
    float w1c[CART ? RA : 1][10], w3c[RB][2], b1[RA][2], b2[RB][2], b3;
    float* const ups1 = ups + 16 * tile0 + g, *const ups2 = ups1 + 16 * MW * RT, *const ups3 = ups + 2 * 16 * MW * RT + g;       // + 16 apart per tile
    uint4* const w2l_s = reinterpret_cast<uint4*>(stage) + warp * (RB * KT * 32) + lane;
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        const int tile = tile_of(r), u0 = 16 * tile + g, u1 = u0 + 8;             // this lane's two units
        if (r < RB) { b2[r < RB ? r : 0][0] = u0 < n2 ? times_f(B2[u0]) : 0.f; b2[r < RB ? r : 0][1] = u1 < n2 ? times_f(B2[u1]) : 0.f; }
        if (r < RA) { b1[r < RA ? r : 0][0] = u0 < n1 ? times_f(B1[u0]) : 0.f; b1[r < RA ? r : 0][1] = u1 < n1 ? times_f(B1[u1]) : 0.f; }
        if constexpr (CART) {                                        // the observation is taken as it is, in fp32
            if (r < RA) {
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    w1c[r < RA ? r : 0][k] = u0 < n1 ? times_f(W1[u0 * 5 + k]) : 0.f;
                    w1c[r < RA ? r : 0][5 + k] = u1 < n1 ? times_f(W1[u1 * 5 + k]) : 0.f;
                }
            }
            if (r < RB) { w3c[r < RB ? r : 0][0] = u0 < n2 ? kF * kActInv * W3[u0] : 0.f; w3c[r < RB ? r : 0][1] = u1 < n2 ? kF * kActInv * W3[u1] : 0.f; }
        } else {
            int s0 = 0, s1 = 0, s3 = 0, none;
            if (scaled) {
                row_exponents(W1, nin, n1, 16 * tile, 2, lane, s0, s1);
                row_exponents(W3, n2, nout, 0, mt2, lane, s3, none);
                if (r < RA) { ups1[16 * r * apart] = scale_up(s0); ups1[16 * r * apart + 8] = scale_up(s1); }
                ups3[0] = scale_up(s3);
            }
            if (r < RA) {
#pragma unroll
                for (int k = 0; k < 2; ++k) load_tile(W1, nin, n1, 16 * tile, 16 * k, lane, s0, s1, w1h[r < RA ? r : 0][k], w1l[r < RA ? r : 0][k]);
            }
            if (r < RB) {
                uint4 lo3;
                load_tile(W3, n2, nout, 0, 16 * tile, lane, s3, 0, w3[r < RB ? r : 0], lo3);
                w3[r < RB ? r : 0].y = lo3.x; w3[r < RB ? r : 0].w = lo3.z;
            }
        }
    }
    if constexpr (RT > 1) __syncthreads();                           // every warp has read the first layer out of `stage`
#pragma unroll
    for (int r = 0; r < RB; ++r) {
        int s0 = 0, s1 = 0;
        if (scaled) {
            row_exponents(W2, n1, n2, 16 * tile_of(r), KT, lane, s0, s1);
            ups2[16 * r * apart] = scale_up(s0); ups2[16 * r * apart + 8] = scale_up(s1);
        }
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            uint4 lo;
            load_tile(W2, n1, n2, 16 * tile_of(r), 16 * k, lane, s0, s1, w2h[r][k], lo, pairs);
            if constexpr (RT == 1) w2l[k] = lo;
            else w2l_s[32 * (r * KT + k)] = lo;
        }
    }
    if constexpr (CART) {
        b3 = times_f(B3[0]);
    } else {
        b3 = times_f(B3[g]);
        for (int i = warp; i < static_cast<int>(kDynTiles); i += nw) {
            uint4 hi, lo;
            int s0, s1;
            load_dynamics(a.task_const, a.action_scale, i, lane, scaled, s0, s1, hi, lo);
            if (scaled) { ups3[8 + 16 * (i / 3)] = scale_up(s0); ups3[16 + 16 * (i / 3)] = scale_up(s1); }
            dyn[i * 64 + lane] = hi;
            dyn[i * 64 + 32 + lane] = lo;
        }
    }

    // ---- reset: seeded start states, the same for every member -------------------------------------------
    CartpoleFast cpc{};
    CpState cps{};
    float snc = 0.f, csc = 1.f, ret = 0.f, ret2 = 0.f;
    float xcur[NV];                                                  // tanh-linear, the two warps that step the task: the state, fp32
#pragma unroll
    for (int i = 0; i < NV; ++i) xcur[i] = 0.f;
    const int te = lane % EB;                                        // cart-pole: this lane's episode (others mirror)
    const uint32_t h1_row = U::row(smem_u32(h1), kPitch, lane);
    const uint32_t x_row = U::row(smem_u32(xop), kXPitch, lane);
    constexpr uint32_t kXBytes = U::kRows * kXPitch;
    if constexpr (CART) {
        if (tw) {
            cpc = cartpole_fast_const(a.tp);
            cps = cartpole_reset(key, generation, e0 + min(te, nE - 1), a.tp[EVO_CP_INIT_RANGE]);
            sincos_fast(cps.th, snc, csc);
            if (lane < EB) { obs[0][te] = cps.x; obs[1][te] = cps.xd; obs[2][te] = csc; obs[3][te] = snc; obs[4][te] = cps.thd; }
        }
    } else {
        for (int i = tid; i < (static_cast<int>(kTlNx) / 4) * EB; i += blockDim.x) {
            const int q = i / EB, e = i % EB;
            const float4 z = stream_normal4(key, 1u, generation, e0 + min(e, nE - 1), q);
            x0s[4 * q][e] = z.x; x0s[4 * q + 1][e] = z.y; x0s[4 * q + 2][e] = z.z; x0s[4 * q + 3][e] = z.w;
        }
        __syncthreads();
        if (tw) {
            float v[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const int unit = 16 * warp + g + (i >= NH ? 8 : 0);
                xcur[i] = unit < static_cast<int>(kTlNx) ? x0s[unit][U::episode(i, t)] : 0.f;
                v[i] = kAct * xcur[i];
            }
            U::store(x_row + 32u * warp, v);
        }
    }
    __syncthreads();

    // ---- time loop ------------------------------------------------------------------------------------------
    uint32_t xin = x_row, xout = x_row + kXBytes;
    // (kActInv where nothing is scaled, but as a constant it becomes immediate operands: 28-128-128-8, 4,096 members then take 12.1 us
    // a step, and 11.5 us with a register)
    const float up = scale_up(most);
    auto roll = [&](auto with_scales) {
        constexpr bool kScaled = decltype(with_scales)::value;
        for (uint32_t step = 0; step < a.T; ++step) {
            if (tile0 < mt1) {
                float v[RA][NV];
                if constexpr (CART) {
                    float o[5][NH];
#pragma unroll
                    for (int k = 0; k < 5; ++k) {
                        if constexpr (EB == 4) o[k][0] = obs[k][t];
                        else { const float2 q = *reinterpret_cast<const float2*>(&obs[k][2 * t]); o[k][0] = q.x; o[k][1] = q.y; }
                    }
#pragma unroll
                    for (int r = 0; r < RA; ++r)
#pragma unroll
                        for (int i = 0; i < NV; ++i) {
                            float s = b1[r][i / NH];
#pragma unroll
                            for (int k = 0; k < 5; ++k) s = fmaf(w1c[r][5 * (i / NH) + k], o[k][i % NH], s);
                            v[r][i] = s;
                        }
                } else {
                    U acc[RA];
                    uint32_t b[2][4];
                    U::load(xin, b);
                    if (U::kLoadTiles == 1) U::load(xin + 32u, b + 1);
#pragma unroll
                    for (int r = 0; r < RA; ++r) acc[r].first(w1h[r][0], w1l[r][0], b[0]);
#pragma unroll
                    for (int r = 0; r < RA; ++r) acc[r].add(w1h[r][1], w1l[r][1], b[1]);
#pragma unroll
                    for (int r = 0; r < RA; ++r) acc[r].sums(kScaled ? ups1[16 * r * apart] : up, kScaled ? ups1[16 * r * apart + 8] : up, b1[r][0], b1[r][1], v[r]);
                }
#pragma unroll
                for (int r = 0; r < RA; ++r) {
                    tanh_units<EB, kTanh>(v[r]);
                    if (RA == 1 || tile_of(r) < KT) U::store(h1_row + 32u * tile_of(r), v[r]);
                }
            }
            __syncthreads();
            CpAhead ahead;
            {
                U acc[RB];
                if (tile0 < mt2) {
                    uint32_t b[2][2][4];                                 // the operands of two tiles, those of the next two on their way
                    U::load(h1_row, b[0]);
                    if (U::kLoadTiles == 1 && KT > 1) U::load(h1_row + 32u, b[0] + 1);
#pragma unroll
                    for (int k = 0; k < KT; ++k) {
                        uint32_t (&now)[2][4] = b[(k >> 1) & 1], (&next)[2][4] = b[((k >> 1) + 1) & 1];
                        if (!(k & 1) && k + 2 < KT) {
                            U::load(h1_row + 32u * k + 64u, next);
                            if (U::kLoadTiles == 1 && k + 3 < KT) U::load(h1_row + 32u * k + 96u, next + 1);
                        }
#pragma unroll
                        for (int r = 0; r < RB; ++r) {
                            const uint4 lo = RT == 1 ? w2l[RT == 1 ? k : 0] : w2l_s[32 * (r * KT + k)];
                            if (k == 0) acc[r].first(w2h[r][k], lo, now[0]);
                            else acc[r].add(w2h[r][k], lo, now[k & 1]);
                        }
                    }
                }
                if (!CART) {                                             // under the MMAs: reward on the pre-step state (0 in other warps, padding rows)
#pragma unroll
                    for (int i = 0; i < NV; ++i) {
                        if (EB == 4 || !(i & 1)) ret = fmaf(-xcur[i], xcur[i], ret); else ret2 = fmaf(-xcur[i], xcur[i], ret2);
                    }
                } else if (tw) {
                    ahead = cartpole_ahead(cpc, cps, snc, csc);
                    if (step > 0u) ret = fmaf(csc, __expf(-cps.x * cps.x), ret);        // reward of the step before, on its post-step state
                }
                if (tile0 < mt2) {
                    float v[RB][NV];
#pragma unroll
                    for (int r = 0; r < RB; ++r) {
                        acc[r].sums(kScaled ? ups2[16 * r * apart] : up, kScaled ? ups2[16 * r * apart + 8] : up, b2[r][0], b2[r][1], v[r]);
                        tanh_units<EB, kTanh>(v[r]);
                    }
                    if constexpr (CART) {
                        float p[NH];
#pragma unroll
                        for (int i = 0; i < NH; ++i) {
                            p[i] = fmaf(w3c[0][1], v[0][NH + i], w3c[0][0] * v[0][i]);
                            if constexpr (RB == 2) p[i] = fmaf(w3c[RB - 1][1], v[RB - 1][NH + i], fmaf(w3c[RB - 1][0], v[RB - 1][i], p[i]));
                        }
                        if constexpr (EB == 4) part_c[warp][lane] = p[0];
                        else *reinterpret_cast<float2*>(&part_c[warp][2 * lane]) = make_float2(p[0], p[1]);
                    } else {                                             // the action layer's share of the warp's units
                        uint32_t b[RB][4];
                        float p[RB][2];
#pragma unroll
                        for (int r = 0; r < RB; ++r) U::transpose(v[r], b[r]);
#pragma unroll
                        for (int r = 0; r < RB; ++r) U::eight(w3[r], b[r], kScaled ? ups3[0] : up, 0.f, p[r]);
                        if constexpr (RB == 2) { p[0][0] += p[RB - 1][0]; p[0][1] += p[RB - 1][1]; }
                        if constexpr (EB == 4) part_t[warp][lane] = p[0][0];
                        else *reinterpret_cast<float2*>(&part_t[warp][2 * lane]) = make_float2(p[0][0], p[0][1]);
                    }
                }
            }
            __syncthreads();
            if constexpr (CART) {
                if (tw) {
                    // the shares of episode te, [warp][g]: this lane adds a quarter (an eighth) of them
                    float p[EB];
#pragma unroll
                    for (int i = 0; i < EB; ++i) p[i] = (&part_c[0][0])[lane + 32 * i];
                    if constexpr (MW > 4) {
#pragma unroll
                        for (int i = 0; i < EB; ++i) p[i] += (&part_c[MW - 4][0])[lane + 32 * i];
                    }
#pragma unroll
                    for (int n = EB / 2; n > 0; n >>= 1)
#pragma unroll
                        for (int i = 0; i < n; ++i) p[i] += p[i + n];
                    float pre = p[0];
#pragma unroll
                    for (int off = EB; off < 32; off <<= 1) pre += __shfl_xor_sync(0xffffffffu, pre, off);
                    const float force = a.action_scale * kActInv * tanh_one(pre + b3);
                    cartpole_finish(cpc, ahead, force, cps, snc, csc);
                    if (lane < EB) { obs[0][te] = cps.x; obs[1][te] = cps.xd; obs[2][te] = csc; obs[3][te] = snc; obs[4][te] = cps.thd; }
                    if (step < traced && lane < nE) trace_state(a, status, member, e0 + te, step, cps);
                }
            } else if (tw) {                                              // action (in both warps), then x' = tanh(A x + B a)
                float v[NV], p[4][NH];
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    if constexpr (EB == 4) p[w][0] = part_t[w][lane];
                    else { const float2 q = *reinterpret_cast<const float2*>(&part_t[w][2 * lane]); p[w][0] = q.x; p[w][1] = q.y; }
                }
                if constexpr (MW > 4) {
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        if constexpr (EB == 4) p[w][0] += part_t[MW - 4 + w][lane];
                        else { const float2 q = *reinterpret_cast<const float2*>(&part_t[MW - 4 + w][2 * lane]); p[w][0] += q.x; p[w][1] += q.y; }
                    }
                }
                U acc;
                const uint4* tiles = dyn + 192 * warp + lane;
                uint32_t b[2][4];
                U::load(xin, b);
                if (U::kLoadTiles == 1) U::load(xin + 32u, b + 1);
                acc.first(tiles[0], tiles[32], b[0]);
                acc.add(tiles[64], tiles[96], b[1]);
#pragma unroll
                for (int i = 0; i < NH; ++i) v[i] = tanh_one(((p[0][i] + p[1][i]) + (p[2][i] + p[3][i])) + b3);
                uint32_t hi, lo;
                split_two(v[0], EB == 4 ? 0.f : v[NH - 1], hi, lo);
                if constexpr (EB == 4) { b[0][0] = transpose8(__byte_perm(hi, lo, 0x5410)); b[0][1] = 0u; }
                else { b[0][0] = transpose8(hi); b[0][1] = 0u; b[0][2] = transpose8(lo); b[0][3] = 0u; }
                if (warp == 0) {                                      // the action's share of the reward
#pragma unroll
                    for (int i = 0; i < NH; ++i) {
                        const float act = a.action_scale * kActInv * v[i];
                        if (i == 0) ret = fmaf(-0.01f * act, act, ret); else ret2 = fmaf(-0.01f * act, act, ret2);
                    }
                }
                acc.add(tiles[128], tiles[160], b[0]);
                acc.sums(kScaled ? ups3[8 + 16 * warp] : kActInv, kScaled ? ups3[16 + 16 * warp] : kActInv, 0.f, 0.f, v);
                tanh_units<EB, kTanh>(v);
                U::store(xout + 32u * warp, v);
#pragma unroll
                for (int i = 0; i < NV; ++i) xcur[i] = kActInv * v[i];              // padding rows: p = 0, exactly 0
                if (step < traced) {
#pragma unroll
                    for (int i = 0; i < NV; ++i) {
                        const int unit = 16 * warp + g + (i >= NH ? 8 : 0), e = U::episode(i, t);
                        if (e < nE && unit < static_cast<int>(kTlNx)) trace_component(a, status, member, e0 + e, step, unit, xcur[i]);
                    }
                }
            }
            const uint32_t x = xin; xin = xout; xout = x;
            __syncthreads();
        }
    };
    if (!scaled) roll(std::false_type{});
    else roll(std::true_type{});

    // ---- block return: fixed order ----------------------------------------------------------------------------
    if constexpr (CART) {
        if (tw && lane < EB) rets[0][te] = fmaf(csc, __expf(-cps.x * cps.x), ret);
    } else if (tw) {
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) {
            ret += __shfl_xor_sync(0xffffffffu, ret, off);
            ret2 += __shfl_xor_sync(0xffffffffu, ret2, off);
        }
        if (g == 0) {
            if (EB == 4) rets[warp][t] = ret;
            else { rets[warp][2 * t] = ret; rets[warp][2 * t + 1] = ret2; }
        }
    }
    __syncthreads();
    if (tid == 0) {
        float s = 0.f;
        for (int e = 0; e < nE; ++e) s += CART ? rets[0][e] : rets[0][e] + rets[1][e];
        store_return(a, status, member, eb, s);
    }
}

// One warp per (member, 4 episodes).  Lane (g, t) steps the task of episode t, mirrored over g, so the first layer's
// inputs are in its registers; a layer's result becomes the next operand by transpose8; the rows of the action
// layer's operand are all the same, so every lane receives its episode's force.
__global__ void __launch_bounds__(32)
k_rollout_cart_solo(const RolloutMlpArgs a, DeviceStatus* status)
{
    using U = Units<4>;
    extern __shared__ __align__(128) float stage[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ int copy_ok;
    const int lane = threadIdx.x, g = lane >> 2, t = lane & 3;
    const uint32_t member = blockIdx.x, eb = blockIdx.y, e0 = eb * 4u;
    const int nE = min(4u, a.E - e0);
    const int n1 = static_cast<int>(a.sizes[1]), n2 = static_cast<int>(a.sizes[2]);
    const PhiloxKey key = philox_key(a.k0, a.k1);
    dep_wait();
    if (!fetch_row(a, status, &bar, &copy_ok, stage, a.theta + static_cast<size_t>(member) * a.ldD, a.ldD, member, eb)) return;
    uint32_t most = 0;
    for (int i = lane; i < 6 * n1 + (n1 + 1) * n2 + n2 + 1; i += 32) most = max(most, magnitude(stage[i]));      // (not the padding)
    const bool scaled = scale_exponent(__reduce_max_sync(0xffffffffu, most)) != 0;
    const uint32_t traced = a.trace ? a.trace_T : 0u;

    const float* W1 = stage;
    const float* B1 = W1 + n1 * 5;
    const float* W2 = B1 + n1;
    const float* B2 = W2 + n2 * n1;
    const float* W3 = B2 + n2;
    float w1[2][6], b2[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int u = g + 8 * i;
#pragma unroll
        for (int k = 0; k < 5; ++k) w1[i][k] = u < n1 ? times_f(W1[u * 5 + k]) : 0.f;
        w1[i][5] = u < n1 ? times_f(B1[u]) : 0.f;
        b2[i] = u < n2 ? times_f(B2[u]) : 0.f;
    }
    uint4 w2h, w2l;
    int s0 = 0, s1 = 0, s3 = 0;
    if (scaled) {
        row_exponents(W2, n1, n2, 0, 1, lane, s0, s1);
        s3 = scale_exponent(__reduce_max_sync(0xffffffffu, lane < n2 ? magnitude(W3[lane]) : 0u));
    }
    load_tile(W2, n1, n2, 0, 0, lane, s0, s1, w2h, w2l);
    uint32_t w3h[2], w3l[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int col = 2 * t + 8 * k;
        split_weights(col < n2 ? finite(W3[col]) : 0.f, col + 1 < n2 ? finite(W3[col + 1]) : 0.f, kF * scale_down(s3), w3h[k], w3l[k]);
    }
    const uint4 w3 = make_uint4(w3h[0], w3l[0], w3h[1], w3l[1]);        // the one output in every row (see Units::eight)
    const float b3 = times_f(W3[n2]);

    const CartpoleFast c = cartpole_fast_const(a.tp);
    CpState s = cartpole_reset(key, status->generation, e0 + min(t, nE - 1), a.tp[EVO_CP_INIT_RANGE]);
    float sn, cs, ret = 0.f;
    sincos_fast(s.th, sn, cs);

    auto roll = [&](auto with_scales) {
        constexpr bool kScaled = decltype(with_scales)::value;
        for (uint32_t step = 0; step < a.T; ++step) {
            float v[2];
            uint32_t b[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                // the velocity and the angle come last out of a step, so they go in last here
                float p = fmaf(w1[i][0], s.x, w1[i][5]);
                p = fmaf(w1[i][1], s.xd, p);
                p = fmaf(w1[i][4], s.thd, p);
                p = fmaf(w1[i][3], sn, p);
                v[i] = tanh_one(fmaf(w1[i][2], cs, p));
            }
            U::transpose(v, b);
            U h2;
            h2.first(w2h, w2l, b);
            const CpAhead ahead = cartpole_ahead(c, s, sn, cs);
            if (step > 0u) ret = fmaf(cs, __expf(-s.x * s.x), ret);       // reward of the step before, on its post-step state
            h2.sums(kScaled ? scale_up(s0) : kActInv, kScaled ? scale_up(s1) : kActInv, b2[0], b2[1], v);
            v[0] = tanh_one(v[0]); v[1] = tanh_one(v[1]);                 // a reciprocal each: the unit is idle, the chain shorter
            U::transpose(v, b);
            U::eight(w3, b, kScaled ? scale_up(s3) : kActInv, b3, v);
            cartpole_finish(c, ahead, a.action_scale * kActInv * tanh_one(v[0]), s, sn, cs);
            if (step < traced && lane < nE) trace_state(a, status, member, e0 + lane, step, s);
        }
    };
    if (scaled) roll(std::true_type{});
    else roll(std::false_type{});
    ret = fmaf(cs, __expf(-s.x * s.x), ret);
    float v = t < nE ? ret : 0.f;
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    if (lane == 0) store_return(a, status, member, eb, v);
}

using Mlp2Kernel = void (*)(const RolloutMlpArgs, DeviceStatus*);

// ra, rb: row tiles per warp of the two layers
template <int EB, bool CART, int KT>
Mlp2Kernel pick_tiles(uint32_t ra, uint32_t rb)
{
    if constexpr (KT == 4) return ra == 1u ? k_rollout_mlp2<EB, CART, KT, 1, 2> : k_rollout_mlp2<EB, CART, KT, 2, 2>;      // (the second layer is the wider one then)
    else return rb == 1u ? k_rollout_mlp2<EB, CART, KT, 2, 1> : k_rollout_mlp2<EB, CART, KT, 2, 2>;
}
template <int EB, bool CART>
Mlp2Kernel pick_kernel(uint32_t kt, uint32_t ra, uint32_t rb)
{
    if (ra + rb > 2u) return kt == 4u ? pick_tiles<EB, CART, 4>(ra, rb) : kt == 6u ? pick_tiles<EB, CART, 6>(ra, rb) : pick_tiles<EB, CART, 8>(ra, rb);
    switch (kt) {
        case 1: return k_rollout_mlp2<EB, CART, 1, 1, 1>;
        case 2: return k_rollout_mlp2<EB, CART, 2, 1, 1>;
        case 3: return k_rollout_mlp2<EB, CART, 3, 1, 1>;
        case 4: return k_rollout_mlp2<EB, CART, 4, 1, 1>;
        case 6: return k_rollout_mlp2<EB, CART, 6, 1, 1>;
        default: return k_rollout_mlp2<EB, CART, 8, 1, 1>;
    }
}

uint32_t hidden_tiles(const uint32_t* sizes) { return ((sizes[1] > sizes[2] ? sizes[1] : sizes[2]) + 15u) / 16u; }

}  // namespace

// Episodes per block; 0: not a policy for these kernels.  Eight episodes take three MMAs per weight tile where four
// take two.
uint32_t rollout_mlp2_eb(uint32_t task, uint32_t n_layers, const uint32_t* sizes, uint32_t episodes)
{
    if (n_layers != 3u || sizes[1] > 128u || sizes[2] > 128u) return 0u;
    if (task == EVO_TASK_CARTPOLE && hidden_tiles(sizes) == 1u) return 4u;
    return episodes > 4u ? 8u : 4u;
}

int launch_rollout_mlp2(cudaStream_t st, const RolloutMlpArgs& a, DeviceStatus* status)
{
    const bool cart = a.task == EVO_TASK_CARTPOLE;
    const uint32_t tiles = hidden_tiles(a.sizes);
    size_t bytes = static_cast<size_t>(a.ldD) * sizeof(float);
    if (cart && tiles == 1u)
        return launch_dependent(k_rollout_cart_solo, dim3(a.P, a.n_eb), dim3(32), bytes, st, a, status) == cudaSuccess ? 1 : -1;
    // Wide policies: all weights in registers as long as no SM gets more than the two members that then fit.
    const uint64_t blocks = static_cast<uint64_t>(a.P) * a.n_eb;
    const bool wide = tiles > 4u, two_tiles = wide && blocks > 2u * kSms;
    uint32_t kt = (a.sizes[1] + 15u) / 16u;
    if (wide) kt = two_tiles && kt <= 4u ? 4u : kt <= 6u ? 6u : 8u;
    uint32_t warps = two_tiles ? (tiles + 1u) / 2u : tiles;
    if (!cart && warps < 2u) warps = 2u;
    const uint32_t ra = two_tiles && (a.sizes[1] + 15u) / 16u > warps ? 2u : 1u, rb = two_tiles && (a.sizes[2] + 15u) / 16u > warps ? 2u : 1u;
    auto kernel = a.EB == 4u ? (cart ? pick_kernel<4, true>(kt, ra, rb) : pick_kernel<4, false>(kt, ra, rb))
                             : (cart ? pick_kernel<8, true>(kt, ra, rb) : pick_kernel<8, false>(kt, ra, rb));
    if (two_tiles) {                                                  // the first layer, then the low parts of the second
        const size_t first = ((a.sizes[0] + 1u) * a.sizes[1] + 3u) * sizeof(float), low = warps * rb * kt * 512u;
        bytes = first > low ? first : low;
    }
    bytes = spread_over_sms(kernel, bytes, blocks);
    if (!a.attr_done &&
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) != cudaSuccess) return -1;
    return launch_dependent(kernel, dim3(a.P, a.n_eb), dim3(32u * warps), bytes, st, a, status) == cudaSuccess ? 1 : -1;
}

}  // namespace evo
