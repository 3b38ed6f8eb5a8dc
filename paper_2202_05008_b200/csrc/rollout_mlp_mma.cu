// Control roll-out for any multi-layer policy whose weights fit one SM's shared memory, on warp-level
// tensor-core products (mma_split.cuh): for those that the kernels with the weights in registers (k_rollout_mlp2, k_rollout_mlp_deep) do
// not take.
//
// Block = (member, EB episodes).  The member's weights are split into fp16 pairs once and kept in shared
// memory in operand order: a 16x16 tile is one 128-bit load per lane and part.  A warp takes 16 units of a
// layer (several if the layer has more than the block's warps), applies bias and tanh to its accumulators in
// registers, and writes the two fp16 parts of the result as the next layer's B operand.  A layer so costs one
// barrier (28-64-64-64-8, 4 episodes, were it to run here: 1.69 us a step with one member on an SM, 2.21 us with four).  The dynamics of the tanh-linear task
// are one more layer ([A | B] on the state with the action behind it); the cart-pole's five inputs are taken
// in fp32, and a warp of its own steps the task, which works on the coming step while the layers run.
//
// Bounds: shared-memory reads of the weight operands (1 KB per tile and step) at many members per SM, the chain
// of a step at few.
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

constexpr uint32_t kXPitch = 48 * 2 + 16;           // bytes per column of the [x 28 | 0 4 | a 8 | 0 8] operand
constexpr size_t kMaxSmem = 222u * 1024u;

struct Plan {
    uint32_t mt[EVO_MAX_LAYERS + 1], kt[EVO_MAX_LAYERS + 1];   // 16-unit and 16-input tiles of a layer; last entry: dynamics
    uint32_t tile0[EVO_MAX_LAYERS + 1];             // first tile of a layer in the operand area
    uint32_t bias0[EVO_MAX_LAYERS + 1];             // first float of a layer's biases
    uint32_t tiles, biases, pitch;                  // pitch: bytes per column of the hidden operands
    uint32_t warps;                                 // layer warps
    bool     fine;                                  // tanh with the polynomial (see tanh_fine)
    size_t   smem;
};

// p of 16 units: tiles = the units' weight tiles in operand order, bias and (SCALED) exponent of units g and g + 8, up = kActInv
template <int EB, bool SCALED>
__device__ __forceinline__ void unit_sums(const uint4* tiles, uint32_t kt, uint32_t in, uint32_t pitch, int lane, float b0, float b1,
                                          const uint8_t* exponent, float up, float* v)
{
    using U = Units<EB>;
    U acc;
    const uint32_t row = U::row(in, pitch, lane);
    tiles += lane;
    {                                                   // tiles two at a time (the operand of a last odd one's partner is read, not used)
        uint32_t b[2][4];
        U::load(row, b);
        acc.first(tiles[0], tiles[32], b[0]);
        if (kt > 1u) {
            if (U::kLoadTiles == 1) U::load(row + 32u, b + 1);
            acc.add(tiles[64], tiles[96], b[1]);
        }
    }
    uint32_t k = 2;
#pragma unroll 2
    for (; k + 1u < kt; k += 2u) {
        const uint4 h0 = tiles[k * 64u], l0 = tiles[k * 64u + 32u], h1 = tiles[k * 64u + 64u], l1 = tiles[k * 64u + 96u];
        uint32_t b[2][4];
        U::load(row + 32u * k, b);
        if (U::kLoadTiles == 1) U::load(row + 32u * k + 32u, b + 1);
        acc.add(h0, l0, b[0]);
        acc.add(h1, l1, b[1]);
    }
    if (k < kt) {
        uint32_t b[2][4];
        U::load(row + 32u * k, b);
        acc.add(tiles[k * 64u], tiles[k * 64u + 32u], b[0]);
    }
    acc.sums(SCALED ? scale_up(exponent[0]) : up, SCALED ? scale_up(exponent[8]) : up, b0, b1, v);
}

template <int EB, bool CART, bool FINE>
__global__ void __launch_bounds__(288)
k_rollout_mlp_mma(const RolloutMlpArgs a, const Plan p, DeviceStatus* status)
{
    constexpr int NV = Units<EB>::kValues;
    extern __shared__ __align__(16) unsigned char mma_smem[];
    __shared__ float obs[5][EB], act[EB], x0s[kTlNx][EB], rets[9][EB];
    __shared__ uint32_t peaks[9];
    uint4* tiles = reinterpret_cast<uint4*>(mma_smem);
    float* bias = reinterpret_cast<float*>(mma_smem + static_cast<size_t>(p.tiles) * 1024u);
    uint8_t* exponents = reinterpret_cast<uint8_t*>(bias + p.biases);
    float* w_in = bias + p.biases + p.biases / 4u;                   // cart-pole: [unit][8] = five weights, bias
    const uint32_t buf0 = smem_u32(w_in + (CART ? p.mt[0] * 128u : 0u));
    const uint32_t buf_bytes = Units<EB>::kRows * p.pitch;
    const uint32_t xbuf = buf0 + 2u * buf_bytes;                     // tanh-linear: two state operands
    constexpr uint32_t xbuf_bytes = Units<EB>::kRows * kXPitch;

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, g = lane >> 2, t = lane & 3;
    const uint32_t member = blockIdx.x, eb = blockIdx.y, e0 = eb * EB;
    const int nE = min(static_cast<uint32_t>(EB), a.E - e0);
    const uint32_t layers = a.n_layers, nw = p.warps;
    const bool layer_warp = warp < static_cast<int>(nw);
    const uint32_t traced = a.trace ? a.trace_T : 0u;
    const PhiloxKey key = philox_key(a.k0, a.k1);
    dep_wait();
    const uint32_t generation = status->generation;
    const float* th = a.theta + static_cast<size_t>(member) * a.ldD;

    // ---- weights: rows of theta -> operand tiles (whole warps, one tile at a time) --------------------
    uint32_t n_params = 0;
    for (uint32_t l = 0; l < layers; ++l) n_params += (a.sizes[l] + 1u) * a.sizes[l + 1];
    uint32_t most = 0;
    for (uint32_t i = tid; i < n_params; i += blockDim.x) most = max(most, magnitude(__ldg(th + i)));
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0) peaks[warp] = most;
    __syncthreads();
    most = 0;
    for (uint32_t i = 0; i < blockDim.x / 32u; ++i) most = max(most, peaks[i]);
    const int largest = scale_exponent(most);
    const bool scaled = largest != 0 || (!CART && scales_dynamics(a.action_scale));
    {
        uint32_t off = 0;
        for (uint32_t l = 0; l < layers; ++l) {
            const int ni = static_cast<int>(a.sizes[l]), no = static_cast<int>(a.sizes[l + 1]);
            const float* W = th + off;
            const float* B = W + ni * no;
            off += static_cast<uint32_t>(ni * no + no);
            if (CART && l == 0) {
                for (uint32_t i = tid; i < p.mt[0] * 128u; i += blockDim.x) {
                    const int u = static_cast<int>(i >> 3), k = static_cast<int>(i & 7u);
                    w_in[i] = (u < no && k < 6) ? times_f(k < 5 ? __ldg(W + u * 5 + k) : __ldg(B + u)) : 0.f;
                }
                continue;
            }
            if (scaled) {
                for (uint32_t m = warp; m < p.mt[l]; m += blockDim.x >> 5) {
                    int n0, n1;
                    row_exponents(W, ni, no, 16 * static_cast<int>(m), static_cast<int>(p.kt[l]), lane, n0, n1);
                    if (t < 2) exponents[p.bias0[l] + 16u * m + g + 8u * t] = static_cast<uint8_t>(t ? n1 : n0);
                }
                __syncthreads();
            }
            for (uint32_t i = warp; i < p.mt[l] * p.kt[l]; i += blockDim.x >> 5) {
                const uint8_t* n = exponents + p.bias0[l] + 16u * (i / p.kt[l]) + g;
                uint4 hi, lo;
                load_tile(W, ni, no, 16 * static_cast<int>(i / p.kt[l]), 16 * static_cast<int>(i % p.kt[l]), lane, scaled ? n[0] : 0,
                          scaled ? n[8] : 0, hi, lo);
                tiles[(p.tile0[l] + i) * 64u + lane] = hi;
                tiles[(p.tile0[l] + i) * 64u + 32u + lane] = lo;
            }
            for (uint32_t i = tid; i < p.mt[l] * 16u; i += blockDim.x)
                bias[p.bias0[l] + i] = static_cast<int>(i) < no ? times_f(__ldg(B + i)) : 0.f;
        }
        if (!CART) {
            for (uint32_t i = warp; i < 6u; i += blockDim.x >> 5) {
                uint4 hi, lo;
                int n0, n1;
                load_dynamics(a.task_const, a.action_scale, static_cast<int>(i), lane, scaled, n0, n1, hi, lo);
                tiles[(p.tile0[layers] + i) * 64u + lane] = hi;
                tiles[(p.tile0[layers] + i) * 64u + 32u + lane] = lo;
                if (t < 2) exponents[p.bias0[layers] + 16u * (i / 3u) + g + 8u * t] = static_cast<uint8_t>(t ? n1 : n0);
            }
            for (uint32_t i = tid; i < 32u; i += blockDim.x) bias[p.bias0[layers] + i] = 0.f;
            for (uint32_t i = tid; i < 2u * xbuf_bytes / 4u; i += blockDim.x)
                reinterpret_cast<uint32_t*>(mma_smem + (xbuf - smem_u32(mma_smem)))[i] = 0u;
        }
    }

    // ---- reset: seeded start states, the same for every member -----------------------------------------
    CartpoleFast cpc{};
    CpState cps{};
    float snc = 0.f, csc = 1.f, ret = 0.f, ret2 = 0.f;
    const int te = lane % EB;                                        // task warp: its lane's episode (others mirror)
    if (CART) {
        if (!layer_warp) {
            cpc = cartpole_fast_const(a.tp);
            cps = cartpole_reset(key, generation, e0 + min(te, nE - 1), a.tp[EVO_CP_INIT_RANGE]);
            sincos_fast(cps.th, snc, csc);
            if (lane < EB) { obs[0][te] = cps.x; obs[1][te] = cps.xd; obs[2][te] = csc; obs[3][te] = snc; obs[4][te] = cps.thd; }
        }
        __syncthreads();
    } else {
        for (int i = tid; i < (static_cast<int>(kTlNx) / 4) * EB; i += blockDim.x) {
            const int q = i / EB, e = i % EB;
            const float4 z = stream_normal4(key, 1u, generation, e0 + min(e, nE - 1), q);
            x0s[4 * q][e] = z.x; x0s[4 * q + 1][e] = z.y; x0s[4 * q + 2][e] = z.z; x0s[4 * q + 3][e] = z.w;
        }
        __syncthreads();
        for (uint32_t m = warp; m < 2u; m += nw) {
            float v[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const uint32_t row = 16u * m + g + (i >= NV / 2 ? 8u : 0u);
                const int e = EB == 4 ? t : 2 * t + (i & 1);
                v[i] = row < kTlNx ? x0s[row][e] : 0.f;
                if (EB == 4 || !(i & 1)) ret = fmaf(-v[i], v[i], ret); else ret2 = fmaf(-v[i], v[i], ret2);
                v[i] *= kAct;
            }
            Units<EB>::store(Units<EB>::row(xbuf, kXPitch, lane) + 32u * m, v);
        }
        __syncthreads();
    }

    // ---- time loop -----------------------------------------------------------------------------------------
    const float up = scale_up(largest);                              // kActInv where nothing is scaled, in a register
    auto roll = [&](auto with_scales) {
        constexpr bool kScaled = decltype(with_scales)::value;
        for (uint32_t step = 0; step < a.T; ++step) {
            const uint32_t xin = xbuf + (step & 1u) * xbuf_bytes, xout = xbuf + ((step + 1u) & 1u) * xbuf_bytes;
            CpAhead ahead{};
            if (CART && !layer_warp) ahead = cartpole_ahead(cpc, cps, snc, csc);
            for (uint32_t l = 0; l < layers; ++l) {
                const bool last = l + 1u == layers;
                const uint32_t in = l == 0u ? xin : buf0 + ((l + 1u) & 1u) * buf_bytes, out = buf0 + (l & 1u) * buf_bytes;
                const uint32_t in_pitch = l == 0u ? kXPitch : p.pitch;
                if (layer_warp) {
                    for (uint32_t m = warp; m < p.mt[l]; m += nw) {
                        float v[NV];
                        if (CART && l == 0u) {
                            const float* wa = w_in + (16u * m + g) * 8u;
                            const float4 w0 = *reinterpret_cast<const float4*>(wa), w1 = *reinterpret_cast<const float4*>(wa + 64);
                            const float2 q0 = *reinterpret_cast<const float2*>(wa + 4), q1 = *reinterpret_cast<const float2*>(wa + 68);
#pragma unroll
                            for (int i = 0; i < NV; ++i) {
                                const int e = EB == 4 ? t : 2 * t + (i & 1);
                                const bool up = i >= NV / 2;
                                float s = fmaf(up ? w1.x : w0.x, obs[0][e], up ? q1.y : q0.y);
                                s = fmaf(up ? w1.y : w0.y, obs[1][e], s);
                                s = fmaf(up ? w1.z : w0.z, obs[2][e], s);
                                s = fmaf(up ? w1.w : w0.w, obs[3][e], s);
                                v[i] = fmaf(up ? q1.x : q0.x, obs[4][e], s);
                            }
                        } else {
                            const uint32_t at = p.bias0[l] + 16u * m + g;
                            unit_sums<EB, kScaled>(tiles + (p.tile0[l] + m * p.kt[l]) * 64u, p.kt[l], in, in_pitch, lane, bias[at],
                                                   bias[at + 8u], exponents + at, up, v);
                        }
                        tanh_units<EB, FINE ? Tanh::kFine : Tanh::kOwn>(v);
                        if (!last) {
                            Units<EB>::store(Units<EB>::row(out, p.pitch, lane) + 32u * m, v);
                        } else if (CART) {
                            if (g == 0) {
                                if (EB == 4) act[t] = v[0];
                                else { act[2 * t] = v[0]; act[2 * t + 1] = v[1]; }
                            }
                        } else {                                         // the action, and its share of the reward (units 8..15 are padding)
                            Units<EB>::store(Units<EB>::row(xin, kXPitch, lane) + 64u, v);
#pragma unroll
                            for (int i = 0; i < NV / 2; ++i) {
                                const float act = a.action_scale * kActInv * v[i];
                                if (i == 0) ret = fmaf(-0.01f * act, act, ret); else ret2 = fmaf(-0.01f * act, act, ret2);
                            }
                        }
                    }
                }
                __syncthreads();
            }
            if (CART) {
                if (!layer_warp) {
                    cartpole_finish(cpc, ahead, a.action_scale * kActInv * act[te], cps, snc, csc);
                    ret = fmaf(csc, __expf(-cps.x * cps.x), ret);         // reward on the post-step state
                    if (lane < EB) {
                        obs[0][te] = cps.x; obs[1][te] = cps.xd; obs[2][te] = csc; obs[3][te] = snc; obs[4][te] = cps.thd;
                        if (step < traced && te < nE) trace_state(a, status, member, e0 + te, step, cps);
                    }
                }
            } else {
                for (uint32_t m = warp; m < 2u; m += nw) {
                    float v[NV];
                    const uint32_t at = p.bias0[layers] + 16u * m + g;
                    unit_sums<EB, kScaled>(tiles + (p.tile0[layers] + m * 3u) * 64u, 3u, xin, kXPitch, lane, bias[at], bias[at + 8u],
                                           exponents + at, kActInv, v);
                    tanh_units<EB, FINE ? Tanh::kFine : Tanh::kOwn>(v);
                    Units<EB>::store(Units<EB>::row(xout, kXPitch, lane) + 32u * m, v);
#pragma unroll
                    for (int i = 0; i < NV; ++i) v[i] *= kActInv;
#pragma unroll
                    for (int i = 0; i < NV; ++i) {
                        const uint32_t row = 16u * m + g + (i >= NV / 2 ? 8u : 0u);
                        const int e = EB == 4 ? t : 2 * t + (i & 1);
                        if (step + 1u < a.T) {                           // reward of the next step: its pre-step state (padding rows are 0)
                            if (EB == 4 || !(i & 1)) ret = fmaf(-v[i], v[i], ret); else ret2 = fmaf(-v[i], v[i], ret2);
                        }
                        if (step < traced && e < nE && row < kTlNx) trace_component(a, status, member, e0 + e, step, row, v[i]);
                    }
                }
            }
            __syncthreads();
        }
    };
    if (scaled) roll(std::true_type{});
    else roll(std::false_type{});

    // ---- block return: fixed order --------------------------------------------------------------------------
    if (CART) {
        if (!layer_warp && lane < EB) rets[0][te] = ret;
    } else {
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
        for (int e = 0; e < nE; ++e)
            for (uint32_t w = 0; w < (CART ? 1u : nw); ++w) s += rets[w][e];
        store_return(a, status, member, eb, s);
    }
}

template <int EB, bool CART>
auto pick_kernel(bool fine) { return fine ? k_rollout_mlp_mma<EB, CART, true> : k_rollout_mlp_mma<EB, CART, false>; }

Plan make_plan(uint32_t task, uint32_t n_layers, const uint32_t* sizes, uint32_t EB)
{
    Plan p = {};
    const bool cart = task == EVO_TASK_CARTPOLE;
    uint32_t widest = 0, narrowest = n_layers > 1u ? ~0u : 0u;
    for (uint32_t l = 0; l < n_layers; ++l) {
        p.mt[l] = (sizes[l + 1] + 15u) / 16u;
        p.kt[l] = l == 0u ? 2u : (sizes[l] + 15u) / 16u;
        p.bias0[l] = p.biases;
        p.tile0[l] = p.tiles;
        if (!(cart && l == 0u)) { p.tiles += p.mt[l] * p.kt[l]; p.biases += p.mt[l] * 16u; }
        if (p.mt[l] > widest) widest = p.mt[l];
        if (l + 1u < n_layers && p.mt[l] < narrowest) narrowest = p.mt[l];
    }
    p.fine = narrowest < 4u;
    p.tile0[n_layers] = p.tiles;
    p.bias0[n_layers] = p.biases;
    p.mt[n_layers] = 2; p.kt[n_layers] = 3;
    if (!cart) { p.tiles += 6u; p.biases += 32u; if (widest < 2u) widest = 2u; }
    p.pitch = (widest + 1u) / 2u * 64u + 16u;           // operands are read two tiles at a time
    p.warps = widest < 8u ? widest : 8u;
    const uint32_t rows = EB == 4u ? 8u : 16u;
    p.smem = static_cast<size_t>(p.tiles) * 1024u + p.biases * 5u + (cart ? p.mt[0] * 512u : 0u) + 2u * rows * p.pitch +
             (cart ? 0u : 2u * rows * kXPitch + 32u);         // (the last column's third tile is read with the 32 bytes behind it)
    return p;
}

}  // namespace

// Episodes per block: 4, or 8 if a member has more (three MMAs then serve twice the episodes that two do; rollout_mlp_plan takes 4
// all the same for small populations).  0: the weights do not fit.
uint32_t rollout_mlp_mma_eb(uint32_t task, uint32_t n_layers, const uint32_t* sizes, uint32_t episodes)
{
    const uint32_t eb = episodes > 4u ? 8u : 4u;
    return make_plan(task, n_layers, sizes, eb).smem <= kMaxSmem ? eb : 0u;
}

// Blocks that an SM holds at once; 0: the weights do not fit, -1: the runtime's error
int rollout_mlp_mma_resident(uint32_t task, uint32_t n_layers, const uint32_t* sizes, uint32_t EB)
{
    const Plan p = make_plan(task, n_layers, sizes, EB);
    if (p.smem > kMaxSmem) return 0;
    const bool cart = task == EVO_TASK_CARTPOLE;
    auto kernel = EB == 4u ? (cart ? pick_kernel<4, true>(p.fine) : pick_kernel<4, false>(p.fine))
                           : (cart ? pick_kernel<8, true>(p.fine) : pick_kernel<8, false>(p.fine));
    static std::atomic<uint64_t> known[2][2][2];
    uint32_t regs;
    size_t fixed;
    if (!kernel_needs(kernel, known[EB == 8u][cart][p.fine], &regs, &fixed)) return -1;
    return static_cast<int>(resident_blocks(regs, p.smem + fixed, 32u * (p.warps + (cart ? 1u : 0u))));
}

int launch_rollout_mlp_mma(cudaStream_t st, const RolloutMlpArgs& a, DeviceStatus* status)
{
    const Plan p = make_plan(a.task, a.n_layers, a.sizes, a.EB);
    if (p.smem > kMaxSmem) return -2;
    const bool cart = a.task == EVO_TASK_CARTPOLE;
    auto kernel = a.EB == 4u ? (cart ? pick_kernel<4, true>(p.fine) : pick_kernel<4, false>(p.fine))
                             : (cart ? pick_kernel<8, true>(p.fine) : pick_kernel<8, false>(p.fine));
    if (!a.attr_done &&
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kMaxSmem)) != cudaSuccess)
        return -1;
    const uint32_t threads = 32u * (p.warps + (cart ? 1u : 0u));
    return launch_dependent(kernel, dim3(a.P, a.n_eb), dim3(threads), p.smem, st, a, p, status) == cudaSuccess ? 1 : -1;
}

}  // namespace evo
