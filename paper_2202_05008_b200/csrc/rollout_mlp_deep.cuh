// Control roll-outs of policies with one, three or four hidden layers of up to 192 units (and of two, one of them above 128), on warp-level
// tensor-core products (mma_split.cuh) with the weights in REGISTERS for all T steps: what k_rollout_mlp2 is for two hidden layers.
//
// Block = (member, EB episodes).  A warp owns 16 units of every layer: it keeps the operand tiles of the first layer, the hi parts of
// its rows of the matrices between hidden layers, and the action layer's columns of its own units in registers; the low parts of the
// matrices lie in shared memory, 16 bytes per lane and tile.  Activations cross warps through two buffers in turn, a
// barrier per layer; the action layer needs no pass of its own (a warp turns its last units into an operand, and partial sums meet).
//
// What bounds it: the serial chain of a step, HIDDEN + 1 barriers long, with as many members per SM as the registers hold
// (28-64-64-64-8, 4 episodes: 0.71 us a step with one member on an SM, 1.11 us with up to four).  k_rollout_mlp_mma, which
// reads the operands of every layer from shared memory in runtime loops, takes 1.69 and 2.21 us.  With the low parts in
// registers too the compiler has none left to work with: 0.86 and 1.19 us, and 4.1 against 2.9 us for 16 episodes of 512 members.
//
// Above 128 units (KT = 12) a block has up to twelve warps, and an SM to itself unless it has one hidden layer (72 to 92 registers a thread: two blocks
// of up to ten warps fit, of twelve for cart-pole and four episodes).  100 members, 4 episodes, us a step, with k_rollout_mlp_mma behind:
// 28-160-8 0.47 / 1.34, 5-190-180-1 1.15 / 3.00, 5-145-52-48-1 1.31 / 2.22, 28-150-60-60-60-8 1.51 / 2.60.
//
// The instances are compiled in two files, by the episodes of a block: 72 kernels, and the longest of all the sources in one (the library in 134 s, now 59).
//
// Paper: Section 2 (roll-out loop, central seeds), Section 4 (get_actions over the population with parameters as
// data; stateless task step; identical initial observations).
#pragma once
#include "internal.h"
#include "async.cuh"
#include "mma_split.cuh"
#include "noise.cuh"
#include "tasks.cuh"

#include <type_traits>

namespace evo {

using DeepKernel = void (*)(const RolloutMlpArgs, DeviceStatus*);
// size: 0 up to 64 units, 1 up to 128, 2 up to 192
DeepKernel rollout_mlp_deep_kernel4(bool cart, uint32_t hidden, uint32_t size, bool fine);
DeepKernel rollout_mlp_deep_kernel8(bool cart, uint32_t hidden, uint32_t size, bool fine);

namespace {

using namespace ms;

constexpr uint32_t kXPitch = 32 * 2 + 16;           // bytes per column of the state operand [x 28 | 0 4]
constexpr uint32_t kDynTiles = 6;                   // [A | B] in operand tiles: two of 16 rows x three of 16 inputs

// HIDDEN: hidden layers; KT: 16-unit tiles of the widest, 4, 8 or 12; FINE: see tanh_fine.
template <int EB, bool CART, int HIDDEN, int KT, bool FINE>
__global__ void __launch_bounds__(32 * KT, KT == 4 ? 4 : KT == 8 && HIDDEN <= 3 ? 2 : 1)
k_rollout_mlp_deep(const RolloutMlpArgs a, DeviceStatus* status)
{
    using U = Units<EB>;
    constexpr int NV = U::kValues, NH = NV / 2;                      // NH: values of one unit in a lane
    constexpr int NM = HIDDEN - 1, NS = NM > 0 ? NM : 1;             // matrices between hidden layers (and room for them)
    constexpr int RM = KT == 12 && NM > 2 ? 2 : NS;                  // of which the hi parts are in registers (48 a matrix and thread)
    constexpr Tanh kTanh = FINE ? Tanh::kFine : Tanh::kOwn;
    constexpr uint32_t kPitch = KT / 2 * 64 + 16;                    // bytes per column of a hidden operand (read two tiles at a time)
    constexpr uint32_t kHidBytes = U::kRows * kPitch;
    extern __shared__ __align__(16) uint4 lows[];                    // low parts of the matrices, [warp][matrix][tile][lane]; KT = 12: see below
    __shared__ uint32_t peak;
    __shared__ __align__(16) unsigned char hid[NM > 1 ? 2 : 1][kHidBytes];               // outputs of the hidden layers, in turn
    __shared__ __align__(16) float obs[CART ? 5 : 1][EB];            // cart-pole: observation
    __shared__ __align__(16) float part_c[CART ? KT : 1][8 * EB];    // ... shares of the action layer, [warp][g][episode]
    __shared__ __align__(16) unsigned char xop[CART ? 16 : 2 * U::kRows * kXPitch];      // tanh-linear: state, two buffers
    __shared__ __align__(16) float part_t[CART ? 1 : KT][CART ? 1 : 32 * NH];            // ... shares of the action layer
    __shared__ uint4 dyn[CART ? 1 : kDynTiles * 64];                 // ... task matrices in operand order
    __shared__ float x0s[CART ? 1 : kTlNx][EB];                      // ... start states
    __shared__ float rets[2][EB];
    __shared__ float ups[HIDDEN * 16 * KT + 8 + (CART ? 0 : 32)];    // scale_up of the units of the hidden layers, the actions, the states

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int nw = static_cast<int>(blockDim.x >> 5);
    const uint32_t member = blockIdx.x, eb = blockIdx.y, e0 = eb * EB;
    const int nE = min(static_cast<uint32_t>(EB), a.E - e0);
    const int nin = CART ? 5 : static_cast<int>(kTlNx), nout = CART ? 1 : static_cast<int>(kTlNa);
    int n[HIDDEN], mt[HIDDEN], at[NS];                               // units and tiles of the hidden layers; first parameter of the matrices
#pragma unroll
    for (int l = 0; l < HIDDEN; ++l) { n[l] = static_cast<int>(a.sizes[l + 1]); mt[l] = (n[l] + 15) >> 4; }
    const int nl = n[HIDDEN - 1];
    int w3_at = (nin + 1) * n[0];
#pragma unroll
    for (int m = 0; m < NM; ++m) { at[m] = w3_at; w3_at += (n[m] + 1) * n[m + 1]; }
    const uint32_t traced = a.trace ? a.trace_T : 0u;
    const PhiloxKey key = philox_key(a.k0, a.k1);
    const bool tw = warp < (CART ? 1 : 2);                           // these also step the task

    if (tid == 0) peak = 0u;
    for (uint32_t i = tid; i < sizeof(hid) / 4u; i += blockDim.x) reinterpret_cast<uint32_t*>(&hid[0][0])[i] = 0u;
    if (CART) for (uint32_t i = tid; i < sizeof(part_c) / 4u; i += blockDim.x) (&part_c[0][0])[i] = 0.f;
    else for (uint32_t i = tid; i < sizeof(part_t) / 4u; i += blockDim.x) (&part_t[0][0])[i] = 0.f;
    dep_wait();
    const uint32_t generation = status->generation;
    const float* row = a.theta + static_cast<size_t>(member) * a.ldD;
    __syncthreads();
    {
        // (of the parameters only: what a caller's matrix has in its padding columns is nobody's)
        uint32_t most = 0;
        const uint32_t n_params = static_cast<uint32_t>(w3_at + (nl + 1) * nout);
        for (uint32_t i = tid; i < n_params / 4u; i += blockDim.x) {
            const float4 w = __ldg(reinterpret_cast<const float4*>(row) + i);
            most = max(max(most, max(magnitude(w.x), magnitude(w.y))), max(magnitude(w.z), magnitude(w.w)));
        }
        if (tid < static_cast<int>(n_params & 3u)) most = max(most, magnitude(row[(n_params & ~3u) + tid]));
        most = __reduce_max_sync(0xffffffffu, most);
        if (lane == 0) atomicMax(&peak, most);
        __syncthreads();
    }
    const int most = scale_exponent(peak);
    const bool scaled = most != 0 || (!CART && scales_dynamics(a.action_scale));

    // ---- weights into registers, times f (see mma_split.cuh) ---------------------------------------
    const float* W1 = row;
    const float* B1 = W1 + n[0] * nin;
    const float* W3 = row + w3_at;
    const float* B3 = W3 + nout * nl;
    const int u0 = 16 * warp + g, u1 = u0 + 8;                       // this lane's two units of every layer
    uint4 wh[RM][KT];
    uint4 w1h[2], w1l[2], w3 = make_uint4(0u, 0u, 0u, 0u);           // w3: the action layer's own inputs (see Units::eight)
    float w1c[10], w3c[2], bias[HIDDEN][2], b3;
    float* const ups1 = ups + u0, *const ups3 = ups + HIDDEN * 16 * KT + g;              // ups1: + 16 KT per layer
    // KT = 12: [matrix][warp][tile][lane], only what the layers have, tiles in fours; behind them the hi parts of a matrix that are not in registers
    uint4* wl[NS];
    uint4* whs = nullptr;
    {
        uint4* to = lows + (KT == 12 ? 0 : warp * (NM * KT * 32)) + lane;
#pragma unroll
        for (int m = 0; m < NS; ++m) {
            if constexpr (KT == 12) {
                const int tiles = m < NM ? (mt[m] + 3) & ~3 : 0, rows = m < NM ? mt[m + 1 < HIDDEN ? m + 1 : m] : 0;
                wl[m] = to + 32 * warp * tiles;
                to += 32 * rows * tiles;
                if (m >= RM) { whs = to + 32 * warp * tiles; to += 32 * rows * tiles; }
            } else {
                wl[m] = to + 32 * m * KT;
            }
        }
    }
    bias[0][0] = u0 < n[0] ? times_f(B1[u0]) : 0.f; bias[0][1] = u1 < n[0] ? times_f(B1[u1]) : 0.f;
    if constexpr (CART) {                                            // the observation is taken as it is, in fp32
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            w1c[k] = u0 < n[0] ? times_f(W1[u0 * 5 + k]) : 0.f;
            w1c[5 + k] = u1 < n[0] ? times_f(W1[u1 * 5 + k]) : 0.f;
        }
        w3c[0] = u0 < nl ? kF * kActInv * W3[u0] : 0.f; w3c[1] = u1 < nl ? kF * kActInv * W3[u1] : 0.f;
        b3 = times_f(B3[0]);
    } else {
        int s0 = 0, s1 = 0, s3 = 0, none;
        if (scaled) {
            row_exponents(W1, nin, n[0], 16 * warp, 2, lane, s0, s1);
            row_exponents(W3, nl, nout, 0, mt[HIDDEN - 1], lane, s3, none);
            ups1[0] = scale_up(s0); ups1[8] = scale_up(s1); ups3[0] = scale_up(s3);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) load_tile(W1, nin, n[0], 16 * warp, 16 * k, lane, s0, s1, w1h[k], w1l[k]);
        uint4 lo3;
        load_tile(W3, nl, nout, 0, 16 * warp, lane, s3, 0, w3, lo3);
        w3.y = lo3.x; w3.w = lo3.z;
        b3 = times_f(B3[g]);
        for (int i = warp; i < static_cast<int>(kDynTiles); i += nw) {
            uint4 hi, lo;
            load_dynamics(a.task_const, a.action_scale, i, lane, scaled, s0, s1, hi, lo);
            if (scaled) { ups3[8 + 16 * (i / 3)] = scale_up(s0); ups3[16 + 16 * (i / 3)] = scale_up(s1); }
            dyn[i * 64 + lane] = hi;
            dyn[i * 64 + 32 + lane] = lo;
        }
    }
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        const float* W = row + at[m];
        const float* B = W + n[m + 1] * n[m];
        const bool pairs = ((n[m] | at[m]) & 1) == 0;                // rows can be read two weights at a time
        bias[m + 1][0] = u0 < n[m + 1] ? times_f(B[u0]) : 0.f; bias[m + 1][1] = u1 < n[m + 1] ? times_f(B[u1]) : 0.f;
        int s0 = 0, s1 = 0;
        if (scaled) {
            row_exponents(W, n[m], n[m + 1], 16 * warp, KT, lane, s0, s1);
            ups1[16 * KT * (m + 1)] = scale_up(s0); ups1[16 * KT * (m + 1) + 8] = scale_up(s1);
        }
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            uint4 hi, lo;
            load_tile(W, n[m], n[m + 1], 16 * warp, 16 * k, lane, s0, s1, hi, lo, pairs);
            if (m < RM) wh[m < RM ? m : 0][k] = hi;
            if (KT < 12 || (warp < mt[m + 1] && k < ((mt[m] + 3) & ~3))) {
                wl[m][32 * k] = lo;
                if (m >= RM) whs[32 * k] = hi;
            }
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
    const uint32_t hid_row = U::row(smem_u32(hid), kPitch, lane);
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
    const float up = scale_up(most);                                 // kActInv where nothing is scaled, in a register
    auto roll = [&](auto with_scales) {
        constexpr bool kScaled = decltype(with_scales)::value;
        for (uint32_t step = 0; step < a.T; ++step) {
            CpAhead ahead;
            auto meanwhile = [&] {                                       // what a step can do before it needs the action
                if constexpr (!CART) {                                   // reward on the pre-step state (0 in other warps, padding rows)
#pragma unroll
                    for (int i = 0; i < NV; ++i) {
                        if (EB == 4 || !(i & 1)) ret = fmaf(-xcur[i], xcur[i], ret); else ret2 = fmaf(-xcur[i], xcur[i], ret2);
                    }
                } else if (tw) {
                    ahead = cartpole_ahead(cpc, cps, snc, csc);
                    if (step > 0u) ret = fmaf(csc, __expf(-cps.x * cps.x), ret);        // reward of the step before, on its post-step state
                }
            };
            auto action_share = [&](const float (&v)[NV]) {              // of the warp's units of the last hidden layer
                if constexpr (CART) {
                    float p[NH];
#pragma unroll
                    for (int i = 0; i < NH; ++i) p[i] = fmaf(w3c[1], v[NH + i], w3c[0] * v[i]);
                    if constexpr (EB == 4) part_c[warp][lane] = p[0];
                    else *reinterpret_cast<float2*>(&part_c[warp][2 * lane]) = make_float2(p[0], p[1]);
                } else {
                    uint32_t b[4];
                    float p[2];
                    U::transpose(v, b);
                    U::eight(w3, b, kScaled ? ups3[0] : up, 0.f, p);
                    if constexpr (EB == 4) part_t[warp][lane] = p[0];
                    else *reinterpret_cast<float2*>(&part_t[warp][2 * lane]) = make_float2(p[0], p[1]);
                }
            };
            if (warp < mt[0]) {
                float v[NV];
                if constexpr (CART) {
                    float o[5][NH];
#pragma unroll
                    for (int k = 0; k < 5; ++k) {
                        if constexpr (EB == 4) o[k][0] = obs[k][t];
                        else { const float2 q = *reinterpret_cast<const float2*>(&obs[k][2 * t]); o[k][0] = q.x; o[k][1] = q.y; }
                    }
#pragma unroll
                    for (int i = 0; i < NV; ++i) {
                        float s = bias[0][i / NH];
#pragma unroll
                        for (int k = 0; k < 5; ++k) s = fmaf(w1c[5 * (i / NH) + k], o[k][i % NH], s);
                        v[i] = s;
                    }
                } else {
                    U acc;
                    uint32_t b[2][4];
                    U::load(xin, b);
                    if (U::kLoadTiles == 1) U::load(xin + 32u, b + 1);
                    acc.first(w1h[0], w1l[0], b[0]);
                    acc.add(w1h[1], w1l[1], b[1]);
                    acc.sums(kScaled ? ups1[0] : up, kScaled ? ups1[8] : up, bias[0][0], bias[0][1], v);
                }
                tanh_units<EB, kTanh>(v);
                if constexpr (NM > 0) U::store(hid_row + 32u * warp, v);
                else action_share(v);
            }
            if (NM == 0) meanwhile();
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                __syncthreads();
                const uint32_t in = hid_row + (m & 1) * kHidBytes, out = hid_row + ((m + 1) & 1) * kHidBytes;
                U acc;
                if (warp < mt[m + 1]) {
                    uint32_t b[2][2][4];                                 // the operands of two tiles, those of the next two on their way
                    U::load(in, b[0]);
                    if (U::kLoadTiles == 1) U::load(in + 32u, b[0] + 1);
                    auto products = [&](int k) {
                        uint32_t (&now)[2][4] = b[(k >> 1) & 1], (&next)[2][4] = b[((k >> 1) + 1) & 1];
                        if (!(k & 1) && k + 2 < KT) {
                            U::load(in + 32u * k + 64u, next);
                            if (U::kLoadTiles == 1) U::load(in + 32u * k + 96u, next + 1);
                        }
                        const uint4 lo = wl[m][32 * k], hi = m < RM ? wh[m < RM ? m : 0][k] : whs[32 * k];
                        if (k == 0) acc.first(hi, lo, now[0]);
                        else acc.add(hi, lo, now[k & 1]);
                    };
#pragma unroll
                    for (int k = 0; k < 4; ++k) products(k);
                    if (KT > 4 && mt[m] > 4) {                           // (not behind a narrow layer of a wide policy)
#pragma unroll
                        for (int k = 4; k < (KT < 8 ? KT : 8); ++k) products(k);
                        if (KT > 8 && mt[m] > 8) {
#pragma unroll
                            for (int k = 8; k < KT; ++k) products(k);
                        }
                    }
                }
                if (m == 0) meanwhile();
                if (warp < mt[m + 1]) {
                    float v[NV];
                    const float* s = ups1 + 16 * KT * (m + 1);
                    acc.sums(kScaled ? s[0] : up, kScaled ? s[8] : up, bias[m + 1][0], bias[m + 1][1], v);
                    tanh_units<EB, kTanh>(v);
                    if (m + 1 < NM) U::store(out + 32u * warp, v);
                    else action_share(v);
                }
            }
            __syncthreads();
            if constexpr (CART) {
                if (tw) {
                    // the shares of episode te, [warp][g]: this lane adds a quarter (an eighth) of them
                    float p[EB];
#pragma unroll
                    for (int i = 0; i < EB; ++i) p[i] = (&part_c[0][0])[lane + 32 * i];
#pragma unroll
                    for (int w = 4; w < KT; w += 4)
#pragma unroll
                        for (int i = 0; i < EB; ++i) p[i] += (&part_c[w][0])[lane + 32 * i];
#pragma unroll
                    for (int k = EB / 2; k > 0; k >>= 1)
#pragma unroll
                        for (int i = 0; i < k; ++i) p[i] += p[i + k];
                    float pre = p[0];
#pragma unroll
                    for (int off = EB; off < 32; off <<= 1) pre += __shfl_xor_sync(0xffffffffu, pre, off);
                    const float force = a.action_scale * kActInv * (FINE ? tanh_fine(pre + b3) : tanh_one(pre + b3));
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
#pragma unroll
                    for (int more = 4; more < KT; more += 4) {
                        if constexpr (EB == 4) p[w][0] += part_t[more + w][lane];
                        else { const float2 q = *reinterpret_cast<const float2*>(&part_t[more + w][2 * lane]); p[w][0] += q.x; p[w][1] += q.y; }
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
                for (int i = 0; i < NH; ++i) {
                    v[i] = ((p[0][i] + p[1][i]) + (p[2][i] + p[3][i])) + b3;
                    v[i] = FINE ? tanh_fine(v[i]) : tanh_one(v[i]);
                }
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

template <int EB, bool CART, int HIDDEN>
DeepKernel pick_size(uint32_t size, bool fine)
{
    if constexpr (HIDDEN == 1) {                                     // (one hidden layer above 64 units is not FINE)
        if (size > 0u) return size == 2u ? k_rollout_mlp_deep<EB, CART, 1, 12, false> : k_rollout_mlp_deep<EB, CART, 1, 8, false>;
    } else {
        if (size == 2u) return fine ? k_rollout_mlp_deep<EB, CART, HIDDEN, 12, true> : k_rollout_mlp_deep<EB, CART, HIDDEN, 12, false>;
    }
    if constexpr (HIDDEN == 2) return nullptr;                       // (k_rollout_mlp2)
    else {
        if constexpr (HIDDEN > 1)
            if (size == 1u) return fine ? k_rollout_mlp_deep<EB, CART, HIDDEN, 8, true> : k_rollout_mlp_deep<EB, CART, HIDDEN, 8, false>;
        return fine ? k_rollout_mlp_deep<EB, CART, HIDDEN, 4, true> : k_rollout_mlp_deep<EB, CART, HIDDEN, 4, false>;
    }
}
template <int EB, bool CART>
DeepKernel pick_kernel(uint32_t hidden, uint32_t size, bool fine)
{
    switch (hidden) {
        case 1u: return pick_size<EB, CART, 1>(size, fine);
        case 2u: return pick_size<EB, CART, 2>(size, fine);
        case 3u: return pick_size<EB, CART, 3>(size, fine);
        default: return pick_size<EB, CART, 4>(size, fine);
    }
}

}  // namespace
}  // namespace evo
