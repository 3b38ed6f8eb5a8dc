// Solver kernels: ask (antithetic sampling), centred rank, ES gradient (stored or regenerated
// noise) and the Adam ascent step.  Paper Section 4 (NEAlgorithm ask / tell), Section 2
// ("Modern ML Optimizers"); the algorithm is PGPE with symmetric sampling (Section 5).
#include "internal.h"
#include "noise.cuh"

#include <type_traits>

namespace evo {

// ------------------------------------------------------------------------------------------
// init / task constants
// ------------------------------------------------------------------------------------------
__global__ void k_init(uint32_t* counters, uint32_t n_counters, float* center, float* m, float* v, float* g, float* sigma_vec, float sigma,
                       uint32_t D, uint32_t ldD, DeviceStatus* status, uint32_t wait_cycles_log2,
                       uint32_t debug_flags)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < ldD) { center[i] = 0.f; m[i] = 0.f; v[i] = 0.f; g[i] = 0.f; sigma_vec[i] = (i < D) ? sigma : 0.f; }
    if (i < n_counters) counters[i] = 0u;
    if (i == 0) {
        status->sticky = 0; status->nonfinite = 0; status->adam_step = 0; status->generation = 0;
        status->wait_cycles_log2 = wait_cycles_log2; status->debug_flags = debug_flags;
        status->bounds_site = 0; status->bounds_index_lo = 0; status->bounds_index_hi = 0; status->reserved = 0;
    }
}

int launch_init(cudaStream_t st, uint32_t* counters, float* center, float* m, float* v, float* g, float* sigma_vec,
                float sigma, uint32_t D, uint32_t ldD, DeviceStatus* status, uint32_t wait_cycles_log2,
                uint32_t debug_flags)
{
    k_init<<<(ldD + 255) / 256, 256, 0, st>>>(counters, static_cast<uint32_t>(tell_counter_words(ldD)), center, m, v, g, sigma_vec, sigma, D, ldD, status,
                                              wait_cycles_log2, debug_flags);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

// Tanh-linear task constants: A[28][28] = z * fp32(0.9/sqrt(28)), B[28][8] = z * fp32(1/sqrt(8)),
// z from stream 4 (row 0 = A, row 1 = B), generation 0.
__global__ void k_tanh_linear_constants(PhiloxKey key, float* out)
{
    const uint32_t quad = threadIdx.x;
    constexpr uint32_t qa = kTlNx * kTlNx / 4, qb = kTlNx * kTlNa / 4;
    if (quad < qa) {
        const float4 z = stream_normal4(key, 4u, 0u, 0u, quad);
        const float sc = __uint_as_float(0x3E2E2A81u);
        float4 r = make_float4(__fmul_rn(z.x, sc), __fmul_rn(z.y, sc), __fmul_rn(z.z, sc), __fmul_rn(z.w, sc));
        reinterpret_cast<float4*>(out)[quad] = r;
    } else if (quad < qa + qb) {
        const float4 z = stream_normal4(key, 4u, 0u, 1u, quad - qa);
        const float sc = __uint_as_float(0x3EB504F3u);
        float4 r = make_float4(__fmul_rn(z.x, sc), __fmul_rn(z.y, sc), __fmul_rn(z.z, sc), __fmul_rn(z.w, sc));
        reinterpret_cast<float4*>(out)[quad] = r;
    }
}

int launch_task_constants(cudaStream_t st, uint32_t task, uint32_t k0, uint32_t k1, float* task_const)
{
    if (task != EVO_TASK_TANH_LINEAR) return 0;
    k_tanh_linear_constants<<<1, 256, 0, st>>>(philox_key(k0, k1), task_const);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

// ------------------------------------------------------------------------------------------
// ask: one thread per (column quad, chunk of pairs).  Writes are 128-bit and coalesced along
// the row; the centre quad is loaded once per thread and reused for all pairs of the chunk.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256, 4)
k_ask(const float* __restrict__ center, const float* __restrict__ sigma_vec, PhiloxKey key,
      const DeviceStatus* __restrict__ status, uint32_t pair0, uint32_t H, uint32_t D, uint32_t ldD, uint32_t pairs_per_thread,
      float* __restrict__ theta, float* __restrict__ eps)
{
    dep_wait();
    dep_trigger();                       // the roll-out that follows may be set up
    const uint32_t quad = blockIdx.x * blockDim.x + threadIdx.x;
    if (quad * 4u >= ldD) return;
    const uint32_t generation = status->generation;
    const uint32_t d0 = quad * 4u;
    const float4 c = reinterpret_cast<const float4*>(center)[quad];
    const float4 sg = reinterpret_cast<const float4*>(sigma_vec)[quad];      // one sigma per dimension
    const bool full = d0 + 4u <= D;
    const PhiloxItem item = philox_item(quad, generation, 0u, key);
    const fp2 c2[2] = { fp2_make(c.x, c.y), fp2_make(c.z, c.w) }, s2[2] = { fp2_make(sg.x, sg.y), fp2_make(sg.z, sg.w) };
    const fp2 n2[2] = { fp2_make(-sg.x, -sg.y), fp2_make(-sg.z, -sg.w) };
    for (uint32_t j = blockIdx.y * pairs_per_thread; j < H; j += gridDim.y * pairs_per_thread) {
        const uint32_t jend = min(j + pairs_per_thread, H);
        for (uint32_t jj = j; jj < jend; ++jj) {
            float4 z = normal4(philox4x32_10(item, pair0 + jj, key));         // counters use the global pair
            if (!full) {                       // ragged tail and padding columns carry zeros
                if (d0 + 0u >= D) z.x = 0.f;
                if (d0 + 1u >= D) z.y = 0.f;
                if (d0 + 2u >= D) z.z = 0.f;
                if (d0 + 3u >= D) z.w = 0.f;
            }
            const fp2 z2[2] = { fp2_make(z.x, z.y), fp2_make(z.z, z.w) };
            float4 tp, tm;
            fp2_split(fp2_fma(s2[0], z2[0], c2[0]), tp.x, tp.y); fp2_split(fp2_fma(s2[1], z2[1], c2[1]), tp.z, tp.w);
            fp2_split(fp2_fma(n2[0], z2[0], c2[0]), tm.x, tm.y); fp2_split(fp2_fma(n2[1], z2[1], c2[1]), tm.z, tm.w);
            float* row = theta + static_cast<size_t>(2u * jj) * ldD + d0;
            if (EVO_IN_BOUNDS(status, EVO_SITE_ASK_THETA, static_cast<size_t>(2u * jj + 1u) * ldD + d0 + 3u,
                              static_cast<size_t>(2u * H) * ldD)) {
                __stcs(reinterpret_cast<float4*>(row), tp);
                __stcs(reinterpret_cast<float4*>(row + ldD), tm);
            }
            if (eps && EVO_IN_BOUNDS(status, EVO_SITE_ASK_EPS, static_cast<size_t>(jj) * ldD + d0 + 3u,
                                     static_cast<size_t>(H) * ldD))
                __stcs(reinterpret_cast<float4*>(eps + static_cast<size_t>(jj) * ldD + d0), z);
        }
    }
}

int launch_ask(cudaStream_t st, const float* center, const float* sigma_vec, uint32_t k0, uint32_t k1,
               const DeviceStatus* status, uint32_t pair0, uint32_t H, uint32_t D, uint32_t ldD, float* theta,
               float* eps)
{
    const uint32_t quads = ldD / 4u;
    // Eight pairs per thread reuse the centre; a small problem is one wave whose length is what a thread does, so it takes fewer.
    const uint32_t bx = (quads + 255u) / 256u;
    uint32_t ppt = 8u;
    while (ppt > 1u && static_cast<uint64_t>(bx) * ((H + ppt - 1u) / ppt) < kSms * 6u) ppt /= 2u;
    dim3 grid(bx, (H + ppt - 1u) / ppt);
    if (grid.y > 65535u) grid.y = 65535u;
    return launch_dependent(k_ask, grid, dim3(256), 0, st, center, sigma_vec, philox_key(k0, k1), status, pair0, H, D, ldD,
                            ppt, theta, eps) == cudaSuccess ? 1 : -1;
}

// ------------------------------------------------------------------------------------------
// centred rank by counting: rank_m = #{k : f_k < f_m or (f_k == f_m and k < m)}
//
// Fitness values become keys whose unsigned order is that of the floats (-0 taken as +0), so that against a run of
// entries that lies wholly on one side of m the whole rule is one comparison, key_k < key_m + (run before m).  A warp
// ranks M members at once: its lanes hold different entries, an entry is loaded once for all M.
// ------------------------------------------------------------------------------------------
// Keys in shared memory at a time.  Few, because the tell kernel's first blocks come to an SM while ranking ends there and find
// the split of shared memory and L1 as it is: with 8,192 keys too little L1 is left for their loads in flight
// (131,072 columns x 16,384 members: tell 848 us instead of 733).
constexpr uint32_t kRankTile = 4096;
constexpr uint32_t kRankRun = 128;               // entries per warp step: four per lane

__device__ __forceinline__ uint32_t rank_key(float f)
{
    const uint32_t b = __float_as_uint(__fadd_rn(f, 0.0f));
    return b ^ (static_cast<uint32_t>(static_cast<int32_t>(b) >> 31) | 0x80000000u);
}

// adds the entries [first, first + n) of the population, whose keys lie at `keys` (padded to whole runs with ~0), to below[]
template <int M>
__device__ __forceinline__ void count_below(const uint32_t* keys, uint32_t first, uint32_t n, uint32_t m0, const uint32_t (&key)[M],
                                            uint32_t (&below)[M], uint32_t lane)
{
    for (uint32_t i = 0; i < n; i += kRankRun) {
        const uint4 k = *reinterpret_cast<const uint4*>(keys + i + 4u * lane);
        const uint32_t at = first + i;
        if (at + kRankRun <= m0 || at >= m0 + M) {
            const uint32_t before = at < m0 ? 1u : 0u;
#pragma unroll
            for (int j = 0; j < M; ++j) {
                const uint32_t t = key[j] + before;
                below[j] += (k.x < t ? 1u : 0u) + (k.y < t ? 1u : 0u) + (k.z < t ? 1u : 0u) + (k.w < t ? 1u : 0u);
            }
        } else {
            const uint32_t kk[4] = { k.x, k.y, k.z, k.w };
#pragma unroll
            for (int j = 0; j < M; ++j)
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    below[j] += (kk[c] < key[j] || (kk[c] == key[j] && at + 4u * lane + c < m0 + j)) ? 1u : 0u;
        }
    }
}

__device__ __forceinline__ float centred_rank(uint32_t below, uint32_t P)
{
    return __fadd_rn(__fdiv_rn(__uint2float_rn(below), __uint2float_rn(P - 1u)), -0.5f);
}

template <int M>
__global__ void __launch_bounds__(256)
k_rank(const float* __restrict__ fitness, uint32_t P, int32_t* __restrict__ rank, float* __restrict__ u, DeviceStatus* status)
{
    __shared__ __align__(16) uint32_t keys[kRankTile];
    dep_wait();
    dep_trigger();
    const uint32_t lane = threadIdx.x & 31u, m0 = (blockIdx.x * 8u + (threadIdx.x >> 5)) * M;
    uint32_t key[M], below[M];
#pragma unroll
    for (int j = 0; j < M; ++j) {
        const float f = m0 + j < P ? fitness[m0 + j] : 0.f;
        if (lane == 0 && f != f) atomicOr(&status->nonfinite, 1u);
        key[j] = rank_key(f);
        below[j] = 0u;
    }
    for (uint32_t base = 0; base < P; base += kRankTile) {
        const uint32_t n = min(kRankTile, P - base), padded = (n + kRankRun - 1u) / kRankRun * kRankRun;
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < padded; i += blockDim.x) keys[i] = i < n ? rank_key(fitness[base + i]) : 0xFFFFFFFFu;
        __syncthreads();
        if (m0 < P) count_below<M>(keys, base, n, m0, key, below, lane);
    }
#pragma unroll
    for (int j = 0; j < M; ++j) {
        const uint32_t r = __reduce_add_sync(0xffffffffu, below[j]);
        if (lane == 0 && m0 + j < P && EVO_IN_BOUNDS(status, EVO_SITE_RANK, m0 + j, P)) {
            rank[m0 + j] = static_cast<int32_t>(r);
            u[m0 + j] = centred_rank(r, P);
        }
    }
}

int launch_rank(cudaStream_t st, const float* fitness, uint32_t P, int32_t* rank, float* u,
                DeviceStatus* status)
{
    // About 128 blocks of eight warps up to P = 4,096, where the kernel is a matter of latency (P = 1,024: 5 us against 17 for
    // one thread per member); from there on four members per warp, bound by the comparisons (P = 16,384: 64 us; one
    // thread per member, split over blocks with atomics: 88; eight members per warp: 66).
    const uint32_t m = P <= 1024u ? 1u : P <= 2048u ? 2u : 4u;
    auto kernel = m == 1u ? k_rank<1> : m == 2u ? k_rank<2> : k_rank<4>;
    return launch_dependent(kernel, dim3((P + 8u * m - 1u) / (8u * m)), dim3(256), 0, st, fitness, P, rank, u, status) == cudaSuccess
               ? 1 : -1;
}

// ------------------------------------------------------------------------------------------
// tell: ES gradient and optimiser step in one kernel.
//
// Block = (64 column quads) x (a split of the pairs); its 256 threads are 64 quads x 4 pair lanes, so even a few hundred
// columns keep a few blocks' worth of loads in flight (256 quads x 1 lane where the columns are many: 643 us against 621 at
// 131,072 columns, 8,192 pairs).  Stored noise wants five blocks per SM: 64 bytes per thread in flight (four blocks: 745
// against 733 us with the ranking).  Products and sums are fp64: the Adam step lr*g/(|g|+eps) is
// ill-conditioned where |g| is near adam_eps, so the cancellation error of an fp32 sum (~1e-7 of RMS(g)) would
// move those coordinates by far more than the 1e-5 parity bound.  The stored-noise form is HBM-bound (4 bytes
// per term; 4.3 GB in 621 us), so the fp64 arithmetic is hidden.  REGEN recomputes eps from the Philox counters instead of
// reading it.  SIGMA also accumulates the PGPE sigma gradient sum_j ((u[2j]+u[2j+1])/2) (eps^2 - 1), whose partial sums are fp32 (a plain
// step on sigma follows, which is not ill-conditioned like Adam's normalised step).
//
// The block that finds itself the last of its columns (a counter, no waiting) adds the splits' partial sums and takes the step
// for them; the last of those closes the tell.  RANK: each block also ranks the members of its own pairs.  A tell of a
// small problem is then one launch where it was four (rank, gradient, update, close): a matter of launches
// and of memory round trips between them (generation of the CNN, 64 members: 106 -> 98 us).
// All summation orders are fixed; no floating-point atomics anywhere, so results are run-to-run identical.
// ------------------------------------------------------------------------------------------
constexpr uint32_t kTellQuads = 64, kTellLanes = 4;
constexpr int kGradRows = 4;           // noise rows in flight per thread
constexpr uint32_t kRankInTell = 2048; // largest population ranked inside k_tell
constexpr uint32_t kTellPairs = 256;   // ... and most pairs of a split then

struct Acc4 { double x, y, z, w; };

__device__ __forceinline__ void acc_fma(Acc4& a, double wd, const float4& e)
{
    a.x = fma(wd, static_cast<double>(e.x), a.x);
    a.y = fma(wd, static_cast<double>(e.y), a.y);
    a.z = fma(wd, static_cast<double>(e.z), a.z);
    a.w = fma(wd, static_cast<double>(e.w), a.w);
}
// A thread's sums of the sigma gradient.  Stored noise streams and leaves the fp64 pipe time: sums in fp64, one rounding when they leave the thread.
// In fp32 their error grew with the pairs of a split, of which there are fewer than room for (see whole_waves): relative RMS
// error of the gradient with all splits / with these / these in fp64, 300 members x 40,256 columns 7.8 / 8.4 / 5.2e-8, 4,096 x 20,872 10.2 / 14.6 /
// 6.4e-8, 16,384 x 131,072 21 / 25 / 6.6e-8.
struct SigmaSums64 {
    Acc4 a = { 0., 0., 0., 0. };
    __device__ __forceinline__ static void term(double& s, double w, float e) { const double z = e; s = fma(w, fma(z, z, -1.0), s); }
    __device__ __forceinline__ void add(int, const float2& uu, const float4& e)
    {
        const double d = 0.5 * (static_cast<double>(uu.x) + static_cast<double>(uu.y));
        term(a.x, d, e.x); term(a.y, d, e.y); term(a.z, d, e.z); term(a.w, d, e.w);
    }
    __device__ __forceinline__ void sums(float (&r)[4]) const
    {
        r[0] = static_cast<float>(a.x); r[1] = static_cast<float>(a.y); r[2] = static_cast<float>(a.z); r[3] = static_cast<float>(a.w);
    }
};
// Recomputed noise is bound by issue: packed fp32, two chains.
struct SigmaSums32 {
    fp2 a[2][2] = { { 0ull, 0ull }, { 0ull, 0ull } };
    __device__ __forceinline__ void add(int i, const float2& uu, const float4& e)
    {
        const fp2 s = fp2_both(0.5f * (uu.x + uu.y)), z[2] = { fp2_make(e.x, e.y), fp2_make(e.z, e.w) };
#pragma unroll
        for (int k = 0; k < 2; ++k) a[i & 1][k] = fp2_fma(s, fp2_fma(z[k], z[k], fp2_both(-1.0f)), a[i & 1][k]);
    }
    __device__ __forceinline__ void sums(float (&r)[4]) const
    {
        fp2_split(fp2_add(a[0][0], a[1][0]), r[0], r[1]);
        fp2_split(fp2_add(a[0][1], a[1][1]), r[2], r[3]);
    }
};

__device__ __forceinline__ double power(double b, uint32_t n)
{
    double r = 1.0;
    for (; n; n >>= 1, b *= b)
        if (n & 1u) r *= b;
    return r;
}

enum : uint32_t { kStepAdam = 0, kStepClipup = 1, kStepSums = 2 };

struct StepArgs {
    uint32_t mode, ldD;
    double inv_pop;
    float lr, beta1, beta2, adam_eps, momentum, max_speed, sigma_lr, sigma_max_change, inv_pairs;
    float *sigma_vec, *center, *m, *v, *g;
    double* grad_sum; float* sigma_sum;      // kStepSums: where the sums go
    double* norms;                           // ClipUp: per column block |v|^2, v.g, |g|^2; then the two factors of the step and whether to take it
    DeviceStatus* status;
};

// What a step reads of a column quad.
struct QuadState { float4 sigma, m, center, v; };
__device__ __forceinline__ QuadState load_quad(const StepArgs& a, uint32_t quad)
{
    QuadState q;
    q.sigma = reinterpret_cast<const float4*>(a.sigma_vec)[quad];
    q.m = reinterpret_cast<const float4*>(a.m)[quad];
    q.center = q.v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a.mode == kStepAdam) {
        q.center = reinterpret_cast<const float4*>(a.center)[quad];
        q.v = reinterpret_cast<const float4*>(a.v)[quad];
    }
    return q;
}

// One column quad's step from its summed gradient (fp64, unscaled) and sigma gradient.
__device__ __forceinline__ void quad_step(const StepArgs& a, uint32_t quad, const double (&sum)[4], const float (&ss)[4], bool sigma,
                                          const QuadState& q, float corr1, float corr2, double (&dots)[3])
{
    if (a.mode == kStepSums) {
        double2* out = reinterpret_cast<double2*>(a.grad_sum) + 2u * quad;
        out[0] = make_double2(sum[0], sum[1]);
        out[1] = make_double2(sum[2], sum[3]);
        if (sigma) reinterpret_cast<float4*>(a.sigma_sum)[quad] = make_float4(ss[0], ss[1], ss[2], ss[3]);
        return;
    }
    float sg[4] = { q.sigma.x, q.sigma.y, q.sigma.z, q.sigma.w }, gg[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) gg[i] = static_cast<float>(sum[i] * (static_cast<double>(sg[i]) * a.inv_pop));
    reinterpret_cast<float4*>(a.g)[quad] = make_float4(gg[0], gg[1], gg[2], gg[3]);
    float mm[4] = { q.m.x, q.m.y, q.m.z, q.m.w };
    if (a.mode == kStepAdam) {
        float cc[4] = { q.center.x, q.center.y, q.center.z, q.center.w }, vv[4] = { q.v.x, q.v.y, q.v.z, q.v.w };
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            mm[i] = a.beta1 * mm[i] + (1.f - a.beta1) * gg[i];
            vv[i] = a.beta2 * vv[i] + (1.f - a.beta2) * gg[i] * gg[i];
            const float mhat = mm[i] * corr1;
            const float vhat = vv[i] * corr2;
            cc[i] += a.lr * mhat / (sqrtf(vhat) + a.adam_eps);
        }
        reinterpret_cast<float4*>(a.m)[quad] = make_float4(mm[0], mm[1], mm[2], mm[3]);
        reinterpret_cast<float4*>(a.v)[quad] = make_float4(vv[0], vv[1], vv[2], vv[3]);
        if (EVO_IN_BOUNDS(a.status, EVO_SITE_UPDATE, 4u * quad + 3u, a.ldD))
            reinterpret_cast<float4*>(a.center)[quad] = make_float4(cc[0], cc[1], cc[2], cc[3]);
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            dots[0] += static_cast<double>(mm[i]) * mm[i];
            dots[1] += static_cast<double>(mm[i]) * gg[i];
            dots[2] += static_cast<double>(gg[i]) * gg[i];
        }
    }
    if (sigma) {                             // PGPE sigma step with a relative-change limit
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float gs = sg[i] * a.inv_pairs * ss[i];
            const float lo = sg[i] * (1.f - a.sigma_max_change), hi = sg[i] * (1.f + a.sigma_max_change);
            sg[i] = fminf(fmaxf(sg[i] + a.sigma_lr * gs, lo), hi);
        }
        reinterpret_cast<float4*>(a.sigma_vec)[quad] = make_float4(sg[0], sg[1], sg[2], sg[3]);
    }
}

// ClipUp: vel = momentum vel + (lr / |g|) g, scaled back if it is longer than max_speed; center += vel.  The length follows
// from the three dot products, so one pass is enough.  factor = lr / |g|, scale = the clip.
__device__ __forceinline__ void clipup_quad(const StepArgs& a, uint32_t quad, float factor, float scale)
{
    const float4 g4 = reinterpret_cast<const float4*>(a.g)[quad];
    float4 v4 = reinterpret_cast<const float4*>(a.m)[quad], c4 = reinterpret_cast<const float4*>(a.center)[quad];
    v4.x = scale * fmaf(a.momentum, v4.x, factor * g4.x); v4.y = scale * fmaf(a.momentum, v4.y, factor * g4.y);
    v4.z = scale * fmaf(a.momentum, v4.z, factor * g4.z); v4.w = scale * fmaf(a.momentum, v4.w, factor * g4.w);
    c4.x += v4.x; c4.y += v4.y; c4.z += v4.z; c4.w += v4.w;
    reinterpret_cast<float4*>(a.m)[quad] = v4;
    reinterpret_cast<float4*>(a.center)[quad] = c4;
}

// fixed-order sum over the block of three values per thread; every thread gets them
__device__ __forceinline__ void block_dots(double (&d)[3], double (*red)[3])
{
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
        for (int i = 0; i < 3; ++i) d[i] += __shfl_xor_sync(0xffffffffu, d[i], off);
    if (lane == 0)
        for (int i = 0; i < 3; ++i) red[warp][i] = d[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w][i];
        d[i] = t;
    }
    __syncthreads();
}

// Closes a tell (256 threads of one block, after every column's step): ClipUp's factors, and its step where the columns are
// few; the counters.
// Most column quads a single block moves; more take a kernel of their own.  64 members, ask and tell, in the block / in a kernel: 8,192
// columns 13.2 / 14.6 us, 12,288 14.8 / 14.6, 16,384 16.9 / 14.5, 32,768 23.3 / 16.8.
constexpr uint32_t kClipupInClose = 3072;

__device__ __forceinline__ void close_tell(const StepArgs& a, uint32_t n_blocks, bool skip, double (*red)[3])
{
    if (a.mode == kStepClipup && !skip) {
        double d[3] = { 0., 0., 0. };
        for (uint32_t b = threadIdx.x; b < n_blocks; b += 256u)
            for (int i = 0; i < 3; ++i) d[i] += __ldcg(a.norms + 3u * b + i);
        block_dots(d, red);
        const double k = d[2] > 0.0 ? static_cast<double>(a.lr) / sqrt(d[2]) : 0.0, mom = a.momentum;
        const double vn = sqrt(fmax(mom * mom * d[0] + 2.0 * mom * k * d[1] + k * k * d[2], 0.0));
        const float factor = static_cast<float>(k);
        const float scale = vn > static_cast<double>(a.max_speed) ? static_cast<float>(static_cast<double>(a.max_speed) / vn) : 1.0f;
        if (a.ldD / 4u <= kClipupInClose) {
            for (uint32_t q = threadIdx.x; q < a.ldD / 4u; q += 256u) clipup_quad(a, q, factor, scale);
        } else if (threadIdx.x == 0) {
            a.norms[3u * n_blocks] = factor; a.norms[3u * n_blocks + 1u] = scale; a.norms[3u * n_blocks + 2u] = 1.0;
        }
    } else if (a.mode == kStepClipup && threadIdx.x == 0) {
        a.norms[3u * n_blocks + 2u] = 0.0;                   // the step is left out
    }
    if (threadIdx.x == 0) {
        if (skip) {
            a.status->sticky |= (1u << EVO_ERR_NONFINITE);
            a.status->nonfinite = 0;
        } else {
            a.status->adam_step += 1u;
        }
        a.status->generation += 1u;
    }
}

// Whether this block is the last of n to arrive at a counter; the last one sets it back to zero.  What the others wrote
// before they arrived is visible to it.
__device__ __forceinline__ bool last_to_arrive(uint32_t* counter, uint32_t n, uint32_t* shared_flag)
{
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t before = atomicAdd(counter, 1u);
        *shared_flag = before + 1u == n;
        if (before + 1u == n) *counter = 0u;
    }
    __syncthreads();
    if (*shared_flag) __threadfence();
    return *shared_flag != 0u;
}

// Blocks of k_tell that an SM holds
constexpr uint32_t tell_resident(bool regen, bool sigma, bool rank) { return sigma || rank || regen ? 3u : 5u; }

// counters: [0, column blocks) splits that have arrived, [column blocks] columns
template <bool REGEN, bool SIGMA, bool RANK>
__global__ void __launch_bounds__(256, tell_resident(REGEN, SIGMA, RANK))
k_tell(const float* __restrict__ fitness, int32_t* __restrict__ rank, float* __restrict__ u, const float* __restrict__ eps,
       PhiloxKey key, uint32_t pair0, uint32_t H, uint32_t P, uint32_t D, uint32_t pairs_per_split, double* __restrict__ partial,
       float* __restrict__ sigma_partial, uint32_t* __restrict__ counters, const StepArgs a)
{
    __shared__ double sums[kTellLanes - 1][kTellQuads][4];
    __shared__ float ssums[SIGMA ? kTellLanes - 1 : 1][SIGMA ? kTellQuads : 1][4];
    __shared__ __align__(16) uint32_t keys[RANK ? kRankInTell : 4];
    __shared__ float2 uu_s[RANK ? kTellPairs : 1];
    __shared__ double red[8][3];
    __shared__ float corr[2];
    __shared__ uint32_t flag;
    dep_wait();
    dep_trigger();
    DeviceStatus* status = a.status;
    const uint32_t ldD = a.ldD;
    const uint32_t q = threadIdx.x % kTellQuads, lane = threadIdx.x / kTellQuads;
    const uint32_t quad = blockIdx.x * kTellQuads + q;
    const bool live = quad * 4u < ldD;
    const uint32_t generation = status->generation;
    const uint32_t j0 = blockIdx.y * pairs_per_split;
    const uint32_t j1 = min(H, j0 + pairs_per_split);
    const uint32_t first = j0 + lane;
    const float2* up = reinterpret_cast<const float2*>(u) + pair0;    // u is global, eps rows are the shard's
    PhiloxItem item;
    if (REGEN) item = philox_item(quad, generation, 0u, key);
    auto noise = [&](uint32_t j) -> float4 {
        if (REGEN) return normal4(philox4x32_10(item, pair0 + j, key));
        return __ldcs(reinterpret_cast<const float4*>(eps + static_cast<size_t>(j) * ldD) + quad);
    };
    constexpr bool kPrefetch = RANK && !REGEN;             // the first rows of stored noise are on their way while the ranks are counted
    float4 e[kGradRows];
    if constexpr (kPrefetch) {
#pragma unroll
        for (int i = 0; i < kGradRows; ++i) e[i] = live && first < j1 ? noise(min(first + i * kTellLanes, j1 - 1u)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    // A small problem is a chain of memory round trips: what the step will need is asked for (and Adam's corrections are
    // computed) while the ranks are counted (generation of the CNN, 64 members: 93.8 -> 92.5 us).
    QuadState state;
    if (RANK && lane == 0 && live && a.mode != kStepSums) state = load_quad(a, quad);
    auto corrections = [&](uint32_t t) {
        if (a.mode != kStepAdam || t >= 2u) return;
        const double beta = t ? a.beta2 : a.beta1;
        corr[t] = static_cast<float>(1.0 / (1.0 - power(beta, status->adam_step + 1u)));
    };
    if (RANK) corrections(threadIdx.x - 224u);                  // (the last warp's)
    if constexpr (RANK) {
        const uint32_t wl = threadIdx.x & 31u, padded = (P + kRankRun - 1u) / kRankRun * kRankRun;
        for (uint32_t i = threadIdx.x; i < padded; i += 256u) {
            const float f = i < P ? fitness[i] : 0.f;
            if (f != f) atomicOr(&status->nonfinite, 1u);
            keys[i] = i < P ? rank_key(f) : 0xFFFFFFFFu;
        }
        __syncthreads();
        for (uint32_t j = j0 + (threadIdx.x >> 5); j < j1; j += 8u) {          // a warp ranks a pair
            const uint32_t mk[2] = { keys[2u * j], keys[2u * j + 1u] };
            uint32_t below[2] = { 0u, 0u };
            count_below<2>(keys, 0u, P, 2u * j, mk, below, wl);
            const uint32_t r0 = __reduce_add_sync(0xffffffffu, below[0]), r1 = __reduce_add_sync(0xffffffffu, below[1]);
            if (wl == 0) {
                const float2 uu = make_float2(centred_rank(r0, P), centred_rank(r1, P));
                uu_s[j - j0] = uu;
                if (blockIdx.x == 0 && EVO_IN_BOUNDS(status, EVO_SITE_RANK, 2u * j + 1u, P)) {
                    reinterpret_cast<int2*>(rank)[j] = make_int2(static_cast<int>(r0), static_cast<int>(r1));
                    reinterpret_cast<float2*>(u)[j] = uu;
                }
            }
        }
        __syncthreads();
    }

    Acc4 acc = { 0., 0., 0., 0. }, acc2 = acc;             // two chains of sums
    std::conditional_t<REGEN, SigmaSums32, SigmaSums64> sacc;
    if (live) {
        auto weight = [&](uint32_t j) { return RANK ? uu_s[j - j0] : __ldg(up + j); };
        auto add = [&](int i, const float2& uu, const float4& z) {
            acc_fma(i & 1 ? acc2 : acc, static_cast<double>(uu.x) - static_cast<double>(uu.y), z);            // (exact difference)
            if (SIGMA) sacc.add(i, uu, z);
        };
        uint32_t j = first;
        if constexpr (kPrefetch) {
            // rows beyond the split are its last row again, with weight 0
#pragma unroll
            for (int i = 0; i < kGradRows; ++i)
                add(i, j + i * kTellLanes < j1 ? weight(j + i * kTellLanes) : make_float2(0.f, 0.f), e[i]);
            j += kGradRows * kTellLanes;
        }
        if constexpr (REGEN) {
            // (four rows sampled before the first is added: 1,440 us instead of 1,399 at 1,000,003 columns, 1,000 pairs)
#pragma unroll 4
            for (; j < j1; j += kTellLanes) add(0, weight(j), noise(j));
        } else {
            for (; j + (kGradRows - 1) * kTellLanes < j1; j += kGradRows * kTellLanes) {
                float2 w[kGradRows];
#pragma unroll
                for (int i = 0; i < kGradRows; ++i) { e[i] = noise(j + i * kTellLanes); w[i] = weight(j + i * kTellLanes); }
#pragma unroll
                for (int i = 0; i < kGradRows; ++i) add(i, w[i], e[i]);
            }
#pragma unroll
            for (int i = 0; i < kGradRows - 1; ++i)
                if (j + i * kTellLanes < j1) add(i, weight(j + i * kTellLanes), noise(j + i * kTellLanes));
        }
        acc.x += acc2.x; acc.y += acc2.y; acc.z += acc2.z; acc.w += acc2.w;
    }
    float sr[4];
    sacc.sums(sr);
    // the pair lanes in order
    if (lane > 0) {
        sums[lane - 1u][q][0] = acc.x; sums[lane - 1u][q][1] = acc.y; sums[lane - 1u][q][2] = acc.z; sums[lane - 1u][q][3] = acc.w;
        if (SIGMA) { ssums[lane - 1u][q][0] = sr[0]; ssums[lane - 1u][q][1] = sr[1]; ssums[lane - 1u][q][2] = sr[2]; ssums[lane - 1u][q][3] = sr[3]; }
    }
    __syncthreads();
    double r[4] = { acc.x, acc.y, acc.z, acc.w };
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool real = quad * 4u + i < D;           // padding columns carry nothing (recomputed noise exists there too)
            r[i] = real ? ((r[i] + sums[0][q][i]) + (sums[1][q][i] + sums[2][q][i])) : 0.0;
            if (SIGMA) sr[i] = real ? ((sr[i] + ssums[0][q][i]) + (ssums[1][q][i] + ssums[2][q][i])) : 0.0f;
        }
    }
    if (gridDim.y > 1u) {
        if (lane == 0 && live) {
            double2* out = reinterpret_cast<double2*>(partial + static_cast<size_t>(blockIdx.y) * ldD) + 2u * quad;
            if (EVO_IN_BOUNDS(status, EVO_SITE_GRAD_PARTIAL, static_cast<size_t>(blockIdx.y) * ldD + 4u * quad + 3u,
                              static_cast<size_t>(gridDim.y) * ldD)) {
                out[0] = make_double2(r[0], r[1]);
                out[1] = make_double2(r[2], r[3]);
            }
            if (SIGMA) reinterpret_cast<float4*>(sigma_partial + static_cast<size_t>(blockIdx.y) * ldD)[quad] = make_float4(sr[0], sr[1], sr[2], sr[3]);
        }
        if (!last_to_arrive(counters + blockIdx.x, gridDim.y, &flag)) return;
        // the last block of these columns: the splits, an equal part of them per pair lane, the parts in order
        const uint32_t per = (gridDim.y + kTellLanes - 1u) / kTellLanes;
        double t[4] = { 0., 0., 0., 0. };
        float st[4] = { 0.f, 0.f, 0.f, 0.f };
        if (live)
#pragma unroll 4
            for (uint32_t k = lane * per; k < min((lane + 1u) * per, gridDim.y); ++k) {
                const double2* p = reinterpret_cast<const double2*>(partial + static_cast<size_t>(k) * ldD) + 2u * quad;
                const double2 x = __ldcg(p), y = __ldcg(p + 1);
                t[0] += x.x; t[1] += x.y; t[2] += y.x; t[3] += y.y;
                if (SIGMA) {
                    const float4 z = __ldcg(reinterpret_cast<const float4*>(sigma_partial + static_cast<size_t>(k) * ldD) + quad);
                    st[0] += z.x; st[1] += z.y; st[2] += z.z; st[3] += z.w;
                }
            }
        if (lane > 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) { sums[lane - 1u][q][i] = t[i]; if (SIGMA) ssums[lane - 1u][q][i] = st[i]; }
        }
        __syncthreads();
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                r[i] = (t[i] + sums[0][q][i]) + (sums[1][q][i] + sums[2][q][i]);
                if (SIGMA) sr[i] = (st[i] + ssums[0][q][i]) + (ssums[1][q][i] + ssums[2][q][i]);
            }
        }
    }

    // this block has its columns' sums in lane 0's threads; a NaN fitness leaves everything as it is
    const bool skip = *reinterpret_cast<volatile uint32_t*>(&status->nonfinite) != 0u;
    if (!RANK) {
        corrections(threadIdx.x);
        __syncthreads();
    }
    double dots[3] = { 0., 0., 0. };
    if (lane == 0 && live) {
        if (!RANK && a.mode != kStepSums) state = load_quad(a, quad);
        if (a.mode == kStepSums && skip) {                 // the all-reduce still runs on defined values
#pragma unroll
            for (int i = 0; i < 4; ++i) { r[i] = 0.0; sr[i] = 0.0f; }
        }
        if (a.mode == kStepSums || !skip) quad_step(a, quad, r, sr, SIGMA, state, corr[0], corr[1], dots);
    }
    if (a.mode == kStepSums) return;
    if (a.mode == kStepClipup) {
        block_dots(dots, red);
        if (threadIdx.x < 3u) a.norms[3u * blockIdx.x + threadIdx.x] = dots[threadIdx.x];
    }
    if (last_to_arrive(counters + gridDim.x, gridDim.x, &flag)) close_tell(a, gridDim.x, skip, red);
}

// The second half of a sharded tell: the step from the sums that the caller has added over the shards.
__global__ void __launch_bounds__(256)
k_step_from_sums(uint32_t* __restrict__ counters, bool sigma, const StepArgs a)
{
    __shared__ double red[8][3];
    __shared__ float corr[2];
    __shared__ uint32_t flag;
    dep_wait();
    dep_trigger();
    const bool skip = a.status->nonfinite != 0u;
    if (a.mode == kStepAdam && threadIdx.x < 2u) {
        const double beta = threadIdx.x ? a.beta2 : a.beta1;
        corr[threadIdx.x] = static_cast<float>(1.0 / (1.0 - power(beta, a.status->adam_step + 1u)));
    }
    __syncthreads();
    const uint32_t quad = blockIdx.x * 256u + threadIdx.x;
    double dots[3] = { 0., 0., 0. };
    if (quad * 4u < a.ldD && !skip) {
        const double2* p = reinterpret_cast<const double2*>(a.grad_sum) + 2u * quad;
        const double2 x = p[0], y = p[1];
        const double r[4] = { x.x, x.y, y.x, y.y };
        float sr[4] = { 0.f, 0.f, 0.f, 0.f };
        if (sigma) {
            const float4 z = reinterpret_cast<const float4*>(a.sigma_sum)[quad];
            sr[0] = z.x; sr[1] = z.y; sr[2] = z.z; sr[3] = z.w;
        }
        quad_step(a, quad, r, sr, sigma, load_quad(a, quad), corr[0], corr[1], dots);
    }
    if (a.mode == kStepClipup) {
        block_dots(dots, red);
        if (threadIdx.x < 3u) a.norms[3u * blockIdx.x + threadIdx.x] = dots[threadIdx.x];
    }
    if (last_to_arrive(counters, gridDim.x, &flag)) close_tell(a, gridDim.x, skip, red);
}

// ClipUp's step for many columns (a single block took 39 us for 1,000,003 of them, and as long again for the length)
__global__ void __launch_bounds__(256)
k_clipup_apply(uint32_t n_blocks, const StepArgs a)
{
    dep_wait();
    dep_trigger();
    if (a.norms[3u * n_blocks + 2u] == 0.0) return;
    const float factor = static_cast<float>(a.norms[3u * n_blocks]), scale = static_cast<float>(a.norms[3u * n_blocks + 1u]);
    const uint32_t quad = blockIdx.x * 256u + threadIdx.x;
    if (quad * 4u < a.ldD) clipup_quad(a, quad, factor, scale);
}

static uint32_t tell_blocks(uint32_t ldD) { return (ldD / 4u + kTellQuads - 1u) / kTellQuads; }

uint32_t gradient_splits(uint32_t H, uint32_t ldD)
{
    // 32 blocks per SM in all, six waves and more (with half as many the last one shows: 131,072 columns, 8,192 pairs 745 us against 660),
    // as long as every pair lane keeps two rounds of loads; a pure function of the shape.
    const uint32_t bx = tell_blocks(ldD);
    uint32_t s = (kSms * 32u + bx - 1u) / bx;
    if (s > 64u) s = 64u;
    const uint32_t most = (H + 2u * kGradRows * kTellLanes - 1u) / (2u * kGradRows * kTellLanes);
    if (s > most) s = most;
    return s < 1u ? 1u : s;
}

// The splits of a launch with stored noise, out of at most `most`: as many waves of blocks as it takes, each as long as a block's pairs and what
// a block costs besides, about 20 pairs (its first loads, the sums of its lanes, the partial sums' way through memory).  tell, with all
// splits / with these, sigma constant and adapted: 300 members x 40,256 columns 23.2 / 21.6 and 25.7 / 22.6 us, 500 x 60,000 28.6 / 23.6 and 33.8 / 29.7,
// 600 x 90,000 40.0 / 31.8 and 52.3 / 42.1, 200 x 100,000 27.6 / 23.8 and 32.7 / 21.0; 131,072 x 16,384 and few columns keep theirs.  Recomputed
// noise is bound by issue and keeps all (300 x 40,256 29.2 / 29.2, 1,000 x 48,000 52.3 / 56.1, 600 x 90,000 58.4 / 56.3).
static uint32_t whole_waves(uint32_t bx, uint32_t H, uint32_t most, uint32_t places)
{
    uint32_t best = most;
    uint64_t least = ~0ull;
    for (uint32_t s = most; s >= 1u; --s) {
        const uint64_t time = (static_cast<uint64_t>(bx) * s + places - 1u) / places * ((H + s - 1u) / s + 20u);
        if (time < least) { least = time; best = s; }
    }
    return best;
}

size_t clipup_norm_doubles(uint32_t ldD) { return 3u * (tell_blocks(ldD) + 1u); }
size_t tell_counter_words(uint32_t ldD) { return tell_blocks(ldD) + 1u; }

static StepArgs step_args(const TellArgs& a, uint32_t mode, double* grad_sum, float* sigma_sum)
{
    StepArgs s;
    s.mode = mode; s.ldD = a.ldD;
    s.inv_pop = 1.0 / static_cast<double>(a.P);
    s.lr = a.lr; s.beta1 = a.beta1; s.beta2 = a.beta2; s.adam_eps = a.adam_eps; s.momentum = a.clipup_momentum;
    s.max_speed = a.clipup_max_speed; s.sigma_lr = a.sigma_lr; s.sigma_max_change = a.sigma_max_change;
    s.inv_pairs = 2.0f / static_cast<float>(a.P);
    s.sigma_vec = a.sigma_vec; s.center = a.center; s.m = a.m; s.v = a.v; s.g = a.g;
    s.grad_sum = grad_sum; s.sigma_sum = sigma_sum; s.norms = a.norms; s.status = a.status;
    return s;
}

template <bool REGEN, bool SIGMA>
static cudaError_t launch_tell_kernel(cudaStream_t st, const TellArgs& a, const StepArgs& s, bool ranks, dim3 grid, uint32_t pps)
{
    auto kernel = ranks ? k_tell<REGEN, SIGMA, true> : k_tell<REGEN, SIGMA, false>;
    return launch_dependent(kernel, grid, dim3(256), 0, st, a.fitness, a.rank, a.u, a.eps, philox_key(a.k0, a.k1), a.pair0, a.H, a.P,
                            a.D, pps, a.partial, a.sigma_partial, a.counters, s);
}

// ranks + gradient sums (+ the step, unless mode is kStepSums)
static int launch_tell(cudaStream_t st, const TellArgs& a, uint32_t mode, double* grad_sum, float* sigma_sum)
{
    // (places without ranks: what is ranked inside is one wave, or has a single split)
    const uint32_t splits = a.eps ? whole_waves(tell_blocks(a.ldD), a.H, a.splits, kSms * tell_resident(false, a.sigma_partial != nullptr, false)) : a.splits;
    const uint32_t pps = (a.H + splits - 1u) / splits;
    const dim3 grid(tell_blocks(a.ldD), (a.H + pps - 1u) / pps);       // splits that own at least one pair
    // Every column block repeats the ranking of its split's members, P comparisons each: worth it while the repetition costs
    // less than a launch.  A generation of ask and tell, ranked inside / by k_rank: 128 members x 2,000 columns 12.8 / 14.8 us, 200 x 6,000
    // (24 column blocks) 13.9 / 14.7, 256 x 4,609 14.4 / 15.1, 300 x 4,000 15.0 / 14.2, 512 x 4,000 16.2 / 15.5, 2,048 x 8,000 62.8 / 42.4.
    const bool whole = 2u * a.H == a.P && a.pair0 == 0u;
    const bool ranks = whole && a.P <= kRankInTell && pps <= kTellPairs && static_cast<uint64_t>(grid.x) * a.P <= 5000u;
    int launches = 1;
    if (!ranks) {
        if (launch_rank(st, a.fitness, a.P, a.rank, a.u, a.status) < 0) return -1;
        ++launches;
    }
    const StepArgs s = step_args(a, mode, grad_sum, sigma_sum);
    const bool sig = a.sigma_partial != nullptr;
    const cudaError_t e = a.eps ? (sig ? launch_tell_kernel<false, true>(st, a, s, ranks, grid, pps) : launch_tell_kernel<false, false>(st, a, s, ranks, grid, pps))
                                : (sig ? launch_tell_kernel<true, true>(st, a, s, ranks, grid, pps) : launch_tell_kernel<true, false>(st, a, s, ranks, grid, pps));
    if (e != cudaSuccess) return -1;
    if (mode == kStepClipup && a.ldD / 4u > kClipupInClose) {
        if (launch_dependent(k_clipup_apply, dim3((a.ldD / 4u + 255u) / 256u), dim3(256), 0, st, grid.x, s) != cudaSuccess) return -1;
        ++launches;
    }
    return launches;
}

int launch_gradient_update(cudaStream_t st, const TellArgs& a)
{
    return launch_tell(st, a, a.optimizer == EVO_OPT_ADAM ? kStepAdam : kStepClipup, nullptr, nullptr);
}

int launch_gradient_sums(cudaStream_t st, const TellArgs& a, double* grad_sum, float* sigma_sum)
{
    return launch_tell(st, a, kStepSums, grad_sum, sigma_sum);
}

int launch_update_from_sums(cudaStream_t st, const TellArgs& a, double* grad_sum, float* sigma_sum)
{
    const uint32_t mode = a.optimizer == EVO_OPT_ADAM ? kStepAdam : kStepClipup;
    const StepArgs s = step_args(a, mode, grad_sum, sigma_sum);
    const uint32_t nb = (a.ldD / 4u + 255u) / 256u;
    if (launch_dependent(k_step_from_sums, dim3(nb), dim3(256), 0, st, a.counters, a.sigma_partial != nullptr, s) != cudaSuccess) return -1;
    if (mode == kStepClipup && a.ldD / 4u > kClipupInClose) {
        if (launch_dependent(k_clipup_apply, dim3(nb), dim3(256), 0, st, nb, s) != cudaSuccess) return -1;
        return 2;
    }
    return 1;
}

}  // namespace evo
