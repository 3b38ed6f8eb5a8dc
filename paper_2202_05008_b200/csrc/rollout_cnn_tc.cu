// Supervised rollout on the 5th-generation tensor cores (tcgen05, accumulators in TMEM).
//
// The convolutional policy (conv 1->8 5x5, ReLU, pool; conv 8->16 5x5, ReLU, pool; linear
// 256->10) evaluated for every member on the same batch is two dense contractions:
//
//   k_cnn_conv1_tc   conv1 for a group of members at once.  The batch is shared, so a GEMM row (a pooled
//                    pixel) has one A operand for every member: the 6x6 image patch under its pooling
//                    window (K = 36, + 3 entries that carry the bias, padded to 48).  A member's B operand
//                    places its 8 filters at the four positions of the window (N = 32 per member), so
//                    the four conv outputs of a window are four columns of one thread and the 2x2
//                    max-pool is a max over registers.  The epilogue applies ReLU and writes the
//                    pooled activation as bf16, 8 channels = 16 bytes per pixel, in the operand
//                    layout of conv2.
//   k_cnn_conv2_tc   per member and group of 16 images: conv2 as a contraction over whole input
//                    rows.  The member's filter rows, as banded matrices, stay in TENSOR MEMORY as the A
//                    operand (M = 8 output columns x 16 filters, K = 12 input columns x 8 channels);
//                    the activations are the B operand with NO im2col copy: the 8 channels of a pixel
//                    are one 16-byte row of a UMMA core matrix, 8 images are its 8 rows, and filter
//                    row and K-step are address offsets into the group that a single bulk copy
//                    brought in.  D[8 columns x 16 filters][8 rows x 16 images] in TMEM; pool, linear
//                    layer and cross-entropy on CUDA cores.
//
// Few wide MMAs: an MMA of N = 16 or 64 holds the tensor pipe about as long as one of N = 128.
//
// Operands are bf16 (round to nearest even), accumulation fp32 in TMEM.  Every wait is bounded:
// on expiry the block records EVO_ERR_TIMEOUT, frees its TMEM and leaves.
// Paper: Section 3 (supervised tasks are single-step tasks; ConvNet on 28x28 images).
#include "internal.h"
#include "async.cuh"
#include "umma.cuh"
#include "fp32x2.cuh"

namespace evo {

// ------------------------------------------------------------------------------------------
// conv1 for a group of up to 32 members.
//
// GEMM rows are POOLED pixels (128 per tile).  The A operand of a row is the 6x6 image patch under
// its pooling window (K = 36, padded to 48 with three constant-1 entries that carry the bias), the
// same for every member.  A member's B operand has 32 columns: the 8 filters at each of the four
// positions of the pooling window, i.e. the 5x5 filter placed at offset (dy, dx) in the 6x6 patch
// (25/36 dense).  The four conv outputs of a window so land in four columns of one thread, and the
// max-pool is a max over registers, with no shuffles.  Unit of work = (tile, 8 members): 3 MMAs
// (K = 3 x 16) of N = 256 into one of two 256-column accumulators: an MMA of N = 64 holds the tensor
// pipe about as long as one of N = 128, so few wide MMAs beat the 8 narrow ones that separate
// per-position A operands needed.  One warp issues the MMAs and runs ahead; sixteen read the
// accumulators (pool, ReLU, bf16) and store 16 bytes per (member, pixel); four build the next
// tile's A operand while the epilogues run.
// ------------------------------------------------------------------------------------------
constexpr int kC1EpiThreads = 512;                     // four warps per TMEM lane quarter
constexpr int kC1PerThread = 8 * 128 / kC1EpiThreads;  // members of a unit per epilogue thread
constexpr int kC1StageThreads = 128;                   // one thread per pooled pixel of a tile: builds the A operand
constexpr int kC1Threads = kC1EpiThreads + 32 + kC1StageThreads;
constexpr uint32_t kC1Group = 32;                      // members per block
constexpr uint32_t kC1KGroups = 6;                     // K = 48 in groups of 8
constexpr uint32_t kC1NGroups = kC1Group * 32 / 8;     // N = 32 columns per member, in groups of 8
constexpr int kC1SmemB = kC1KGroups * kC1NGroups * 128;   // 96 KB: all members of the group, bf16
constexpr int kC1SmemA = kC1KGroups * 16 * 128;        // 12 KB: one tile
// the block owns all 512 TMEM columns, so it must be alone on its SM: it uses more than half of
// the SM's shared memory
constexpr int kC1DynRequest = kC1SmemB + 2 * kC1SmemA;

struct C1Ctl {
    uint64_t a_full[2];          // the A operand of a tile is staged
    uint64_t a_free[2];          // every MMA that read an A buffer has completed
    uint64_t mma_done[2];        // an accumulator is complete
    uint64_t acc_free[2];        // an accumulator has been read out
    uint32_t tmem_slot;
    volatile int abort;
};

// pooled-1 layout: [member][group of 16 images][y 12][image octet 2][x 12][image in octet 8][channel 8] bf16,
// i.e. the operand layout of the second convolution.  A GEMM row of conv1 is one 16-byte element of
// it, rows in storage order, so a tile of 128 rows is 2 KB of consecutive output.
struct C1Row { uint32_t image, py, px; };
__device__ __forceinline__ C1Row c1_row(uint32_t r)
{
    const uint32_t group = r / 2304u, e = r % 2304u, q = e / 96u;         // q = y * 2 + octet
    return { group * 16u + (q & 1u) * 8u + (e & 7u), q >> 1, (e >> 3) % 12u };
}

// max of three values in one instruction (the 3-input form of max.f32)
__device__ __forceinline__ float fmax3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// 6x6 image patch under the pooled pixel of GEMM row r (zero for images past the batch)
__device__ __forceinline__ void c1_load_patch(const float* __restrict__ images, uint32_t r, uint32_t batch,
                                              float (&patch)[36])
{
    const C1Row at = c1_row(r);
    if (at.image < batch) {
        const float* src = images + static_cast<size_t>(at.image) * 784u + (2u * at.py) * 28u + 2u * at.px;
#pragma unroll
        for (int r = 0; r < 6; ++r) {
            const float2* row = reinterpret_cast<const float2*>(src + r * 28);     // 2*px is even: 8-byte aligned
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float2 v = __ldg(row + c);
                patch[r * 6 + 2 * c] = v.x; patch[r * 6 + 2 * c + 1] = v.y;
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < 36; ++i) patch[i] = 0.f;
    }
}

// the patch of pooled pixel `row` as its row of the A operand (core matrices: 8 rows x 16 bytes,
// k-group kg at +kg*2048, row group at +128); k = 6 * patch row + patch column, then three times 1
__device__ __forceinline__ void c1_stage_row(unsigned char* Abuf, int row, const float (&patch)[36])
{
    uint32_t packed[24];
#pragma unroll
    for (int k = 0; k < 18; ++k) packed[k] = pack_bf16(patch[2 * k], patch[2 * k + 1]);
    packed[18] = pack_bf16(1.f, 1.f);
    packed[19] = pack_bf16(1.f, 0.f);
#pragma unroll
    for (int k = 20; k < 24; ++k) packed[k] = 0u;
#pragma unroll
    for (int kg = 0; kg < 6; ++kg)
        *reinterpret_cast<uint4*>(Abuf + (kg * 16 + (row >> 3)) * 128 + (row & 7) * 16) =
            make_uint4(packed[4 * kg], packed[4 * kg + 1], packed[4 * kg + 2], packed[4 * kg + 3]);
}

__global__ void __launch_bounds__(kC1Threads, 1)
k_cnn_conv1_tc(const float* __restrict__ theta, uint32_t ldD, uint32_t P, const float* __restrict__ images,
               uint32_t batch, uint4* __restrict__ pooled1, DeviceStatus* status)
{
    extern __shared__ __align__(1024) unsigned char dyn[];
    __shared__ __align__(8) C1Ctl ctl;
    dep_wait();

    unsigned char* Bsm = dyn;                                           // 96 KB
    unsigned char* Asm = dyn + kC1SmemB;                                // 2 x 12 KB

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t group0 = blockIdx.y * kC1Group;                      // first member of this block's group
    const uint32_t n_members = min(kC1Group, P - group0);
    const uint32_t n_gm = (n_members + 7u) / 8u;                        // units per tile
    const uint32_t n_groups = (batch + 15u) / 16u;
    const uint32_t n_tiles = n_groups * 18u;                            // 16 images x 144 pooled pixels = 18 tiles

    // ---- B operand: column n = member * 32 + position (dy, dx) * 8 + filter, K = patch element (r, c):
    //      W1[filter][r - dy][c - dx] where that is a tap, else 0; core matrices (k-group, n / 8).
    //      thread = (member, filter): its 25 taps in registers give its four columns.
    for (uint32_t pair = tid; pair < kC1Group * 8u; pair += kC1Threads) {
        const uint32_t m = pair >> 3, ch = pair & 7u;
        float wv[25], bp[3] = { 0.f, 0.f, 0.f };
#pragma unroll
        for (int i = 0; i < 25; ++i) wv[i] = 0.f;
        if (m < n_members) {
            const float* src = theta + static_cast<size_t>(group0 + m) * ldD;
#pragma unroll
            for (int i = 0; i < 25; ++i) wv[i] = __ldg(src + ch * 25u + i);
            // The bias rides in the contraction: against the three constant-1 entries stand three bf16 pieces
            // of it, b = b0 + b1 + b2 to 24 bits, so the fp32 accumulator starts from the unrounded bias and
            // the epilogue has nothing to add.
            const float b = __ldg(src + 200u + ch);
            bp[0] = __bfloat162float(__float2bfloat16_rn(b));
            bp[1] = __bfloat162float(__float2bfloat16_rn(b - bp[0]));
            bp[2] = (b - bp[0]) - bp[1];
        }
#pragma unroll
        for (int pos = 0; pos < 4; ++pos) {
            const int dy = pos >> 1, dx = pos & 1;
            const uint32_t n = m * 32u + pos * 8u + ch;
#pragma unroll
            for (int kg = 0; kg < 6; ++kg) {
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int k = kg * 8 + i, r = k / 6, c = k % 6;
                    v[i] = 0.f;
                    if (k < 36) { if (r >= dy && r < dy + 5 && c >= dx && c < dx + 5) v[i] = wv[(r - dy) * 5 + (c - dx)]; }
                    else if (k < 39) v[i] = bp[k - 36];
                }
                *reinterpret_cast<uint4*>(Bsm + (kg * kC1NGroups + (n >> 3)) * 128u + (n & 7u) * 16u) =
                    make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
            }
        }
    }

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&ctl.a_full[i]), 1);
            mbar_init(smem_u32(&ctl.a_free[i]), 1);
            mbar_init(smem_u32(&ctl.mma_done[i]), 1);
            mbar_init(smem_u32(&ctl.acc_free[i]), kC1EpiThreads / 32);
        }
        ctl.abort = 0;
        mbar_init_fence();
    }
    __syncwarp();
    if (warp == 0) tmem_alloc(smem_u32(&ctl.tmem_slot), 512);
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl.tmem_slot;
    // conv2 is launched as a programmatic dependent: its blocks may become resident (and fetch their filters)
    // as soon as blocks of this kernel leave; it waits for this whole grid before it reads an activation
    if (tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == kC1EpiThreads / 32) {
        // ================= MMA issuer =============================================================
        if (lane == 0) {
            constexpr uint32_t idesc = umma_idesc_bf16(128, 256);
            const uint32_t a_base = smem_u32(Asm), b_base = smem_u32(Bsm);
            uint32_t u = 0, ti = 0;
            for (uint32_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++ti) {
                try_wait_or_abort(&ctl.abort, &ctl.a_full[ti & 1u], (ti >> 1) & 1u, status);
                const uint32_t a0 = a_base + (ti & 1u) * kC1SmemA;
                for (uint32_t gm = 0; gm < n_gm; ++gm, ++u) {
                    const uint32_t buf = u & 1u;
                    try_wait_or_abort(&ctl.abort, &ctl.acc_free[buf], (u >> 1) & 1u, status);
                    tc_fence_after();
#pragma unroll
                    for (uint32_t ks = 0; ks < 3u; ++ks) {
                        const uint64_t ad = umma_smem_desc(a0 + ks * 2u * 2048u, 2048u, 128u);
                        const uint64_t bd = umma_smem_desc(b_base + ks * 2u * (kC1NGroups * 128u) + gm * 32u * 128u, kC1NGroups * 128u, 128u);
                        umma_bf16(tmem + buf * 256u, ad, bd, idesc, ks);
                    }
                    umma_commit(smem_u32(&ctl.mma_done[buf]));
                }
                umma_commit(smem_u32(&ctl.a_free[ti & 1u]));       // arrives once this tile's MMAs are done
            }
        }
    } else if (warp > kC1EpiThreads / 32) {
        // ================= staging warps: im2col rows of the tiles, one tile ahead of the MMAs ============
        // thread = pooled pixel of the tile; the 6x6 image patch under it is its row of the operand.
        // The buffer of tile ti is free once the MMAs of tile ti - 2 have completed.
        const int row = tid - (kC1EpiThreads + 32);
        float patch[36];
        uint32_t ti = 0;
        for (uint32_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++ti) {
            c1_load_patch(images, tile * 128u + row, batch, patch);
            if (ti >= 2u) try_wait_or_abort(&ctl.abort, &ctl.a_free[ti & 1u], ((ti >> 1) - 1u) & 1u, status);
            unsigned char* Abuf = Asm + (ti & 1u) * kC1SmemA;
            c1_stage_row(Abuf, row, patch);
            fence_async_smem();
            asm volatile("bar.sync 2, %0;" :: "n"(kC1StageThreads) : "memory");
            if (row == 0) mbar_arrive(smem_u32(&ctl.a_full[ti & 1u]));
        }
        // the last arrivals on a_free land in this block's shared memory: see them in before the block ends
        if (row < 2 && ti > static_cast<uint32_t>(row)) {
            const uint32_t n_done = (ti - row + 1u) >> 1;              // completions of buffer `row`
            try_wait_or_abort(&ctl.abort, &ctl.a_free[row], (n_done - 1u) & 1u, status);
        }
    } else {
        // ================= epilogue warps ==========================================================
        if (lane == 0) { mbar_arrive(smem_u32(&ctl.acc_free[0])); mbar_arrive(smem_u32(&ctl.acc_free[1])); }
        const int row = tid & 127, part = tid >> 7;       // my pooled pixel (= TMEM lane) and my share of the members
        uint32_t u = 0, ti = 0;
        for (uint32_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++ti) {
            const uint32_t pix_off = tile * 128u + row;                // my GEMM row = my TMEM lane = my output element
            const bool pix_ok = c1_row(pix_off).image < batch;
            const size_t member_stride = static_cast<size_t>(n_groups) * 2304u;

            for (uint32_t gm = 0; gm < n_gm; ++gm, ++u) {
                const uint32_t buf = u & 1u;
                try_wait_or_abort(&ctl.abort, &ctl.mma_done[buf], (u >> 1) & 1u, status);
                tc_fence_after();
                const uint32_t t0 = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + buf * 256u + part * (32u * kC1PerThread);
                // My members of the unit: a member's 8 filters at the four positions of the pooling window are 32 consecutive
                // columns.  One load instruction per member and one wait for both, then the accumulator is free: the turn of an
                // accumulator (MMAs, hand-over, read, hand-back) paces this kernel, no pipe is more than half busy.
                // 500 members x 1000 images: 252 us; with loads of 8 columns and a wait per member 262; with the
                // two accumulators read by eight warps each 281.
                static_assert(kC1PerThread == 2, "two register buffers");
                uint32_t acc[kC1PerThread][4][8];
#pragma unroll
                for (int j = 0; j < kC1PerThread; ++j) tmem_ld32_issue(t0 + j * 32u, acc[j]);
#pragma unroll
                for (int j = 0; j < kC1PerThread; ++j) tmem_ld8x4_fence(acc[j][0], acc[j][1], acc[j][2], acc[j][3]);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctl.acc_free[buf]));
#pragma unroll
                for (int j = 0; j < kC1PerThread; ++j) {
                    const uint32_t (&cur)[4][8] = acc[j];
                    const uint32_t m = gm * 8u + part * kC1PerThread + j;
                    // the accumulators already contain the bias: relu(max4) = two 3-input max per value
                    uint32_t o[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        float v[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int k = 2 * c + h;
                            const float m3 = fmax3(__uint_as_float(cur[0][k]), __uint_as_float(cur[1][k]), __uint_as_float(cur[2][k]));
                            v[h] = fmax3(m3, __uint_as_float(cur[3][k]), 0.f);
                        }
                        o[c] = pack_bf16(v[0], v[1]);
                    }
                    if (pix_ok && m < n_members)
                        pooled1[pix_off + static_cast<size_t>(group0 + m) * member_stride] = make_uint4(o[0], o[1], o[2], o[3]);
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------------
// conv2 + pool + linear + cross-entropy.  Unit of work = (member, group of 16 images).
//
// The contraction runs over a whole input row at a time, with the member's filters as the operand
// that stays.  For filter row dy, the 8 output columns x 16 filters of an output row (M = 128) are a
// product of a banded matrix, holding the 5 taps of that filter row at the offsets input column -
// output column (zero elsewhere; 5/12 dense), with the 12 input columns x 8 channels (K = 96) of the
// input row dy lower.  The five bands (240 columns) live in TENSOR MEMORY for as long as the member
// lasts, so an MMA reads only its activation operand from shared memory: N = (output row, image), and
// with the group stored as [y][image octet][x][image in octet][8 channels] the 8 images of an octet
// are one core matrix, a step in y is a fixed byte offset, and filter row dy is the same operand
// started dy rows lower.  Per unit: 5 filter rows x 6 K-steps on two halves of N = 60 MMAs of
// M = 128, N = 64, K = 16 that each read 2 KB of shared memory, where a tap-by-tap implicit GEMM with the
// pixels on M (13 MMAs of N = 16 per image pair, 104 per unit) read 4.5 KB each and was paced by that.
//
// Roles: warps 0-3 read the accumulators (2x2 max over two columns of a thread and two lanes,
// bias, ReLU, bf16) into a per-image activation buffer; warps 4-11 run the linear layer and the
// cross-entropy from that buffer; two warps each issue the MMAs of one accumulator; one warp fetches
// the filters of the members to come; one brings the groups in, one bulk copy each, through a ring of three.  The roles meet only
// on mbarriers; every wait is bounded, and after a time-out all later waits fall through so that
// no role is left behind.
// ------------------------------------------------------------------------------------------
constexpr int kC2EpiThreads = 128;
constexpr int kC2LinThreads = 256;
constexpr int kC2Issuers = 2;
constexpr int kC2Threads = kC2EpiThreads + kC2LinThreads + 32 * kC2Issuers + 32 + 32;
constexpr uint32_t kGroupRowBytes = 12 * 8 * 16;         // one (y, image octet): 12 pixels x 8 images x 16 bytes
constexpr uint32_t kGroupBytes = 12 * 2 * kGroupRowBytes;   // 36,864
constexpr uint32_t kC2Ring = 3;                          // groups in flight
constexpr uint32_t kC2BandCols = 48;                     // tensor-memory columns of one band: K = 96 bf16
constexpr uint32_t kC2AccCol = 256;                      // first accumulator column (the bands take 240)
constexpr int kP2Pitch = 264;                            // bf16 per image: 132 words, images fall in distinct banks
constexpr int kRawPitch = 201;                           // floats per filter in the weight scratch (odd: no bank conflicts)

struct __align__(128) C2Smem {
    unsigned char a[kC2Ring][kGroupBytes];               // pooled-1 groups (ring)
    float raw[16 * kRawPitch];                           // W2 as stored, one padded row per filter
    uint4 taps[2][16][25];                               // W2 as bf16: the 8 channels of (filter, tap) = the 4 columns of an input column;
                                                         // [member of the block's range & 1]: the next member's are fetched ahead
    float wfT[2][256 * 12];                              // linear layer transposed [k][class], bf16-rounded, one copy per linear team
    __align__(16) __nv_bfloat16 p2[2][16][kP2Pitch];     // pooled-2 activations of a unit's images, k = pixel*16 + channel
    float part[2][2][4][16][12];                         // [team][unit parity in the team] partial logits of the four warps
    float b2[2][16];
    float bfc[2][12];
    uint64_t a_full[kC2Ring];                            // a group has landed
    uint64_t a_free[kC2Ring];                            // every MMA that read a group has completed
    uint64_t mma_done[2];                                // an accumulator is complete
    uint64_t acc_free[2];                                // an accumulator has been read out
    uint64_t p2_full[2];                                 // the activations of a unit are written
    uint64_t p2_free[2];                                 // ... and have been consumed by the linear layer
    uint64_t drain;                                      // all MMAs of the block have completed
    uint32_t staged;                                     // members of the block's range whose bands have been staged
    uint32_t taps_loaded;                                // ... whose filters are in `taps`
    uint32_t issued[2];                                  // per issuer: one past the last unit whose MMAs it has issued
    uint32_t tmem_slot;
    volatile int abort;
};

__device__ __forceinline__ void c2_wait(C2Smem& S, uint64_t* bar, uint32_t parity, DeviceStatus* status)
{
    try_wait_or_abort(&S.abort, bar, parity, status);
}

// Progress that is counted, not signalled: the members whose bands are staged, the members whose
// filters are in shared memory, the units whose MMAs an issuer has issued.  Every counter has one
// writer and only grows, so a role that skips some values (an issuer with no unit of some member
// when a group count is one) cannot misread it as it could an mbarrier's phase parity.  The wait is
// bounded like every other.
__device__ __forceinline__ void c2_wait_count(C2Smem& S, const uint32_t* counter, uint32_t need, DeviceStatus* status)
{
    const uint32_t addr = smem_u32(counter);
    uint32_t have;
    long long t0 = 0;
    for (;;) {
        asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(have) : "r"(addr) : "memory");
        if (have >= need || S.abort) return;
        if (t0 == 0) t0 = clock64();
        if (clock64() - t0 > (1ll << status->wait_cycles_log2)) {
            S.abort = 1;
            atomicOr(&status->sticky, 1u << EVO_ERR_TIMEOUT);
            return;
        }
        __nanosleep(64);
    }
}
__device__ __forceinline__ void c2_set_count(uint32_t* counter, uint32_t value)
{
    asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" :: "r"(smem_u32(counter)), "r"(value) : "memory");
}

// The 30 MMAs of one half (4 output rows x 16 images) of a unit.  b0 = the group, advanced to the
// half's first row; filter row dy takes band dy and starts the activation operand dy rows lower;
// a K-step is two input columns.
__device__ __forceinline__ void c2_issue_mma(uint32_t bands, uint32_t b0, uint32_t d_tmem)
{
    constexpr uint32_t idesc = umma_idesc_bf16(128, 128);
#pragma unroll
    for (uint32_t dy = 0; dy < 5u; ++dy)
#pragma unroll
        for (uint32_t ks = 0; ks < 6u; ++ks) {
            const uint64_t bd = umma_smem_desc(b0 + dy * 2u * kGroupRowBytes + ks * 256u, 128u, kGroupRowBytes);
            umma_bf16_ts(d_tmem, bands + dy * kC2BandCols + ks * 8u, bd, idesc, dy | ks);
        }
}

__global__ void __launch_bounds__(kC2Threads, 1)
k_cnn_conv2_tc(const float* __restrict__ theta, uint32_t ldD, uint32_t P, const unsigned char* __restrict__ pooled1,
               const int32_t* __restrict__ labels, uint32_t batch,
               float* __restrict__ loss, DeviceStatus* status)
{
    extern __shared__ __align__(1024) unsigned char dyn[];
    C2Smem& S = *reinterpret_cast<C2Smem*>(dyn);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t n_groups = (batch + 15u) / 16u;
    const uint64_t n_units = static_cast<uint64_t>(P) * n_groups;     // (member, group), member-major
    // Units are equal in cost, so every block takes one contiguous range, equal to within one unit.
    // The loss is written per image, so the result does not depend on where the ranges are cut.
    const uint32_t u_begin = static_cast<uint32_t>(static_cast<uint64_t>(blockIdx.x) * n_units / gridDim.x);
    const uint32_t u_end = static_cast<uint32_t>((static_cast<uint64_t>(blockIdx.x) + 1u) * n_units / gridDim.x);
    const uint32_t n_mine = u_end - u_begin;

    if (tid == 0) {
        for (uint32_t i = 0; i < kC2Ring; ++i) {
            mbar_init(smem_u32(&S.a_full[i]), 1);
            mbar_init(smem_u32(&S.a_free[i]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&S.mma_done[i]), 1);
            mbar_init(smem_u32(&S.acc_free[i]), kC2EpiThreads / 32);
            mbar_init(smem_u32(&S.p2_full[i]), kC2EpiThreads / 32);
            mbar_init(smem_u32(&S.p2_free[i]), kC2LinThreads / 64);
        }
        mbar_init(smem_u32(&S.drain), kC2Issuers);
        S.staged = 0;
        S.taps_loaded = 0;
        S.issued[0] = 0;
        S.issued[1] = 0;
        S.abort = 0;
        mbar_init_fence();
    }
    // A block whose range runs into a second member will want that member's parameters in the middle of its
    // work, from memory that is busy streaming activations by then: ask for them now, into L2.
    if ((u_end - 1u) / n_groups != u_begin / n_groups) {
        const float* nxt = theta + static_cast<size_t>(u_begin / n_groups + 1u) * ldD + 208u;     // conv2 and linear layers
        for (uint32_t i = tid; i < (kCnnParams - 208u + 31u) / 32u; i += kC2Threads)
            asm volatile("prefetch.global.L2 [%0];" :: "l"(nxt + 32u * i));
    }
    for (int k = tid; k < 512; k += kC2Threads) { S.wfT[k >> 8][(k & 255) * 12 + 10] = 0.f; S.wfT[k >> 8][(k & 255) * 12 + 11] = 0.f; }
    if (tid < 4) S.bfc[tid >> 1][10 + (tid & 1)] = 0.f;
    __syncwarp();
    if (warp == 0) tmem_alloc(smem_u32(&S.tmem_slot), 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_slot;
    if (tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the finalize kernel may be set up

    if (warp < kC2EpiThreads / 32) {
        // ================= accumulator warps: bands -> tensor memory; pool, bias, ReLU -> activations ===
        // both accumulators start out free
        if (lane == 0) { mbar_arrive(smem_u32(&S.acc_free[0])); mbar_arrive(smem_u32(&S.acc_free[1])); }
        // TMEM lane = output column x (2 per warp) x filter: the warp owns pooled column px = warp; a
        // thread holds the 8 x 16 (output row, image) outputs of its (column, filter).  Row pairs are
        // a max over two registers; the column pair is lane ^ 16, done as an exchange: of a pair of
        // pooled rows (a, a + 2) the thread of the even column keeps row a, that of the odd column a + 2.
        const int f = lane & 15, odd = lane >> 4, px = warp;     // output column 2 * warp + odd
        const uint32_t tm_lane = tmem + (static_cast<uint32_t>(warp * 32) << 16);
        const uint32_t first_member = u_begin / n_groups;
        // A member's filters on their way to tensor memory, in two steps.  The first needs no tensor memory: W2
        // as stored -> shared memory (coalesced) -> bf16, the 8 channels of a (filter, tap) as one 16-byte
        // entry.  Here for the block's first member; the weights warp does it for the later ones, ahead of time.
        auto load_taps = [&](uint32_t member) {
            const float* prm = theta + static_cast<size_t>(member) * ldD;
            const float4* w2v = reinterpret_cast<const float4*>(prm + 208u);          // 16-byte aligned
            float4 t2[7];
#pragma unroll
            for (int k = 0; k < 7; ++k)
                t2[k] = (tid + k * kC2EpiThreads < 800) ? __ldg(w2v + tid + k * kC2EpiThreads) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 7; ++k) {
                const uint32_t i = 4u * (tid + k * kC2EpiThreads);                   // flat (filter*8 + channel)*25 + tap
                if (i < 3200u) {
                    float* d = S.raw + (i / 200u) * kRawPitch + i % 200u;           // 200 = 4 * 50: a float4 stays in its filter
                    d[0] = t2[k].x; d[1] = t2[k].y; d[2] = t2[k].z; d[3] = t2[k].w;
                }
            }
            if (tid < 16) S.b2[0][tid] = prm[3408u + tid];
            asm volatile("bar.sync 1, %0;" :: "n"(kC2EpiThreads) : "memory");
            for (uint32_t i = tid; i < 400u; i += kC2EpiThreads) {
                const float* src = S.raw + (i / 25u) * kRawPitch + i % 25u;           // (filter, tap), channels 25 apart
                S.taps[0][i / 25u][i % 25u] = make_uint4(pack_bf16(src[0], src[25]), pack_bf16(src[50], src[75]),
                                                      pack_bf16(src[100], src[125]), pack_bf16(src[150], src[175]));
            }
            asm volatile("bar.sync 1, %0;" :: "n"(kC2EpiThreads) : "memory");
        };
        // The second step, once every MMA of the previous member has completed: band dy, row (output column
        // xo, filter f), K = (input column xi, channel) is W2[f][channel][dy][xi - xo].  A tensor-memory column
        // holds two consecutive K, 8 columns = two input columns = one K-step.  Only the input columns
        // xo .. xo + 4 of a row are not zero, the same for every member: they lie in the three K-steps from
        // xo / 2 on.  Then the issuers are told.
        auto write_bands = [&](uint32_t member) -> float {
            const uint4 (&taps)[16][25] = S.taps[(member - first_member) & 1u];
#pragma unroll
            for (uint32_t dy = 0; dy < 5u; ++dy)
#pragma unroll
                for (int t = 0; t < 3; ++t) {
                    uint4 q[2];
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int dx = 2 * t + c - odd;                                // xo is 2 * warp + odd
                        q[c] = make_uint4(0u, 0u, 0u, 0u);
                        if (dx >= 0 && dx <= 4) q[c] = taps[f][dy * 5 + dx];
                    }
                    const uint32_t u[8] = { q[0].x, q[0].y, q[0].z, q[0].w, q[1].x, q[1].y, q[1].z, q[1].w };
                    tmem_st8(tm_lane + dy * kC2BandCols + static_cast<uint32_t>(warp + t) * 8u, u);
                }
            tmem_st_wait();
            tc_fence_before();
            const float b = S.b2[(member - first_member) & 1u][f];      // read before the buffer is given back
            asm volatile("bar.sync 1, %0;" :: "n"(kC2EpiThreads) : "memory");
            if (tid == 0) c2_set_count(&S.staged, member - first_member + 1u);
            return b;                                                    // the member's bias for this thread's filter
        };
        {   // the zeros of the bands, once
            const uint32_t z[8] = { 0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u };
#pragma unroll
            for (uint32_t c = 0; c < 5u * kC2BandCols; c += 8u) tmem_st8(tm_lane + c, z);
            tmem_st_wait();
        }
        load_taps(first_member);
        float bias = write_bands(first_member);
        for (uint32_t j = 0; j < n_mine; ++j) {
            const uint32_t member = (u_begin + j) / n_groups, ab = j & 1u, par = (j >> 1) & 1u;
            const bool last_of_member = j + 1u < n_mine && (u_begin + j + 1u) / n_groups != member;
            c2_wait(S, &S.mma_done[ab], par, status);
            tc_fence_after();
            float next_bias = bias;
            if (last_of_member) {
                // This was the member's last MMA, so the bands can be rewritten, and the next member's MMAs
                // run while this unit's accumulator is read out.
                c2_wait_count(S, &S.taps_loaded, member + 1u - first_member + 1u, status);
                next_bias = write_bands(member + 1u);
            }
            c2_wait(S, &S.p2_free[ab], par, status);
            const uint32_t t0 = tm_lane + kC2AccCol + ab * 128u;
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                // accumulator column = output row * 16 + image: pooled rows a and a + 2 are output rows 2a, 2a+1 and 2a+4, 2a+5
                uint32_t lo[2][16], hi[2][16];
                tmem_ld16_issue(t0 + (2 * a) * 16u, lo[0]);     tmem_ld16_issue(t0 + (2 * a + 1) * 16u, lo[1]);
                tmem_ld16_issue(t0 + (2 * a + 4) * 16u, hi[0]); tmem_ld16_issue(t0 + (2 * a + 5) * 16u, hi[1]);
                tmem_ld16_fence(lo[0]); tmem_ld16_fence(lo[1]); tmem_ld16_fence(hi[0]); tmem_ld16_fence(hi[1]);
                if (a == 1) {                                          // the accumulator is in registers now
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&S.acc_free[ab]));
                }
                const int py = a + 2 * odd;
                __nv_bfloat16* dst = &S.p2[ab][0][(py * 4 + px) * 16 + f];
#pragma unroll
                for (int img = 0; img < 16; ++img) {
                    const float va = fmaxf(__uint_as_float(lo[0][img]), __uint_as_float(lo[1][img]));
                    const float vb = fmaxf(__uint_as_float(hi[0][img]), __uint_as_float(hi[1][img]));
                    const float keep = odd ? vb : va;
                    const float give = odd ? va : vb;
                    const float v = fmaxf(fmaxf(keep, __shfl_xor_sync(0xffffffffu, give, 16)) + bias, 0.f);
                    dst[img * kP2Pitch] = __float2bfloat16_rn(v);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&S.p2_full[ab]));
            bias = next_bias;
        }
    } else if (warp < (kC2EpiThreads + kC2LinThreads) / 32) {
        // ================= linear layer 256 -> 10 and cross-entropy ==============================
        // Two teams of four warps take the units in turn (team = unit parity = activation buffer), so a
        // team has two unit times for the chain products -> sums -> barrier -> softmax of its unit.
        // thread = (images ip and ip + 8, slice s of the inputs: the pairs k = 2(s + 16 i), +1); the 16
        // slices meet by two shuffles inside a warp and through shared memory across the four warps.
        const int lt = (tid - kC2EpiThreads) & 127, wl = lt >> 5;
        const uint32_t team = static_cast<uint32_t>(tid - kC2EpiThreads) >> 7;
        if (lane == 0) mbar_arrive(smem_u32(&S.p2_free[team]));
        const int ip = lane & 7, s = wl * 4 + (lane >> 3);
        uint32_t staged_member = 0xFFFFFFFFu;
        for (uint32_t j = team; j < n_mine; j += 2u) {
            const uint32_t unit = u_begin + j, member = unit / n_groups, group = unit % n_groups;
            const uint32_t par = (j >> 1) & 1u;
            // softmax: warp = four images, 8 lanes each, lane = classes c and c + 8; the label comes early
            const int cls = lane & 7, il = 4 * wl + (lane >> 3);
            const uint32_t image = group * 16u + il;
            const int lab = image < batch ? min(max(__ldg(labels + image), 0), 9) : 0;
            if (member != staged_member) {
                // The teams keep their own copy of the layer (theirs to rewrite once they are past the
                // previous unit's products: the barrier below).
                staged_member = member;
                const float* prm = theta + static_cast<size_t>(member) * ldD;
                const float4* wfv = reinterpret_cast<const float4*>(prm + 3424u);     // 16-byte aligned
                float4 tf[5];
#pragma unroll
                for (int k = 0; k < 5; ++k) tf[k] = __ldg(wfv + lt + k * 128);
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    // flat index cls*256 + (c*16 + pos), 4 consecutive pos; stored at row pos*16 + c
                    const uint32_t i = 4u * (lt + k * 128);
                    const uint32_t oc = i >> 8, c = (i >> 4) & 15u, pos = i & 15u;
                    float* d = S.wfT[team] + (pos * 16u + c) * 12u + oc;
                    d[0 * 192]  = __bfloat162float(__float2bfloat16_rn(tf[k].x));
                    d[1 * 192]  = __bfloat162float(__float2bfloat16_rn(tf[k].y));
                    d[2 * 192]  = __bfloat162float(__float2bfloat16_rn(tf[k].z));
                    d[3 * 192]  = __bfloat162float(__float2bfloat16_rn(tf[k].w));
                }
                if (lt < 10) S.bfc[team][lt] = prm[5984u + lt];
                asm volatile("bar.sync %0, 128;" :: "r"(2u + team) : "memory");
            }
            c2_wait(S, &S.p2_full[team], par, status);
            float2 acc[2][5];
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int c = 0; c < 5; ++c) acc[e][c] = make_float2(0.f, 0.f);
            const uint32_t* x0 = reinterpret_cast<const uint32_t*>(&S.p2[team][ip][0]) + s;        // two inputs per word
            const uint32_t* x1 = reinterpret_cast<const uint32_t*>(&S.p2[team][ip + 8][0]) + s;
            const float* wr = S.wfT[team] + s * 24;
#pragma unroll 4
            for (int i = 0; i < 8; ++i) {
                const uint32_t xa = x0[16 * i], xb = x1[16 * i];
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const float fa = __uint_as_float(hh ? (xa & 0xFFFF0000u) : (xa << 16));
                    const float fb = __uint_as_float(hh ? (xb & 0xFFFF0000u) : (xb << 16));
                    const float2 va = make_float2(fa, fa), vb = make_float2(fb, fb);
                    const float* wk = wr + (16 * i) * 24 + hh * 12;
                    const float4 w0 = *reinterpret_cast<const float4*>(wk);
                    const float4 w1 = *reinterpret_cast<const float4*>(wk + 4);
                    const float2 w2 = *reinterpret_cast<const float2*>(wk + 8);
                    ffma2(acc[0][0], make_float2(w0.x, w0.y), va); ffma2(acc[1][0], make_float2(w0.x, w0.y), vb);
                    ffma2(acc[0][1], make_float2(w0.z, w0.w), va); ffma2(acc[1][1], make_float2(w0.z, w0.w), vb);
                    ffma2(acc[0][2], make_float2(w1.x, w1.y), va); ffma2(acc[1][2], make_float2(w1.x, w1.y), vb);
                    ffma2(acc[0][3], make_float2(w1.z, w1.w), va); ffma2(acc[1][3], make_float2(w1.z, w1.w), vb);
                    ffma2(acc[0][4], w2, va);                      ffma2(acc[1][4], w2, vb);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&S.p2_free[team]));    // the activations have been read
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int c = 0; c < 5; ++c) {
                    float2 v = acc[e][c];
                    v.x += __shfl_xor_sync(0xffffffffu, v.x, 8);  v.y += __shfl_xor_sync(0xffffffffu, v.y, 8);
                    v.x += __shfl_xor_sync(0xffffffffu, v.x, 16); v.y += __shfl_xor_sync(0xffffffffu, v.y, 16);
                    acc[e][c] = v;
                }
            if (lane < 8) {
                if (wl == 0) {                          // the bias joins the first warp's part: nothing reads it after the barrier
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int c = 0; c < 5; ++c) { acc[e][c].x += S.bfc[team][2 * c]; acc[e][c].y += S.bfc[team][2 * c + 1]; }
                }
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    float* d = &S.part[team][par][wl][ip + 8 * e][0];
                    *reinterpret_cast<float4*>(d) = make_float4(acc[e][0].x, acc[e][0].y, acc[e][1].x, acc[e][1].y);
                    *reinterpret_cast<float4*>(d + 4) = make_float4(acc[e][2].x, acc[e][2].y, acc[e][3].x, acc[e][3].y);
                    *reinterpret_cast<float2*>(d + 8) = acc[e][4];
                }
            }
            asm volatile("bar.sync %0, 128;" :: "r"(2u + team) : "memory");
            {
                const float* q = &S.part[team][par][0][il][cls];             // warps added in a fixed order
                const float lg0 = (q[0] + q[192]) + (q[384] + q[576]);
                const float lg1 = cls < 2 ? (q[8] + q[200]) + (q[392] + q[584]) : -INFINITY;
                float mx = fmaxf(lg0, lg1);
#pragma unroll
                for (int d = 4; d > 0; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
                float se = expf(lg0 - mx) + (cls < 2 ? expf(lg1 - mx) : 0.f);
#pragma unroll
                for (int d = 4; d > 0; d >>= 1) se += __shfl_xor_sync(0xffffffffu, se, d);
                const float a0 = __shfl_sync(0xffffffffu, lg0, (lane & 24) + (lab & 7));
                const float a1 = __shfl_sync(0xffffffffu, lg1, (lane & 24) + (lab & 7));
                const float at_label = lab < 8 ? a0 : a1;
                // after a time-out the numbers mean nothing: NaN, which makes tell skip the update
                if (cls == 0 && image < batch)
                    loss[static_cast<size_t>(member) * batch + image] = S.abort ? __int_as_float(0x7FC00000) : (mx + logf(se)) - at_label;
            }
        }
    } else if (warp < (kC2EpiThreads + kC2LinThreads) / 32 + kC2Issuers) {
        // ================= MMA issuers: one thread per (accumulator, half of the output rows) =====
        if (lane == 0) {
            const uint32_t ab = warp - (kC2EpiThreads + kC2LinThreads) / 32;
            const uint32_t first_member = u_begin / n_groups;
            uint32_t seen_member = 0xFFFFFFFFu;
            for (uint32_t j = ab; j < n_mine; j += 2u) {
                const uint32_t member = (u_begin + j) / n_groups, slot = j % kC2Ring;
                if (member != seen_member) {
                    seen_member = member;
                    c2_wait_count(S, &S.staged, member - first_member + 1u, status);
                    // When a member's bands are staged both issuers are let go at once, and the MMAs of two
                    // units taking turns in the pipe would finish the first unit late: in unit order here.
                    c2_wait_count(S, &S.issued[ab ^ 1u], j, status);      // unit j - 1 is the other issuer's
                }
                c2_wait(S, &S.a_full[slot], (j / kC2Ring) & 1u, status);
                c2_wait(S, &S.acc_free[ab], (j >> 1) & 1u, status);
                if (S.abort) break;
                tc_fence_after();
                c2_issue_mma(tmem, smem_u32(S.a[slot]), tmem + kC2AccCol + ab * 128u);
                umma_commit(smem_u32(&S.mma_done[ab]));
                umma_commit(smem_u32(&S.a_free[slot]));
                c2_set_count(&S.issued[ab], j + 1u);
            }
            umma_commit(smem_u32(&S.drain));                          // arrives when all my MMAs have completed
        }
    } else if (warp == (kC2EpiThreads + kC2LinThreads) / 32 + kC2Issuers) {
        // ================= weights warp: the later members' filters, fetched ahead =================
        // For the members after the block's first: W2 -> bf16 entries in the buffer that the member
        // before the previous one has left (its bands are staged), straight from global memory (L2: they
        // were asked for at the start); slow, but a member's worth of units ahead of when it is needed.
        const uint32_t first_member = u_begin / n_groups, n_ord = (u_end - 1u) / n_groups - first_member + 1u;
        for (uint32_t ord = 1; ord < n_ord; ++ord) {
            c2_wait_count(S, &S.staged, ord - 1u, status);
            if (S.abort) break;
            const float* prm = theta + static_cast<size_t>(first_member + ord) * ldD;
            for (uint32_t i = lane; i < 400u; i += 32u) {
                const float* src = prm + 208u + (i / 25u) * 200u + i % 25u;             // (filter, tap), channels 25 apart
                float v[8];
#pragma unroll
                for (int ch = 0; ch < 8; ++ch) v[ch] = __ldg(src + ch * 25);
                S.taps[ord & 1u][i / 25u][i % 25u] = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]),
                                                                pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
            }
            if (lane < 16) S.b2[ord & 1u][lane] = __ldg(prm + 3408u + lane);
            __syncwarp();
            if (lane == 0) c2_set_count(&S.taps_loaded, ord + 1u);
        }
    } else {
        // ================= producer: one bulk copy per unit, up to three units ahead ===============
        if (lane == 0) {
            const unsigned char* src = pooled1 + static_cast<size_t>(u_begin) * kGroupBytes;
            uint32_t issued = 0;
            // a test of the failure path: the first group is never fetched, so the waits for it run out
            const bool drop_first = (status->debug_flags & EVO_DEBUG_DROP_COMPLETION) != 0u;
            asm volatile("griddepcontrol.wait;" ::: "memory");          // the activations are complete and visible
            for (uint32_t j = 0; j < n_mine; ++j) {
                const uint32_t slot = j % kC2Ring;
                if (j >= kC2Ring) c2_wait(S, &S.a_free[slot], (j / kC2Ring - 1u) & 1u, status);
                // the first groups one after the other, so that memory serves every block's first group
                // (and its weights) before anyone's second
                else if (j >= 1u) c2_wait(S, &S.a_full[j - 1u], 0u, status);
                if (S.abort) break;
                if (drop_first && j == 0u) continue;
                bulk_copy_g2s(smem_u32(S.a[slot]), src + static_cast<size_t>(j) * kGroupBytes, kGroupBytes, smem_u32(&S.a_full[slot]));
                issued = j + 1u;
            }
            // no copy may still be in flight when the block ends (only a time-out leaves any unconsumed)
            for (uint32_t slot = 0; slot < kC2Ring; ++slot)
                if (issued > slot) {
                    const uint32_t n_slot = (issued - slot + kC2Ring - 1u) / kC2Ring;     // copies into this slot
                    mbar_wait_bounded(smem_u32(&S.a_full[slot]), (n_slot - 1u) & 1u, &status->wait_cycles_log2);
                }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        // the accumulator warps have waited for every unit's MMAs; after a time-out some may still run
        if (lane == 0) mbar_wait_bounded(smem_u32(&S.drain), 0u, &status->wait_cycles_log2);
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// fitness[m] = -mean over the batch of the per-image losses: one block per member, fixed order
// (thread t adds images t, t + 256, ...; then a tree over the threads)
__global__ void __launch_bounds__(256)
k_cnn_tc_finalize(const float* __restrict__ loss, uint32_t batch, float* __restrict__ fitness)
{
    __shared__ float red[256];
    dep_wait();                                                         // the losses are complete and visible
    dep_trigger();                                                      // the ranking that follows may be set up
    const uint32_t m = blockIdx.x;
    float s = 0.f;
    for (uint32_t i = threadIdx.x; i < batch; i += 256u) s += loss[static_cast<size_t>(m) * batch + i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (uint32_t off = 128u; off > 0u; off >>= 1) {
        if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) fitness[m] = -red[0] / static_cast<float>(batch);
}

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------
size_t cnn_tc_scratch_bytes(uint32_t P, uint32_t batch)
{
    const size_t n_groups = (batch + 15u) / 16u;
    size_t b = (static_cast<size_t>(P) * batch * sizeof(float) + 255) / 256 * 256;      // per-image losses
    b += static_cast<size_t>(P) * n_groups * kGroupBytes;                  // pooled-1 activations
    return b;
}

int launch_rollout_cnn_tc(cudaStream_t st, const float* theta, uint32_t ldD, uint32_t P, const float* images,
                          const int32_t* labels, uint32_t batch, void* scratch, float* fitness,
                          DeviceStatus* status)
{
    static int sm_count = 0;
    if (sm_count == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return -1;
        if (cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
    }
    unsigned char* base = static_cast<unsigned char*>(scratch);
    float* loss = reinterpret_cast<float*>(base);
    unsigned char* pooled1 = base + (static_cast<size_t>(P) * batch * sizeof(float) + 255) / 256 * 256;

    if (cudaFuncSetAttribute(k_cnn_conv1_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kC1DynRequest) != cudaSuccess) return -1;
    const uint32_t n_groups = (batch + 15u) / 16u;
    const uint32_t n_tiles = n_groups * 18u;
    const uint32_t n_member_groups = (P + kC1Group - 1u) / kC1Group;
    dim3 g1(min(max(static_cast<uint32_t>(sm_count) / n_member_groups, 1u), n_tiles), n_member_groups);
    if (launch_dependent(k_cnn_conv1_tc, g1, dim3(kC1Threads), kC1DynRequest, st, theta, ldD, P, images, batch,
                         reinterpret_cast<uint4*>(pooled1), status) != cudaSuccess) return -1;

    const int c2_bytes = static_cast<int>(sizeof(C2Smem));
    if (cudaFuncSetAttribute(k_cnn_conv2_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, c2_bytes) != cudaSuccess) return -1;
    const uint64_t n_units = static_cast<uint64_t>(P) * n_groups;
    const uint32_t g2 = static_cast<uint32_t>(min(n_units, static_cast<uint64_t>(sm_count)));         // one block per SM
    {
        // conv2 may start (its blocks become resident, fetch their filters and build their bands) while the tail
        // of conv1 is still running; it reads no activation before conv1 has completed (griddepcontrol.wait)
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(g2); cfg.blockDim = dim3(kC2Threads); cfg.dynamicSmemBytes = static_cast<size_t>(c2_bytes); cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at; cfg.numAttrs = 1;
        const unsigned char* p1 = pooled1;
        if (cudaLaunchKernelEx(&cfg, k_cnn_conv2_tc, theta, ldD, P, p1, labels, batch, loss, status) != cudaSuccess) return -1;
    }
    {   // likewise a programmatic dependent (of conv2): its launch latency goes under conv2's tail
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(P); cfg.blockDim = dim3(256); cfg.dynamicSmemBytes = 0; cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at; cfg.numAttrs = 1;
        const float* lp = loss;
        if (cudaLaunchKernelEx(&cfg, k_cnn_tc_finalize, lp, batch, fitness) != cudaSuccess) return -1;
    }
    return 3;
}

}  // namespace evo
