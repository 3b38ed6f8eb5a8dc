// Triangle-painting task (paper Section 3, "Concrete and Abstract Painting"): a member is N
// semi-transparent triangles, fitness = minus the mean squared distance between the painted canvas
// and a target image.  The solver is used on its own here (no policy network): the parameter row IS
// the painting.
//
// Conventions: 10 numbers per triangle (x0 y0 x1 y1 x2 y2 r g b a), each mapped to the unit interval
// by u = clamp(0.5 + 0.5 v, 0, 1); canvas = unit square sampled at pixel centres, starting at a
// grey background; triangles composited in order, C <- C + a (c - C).  Which pixels a triangle
// covers is decided in fp32 with singly rounded operations (explicit *_rn intrinsics: no fused
// contraction), so that the decision is the same on every conforming machine: the pixel centre lies
// in the closed bounding box of the vertices and the three edge values
// e = (bx - ax)(py - ay) - (by - ay)(px - ax) are all >= 0 or all <= 0; a triangle without area
// paints nothing.
//
// k_paint: block = (member, a run of 16 x 8 pixel rectangles).  The block turns the member's parameters into
// triangle records in shared memory; after that its four warps are independent.  A warp takes a rectangle at a
// time, 4 adjacent pixels of a row per lane with their colours in registers.  Its lanes first classify 32
// triangles at once against the rectangle: an edge function is linear, so its largest and smallest value over the
// rectangle lie at corners, and a triangle is outside (an edge's largest value is below -kMargin), or an edge is
// passed by the whole rectangle (its smallest value is above kMargin) or has to be tested per pixel.  The margin is several
// times the rounding error of an edge value, so the classes are exact with respect to the fp32 coverage rule above.
// Only the triangles that matter are then walked, in order, from the ballots, with the tests that cut the rectangle; the
// covering ones without any.  Bound by instruction issue (84 %).  64 triangles on 128 x 128 pixels, 1,024 members in
// mid-training: 357 us with tiles of 32 x 16 pixels, a list of the triangles whose bounding box meets the tile and
// every test per pixel; 183 us with the classes; 142 us with the tests per edge; 135 us with only the near triangles classified.
#include "internal.h"

namespace evo {

constexpr int kPaintThreads = 128;
constexpr uint32_t kRectW = 16, kRectH = 8;
constexpr int kPaintMaxTriangles = 512;
constexpr float kMargin = 4e-6f;          // an edge value of points in the unit square is off by less than 1e-6
constexpr float kThin = 2e-5f;            // below this area the three edge values do not tell inside from outside by one sign

// 20 floats: lanes that read consecutive records with 128-bit loads meet no bank conflict
struct PaintTri {
    float4 e[3];                  // x, y of a vertex; x, y of the edge from it, turned so that inside is positive (not if thin)
    float xmin, xmax, ymin, ymax;
    float ar, ag, ab, rest;       // alpha times the colour, 1 - alpha
};
enum : uint8_t { kPaintsNothing = 0, kOrdinary = 1, kThinTriangle = 2 };

__device__ __forceinline__ float paint_unit(float v)
{
    float u = __fmaf_rn(0.5f, v, 0.5f);
    u = (u >= 0.0f) ? u : 0.0f;               // NaN -> 0
    return fminf(u, 1.0f);
}

__device__ __forceinline__ float paint_edge(float ax, float ay, float bx, float by, float px, float py)
{
    const float dx = __fsub_rn(bx, ax), dy = __fsub_rn(by, ay);
    const float qx = __fsub_rn(px, ax), qy = __fsub_rn(py, ay);
    return __fsub_rn(__fmul_rn(dx, qy), __fmul_rn(dy, qx));
}

struct PaintArgs {
    const float* theta; uint32_t ldD, P;
    uint32_t n_tri, W, H;
    float background;
    const float* target;          // [H][W][3]
    float* partial;               // [P][blocks per member] sums of squared differences
    float* canvas;                // nullable: [P][H][W][3]
    uint32_t rects_x, rects, rects_per_block;
};

// NEAR (more than 32 triangles): a warp first lists the triangles whose box overlaps its rectangle, and classifies only these: of 64 triangles of a
// painting on its way 15, one round instead of two.  64 triangles on 128 x 128, 1,024 members 142 -> 135 us; 158 on 61 x 131, 788 members 176 -> 162; 40 on
// 128 x 128, 256 members 35.4 -> 33.4, gathered at the centre 26.0 -> 24.5, uniform over 1.2 times the canvas 37.7 -> 36.3.  Only where nearly every box covers
// the canvas does the list save no round: 40 on 128 x 128 52.3 -> 53.8, 200 196 -> 199.  (Listing only where the boxes' mean share pays, by the last rectangle
// or for the block, takes 6 to 8 registers more and costs every painting 3 to 13 %.)  With 32 triangles and fewer there is one round in either case: 30 on
// 100 x 100, 400 members 29.0 us, with a list 30.3.
template <bool NEAR>
__global__ void __launch_bounds__(kPaintThreads)
k_paint(const PaintArgs a)
{
    // sized by the launch: n_tri records, NEAR: n_tri triangle numbers per warp, then n_tri kinds
    extern __shared__ __align__(16) unsigned char paint_smem[];
    PaintTri* tri = reinterpret_cast<PaintTri*>(paint_smem);
    uint16_t* near = reinterpret_cast<uint16_t*>(paint_smem + sizeof(PaintTri) * a.n_tri) + (threadIdx.x >> 5) * a.n_tri;
    uint8_t* kind = paint_smem + (sizeof(PaintTri) + (NEAR ? kPaintThreads / 32 * sizeof(uint16_t) : 0u)) * a.n_tri;
    __shared__ float warp_sum[kPaintThreads / 32];

    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const uint32_t member = blockIdx.x;
    const float inv_w = __fdiv_rn(1.0f, static_cast<float>(a.W)), inv_h = __fdiv_rn(1.0f, static_cast<float>(a.H));
    const float* p = a.theta + static_cast<size_t>(member) * a.ldD;
    dep_wait();
    dep_trigger();

    for (uint32_t k = tid; k < a.n_tri; k += kPaintThreads) {
        const float2* src = reinterpret_cast<const float2*>(p + k * 10u);     // 40-byte records
        const float2 v0 = __ldg(src), v1 = __ldg(src + 1), v2 = __ldg(src + 2), v3 = __ldg(src + 3), v4 = __ldg(src + 4);
        const float x0 = paint_unit(v0.x), y0 = paint_unit(v0.y), x1 = paint_unit(v1.x), y1 = paint_unit(v1.y);
        const float x2 = paint_unit(v2.x), y2 = paint_unit(v2.y), alpha = paint_unit(v4.y);
        const float area = paint_edge(x0, y0, x1, y1, x2, y2);
        // turning an edge negates its value exactly
        const float s = area <= -kThin ? -1.0f : 1.0f;
        PaintTri t;
        t.e[0] = make_float4(x0, y0, s * __fsub_rn(x1, x0), s * __fsub_rn(y1, y0));
        t.e[1] = make_float4(x1, y1, s * __fsub_rn(x2, x1), s * __fsub_rn(y2, y1));
        t.e[2] = make_float4(x2, y2, s * __fsub_rn(x0, x2), s * __fsub_rn(y0, y2));
        t.xmin = fminf(x0, fminf(x1, x2)); t.xmax = fmaxf(x0, fmaxf(x1, x2));
        t.ymin = fminf(y0, fminf(y1, y2)); t.ymax = fmaxf(y0, fmaxf(y1, y2));
        t.ar = alpha * paint_unit(v3.x); t.ag = alpha * paint_unit(v3.y); t.ab = alpha * paint_unit(v4.x); t.rest = 1.0f - alpha;
        tri[k] = t;
        kind[k] = area == 0.0f || alpha == 0.0f ? kPaintsNothing : fabsf(area) < kThin ? kThinTriangle : kOrdinary;
    }
    __syncthreads();

    float sq = 0.f;
    const uint32_t first = blockIdx.y * a.rects_per_block, last = min(first + a.rects_per_block, a.rects);
    for (uint32_t rect = first + warp; rect < last; rect += kPaintThreads / 32) {
        const uint32_t i0 = (rect % a.rects_x) * kRectW, j0 = (rect / a.rects_x) * kRectH;
        const uint32_t i1 = min(i0 + kRectW, a.W) - 1u, j1 = min(j0 + kRectH, a.H) - 1u;
        // pixel centres at the rectangle's corners
        const float X0 = __fmul_rn(__fadd_rn(static_cast<float>(i0), 0.5f), inv_w), X1 = __fmul_rn(__fadd_rn(static_cast<float>(i1), 0.5f), inv_w);
        const float Y0 = __fmul_rn(__fadd_rn(static_cast<float>(j0), 0.5f), inv_h), Y1 = __fmul_rn(__fadd_rn(static_cast<float>(j1), 0.5f), inv_h);
        const uint32_t prow = j0 + (lane >> 2), col = i0 + (lane & 3u) * 4u;
        const float py = __fmul_rn(__fadd_rn(static_cast<float>(prow), 0.5f), inv_h);
        float px[4], cr[4], cg[4], cb[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            px[q] = __fmul_rn(__fadd_rn(static_cast<float>(col + q), 0.5f), inv_w);
            cr[q] = a.background; cg[q] = a.background; cb[q] = a.background;
        }

        // a pixel centre of the rectangle inside the closed box exists only if the ranges overlap
        auto overlaps = [&](uint32_t k) {
            const float4 box = *reinterpret_cast<const float4*>(&tri[k].xmin);
            return kind[k] != kPaintsNothing && !(box.y < X0 || box.x > X1 || box.w < Y0 || box.z > Y1);
        };
        uint32_t n_tri = a.n_tri;
        if constexpr (NEAR) {                                             // in order
            n_tri = 0;
            __syncwarp();                                                 // everyone is done with the rectangle before
            for (uint32_t base = 0; base < a.n_tri; base += 32u) {
                const uint32_t k = base + lane;
                const bool here = k < a.n_tri && overlaps(k);
                const uint32_t those = __ballot_sync(0xffffffffu, here);
                if (here) near[n_tri + __popc(those & ((1u << lane) - 1u))] = static_cast<uint16_t>(k);
                n_tri += __popc(those);
            }
            __syncwarp();
        }
        for (uint32_t base = 0; base < n_tri; base += 32u) {
            // what the walk has to look at per pixel: the box, each edge, or (thin triangles) the three edges with either sign
            bool walk = false, box_cuts = false, cuts[3] = { false, false, false }, thin = false;
            if (base + lane < n_tri) {
                const uint32_t k = NEAR ? near[base + lane] : base + lane;
                const PaintTri& t = tri[k];
                walk = NEAR || overlaps(k);
                thin = kind[k] == kThinTriangle;
                box_cuts = t.xmin > X0 || t.xmax < X1 || t.ymin > Y0 || t.ymax < Y1;
                if (walk && !thin) {
                    float highest = 1.0f;                             // smallest of the edges' largest values
                    bool any = false;
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        const float4 e = t.e[i];
                        const float ya = e.z * (Y0 - e.y), yb = e.z * (Y1 - e.y), xa = e.w * (X0 - e.x), xb = e.w * (X1 - e.x);
                        highest = fminf(highest, fmaxf(ya, yb) - fminf(xa, xb));
                        cuts[i] = fminf(ya, yb) - fmaxf(xa, xb) <= kMargin;
                        any = any || cuts[i];
                    }
                    walk = highest >= -kMargin;
                    box_cuts = box_cuts && any;                       // inside all edges by the margin is inside the box
                }
            }
            uint32_t todo = __ballot_sync(0xffffffffu, walk);
            const uint32_t boxes = __ballot_sync(0xffffffffu, box_cuts), thins = __ballot_sync(0xffffffffu, thin);
            const uint32_t cut0 = __ballot_sync(0xffffffffu, cuts[0]), cut1 = __ballot_sync(0xffffffffu, cuts[1]),
                           cut2 = __ballot_sync(0xffffffffu, cuts[2]);
            const uint32_t tested = boxes | thins | cut0 | cut1 | cut2;
            while (todo) {
                const uint32_t n = __ffs(static_cast<int>(todo)) - 1u, bit = todo & (0u - todo);
                todo ^= bit;
                const PaintTri& t = tri[NEAR ? near[base + n] : base + n];
                const float4 c = *reinterpret_cast<const float4*>(&t.ar);
                if (!(tested & bit)) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        cr[q] = fmaf(c.w, cr[q], c.x); cg[q] = fmaf(c.w, cg[q], c.y); cb[q] = fmaf(c.w, cb[q], c.z);
                    }
                    continue;
                }
                float lo[4] = { 0.f, 0.f, 0.f, 0.f };                 // inside: >= 0
                auto edge = [&](const float4 e, float* f) {
                    const float ty = __fmul_rn(e.z, __fsub_rn(py, e.y));
#pragma unroll
                    for (int q = 0; q < 4; ++q) f[q] = __fsub_rn(ty, __fmul_rn(e.w, __fsub_rn(px[q], e.x)));
                };
                if (thins & bit) {
                    float f0[4], f1[4], f2[4];
                    edge(t.e[0], f0); edge(t.e[1], f1); edge(t.e[2], f2);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float least = fminf(f0[q], fminf(f1[q], f2[q])), most = fmaxf(f0[q], fmaxf(f1[q], f2[q]));
                        lo[q] = fmaxf(least, -most);
                    }
                } else {
                    float f[4];
                    if (cut0 & bit) {
                        edge(t.e[0], f);
#pragma unroll
                        for (int q = 0; q < 4; ++q) lo[q] = f[q];
                    }
                    if (cut1 & bit) {
                        edge(t.e[1], f);
#pragma unroll
                        for (int q = 0; q < 4; ++q) lo[q] = fminf(lo[q], f[q]);
                    }
                    if (cut2 & bit) {
                        edge(t.e[2], f);
#pragma unroll
                        for (int q = 0; q < 4; ++q) lo[q] = fminf(lo[q], f[q]);
                    }
                }
                if (boxes & bit) {
                    const float4 box = *reinterpret_cast<const float4*>(&t.xmin);
                    const bool in_rows = py >= box.z && py <= box.w;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (!(in_rows && px[q] >= box.x && px[q] <= box.y)) lo[q] = -1.0f;
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (lo[q] >= 0.0f) {
                        cr[q] = fmaf(c.w, cr[q], c.x); cg[q] = fmaf(c.w, cg[q], c.y); cb[q] = fmaf(c.w, cb[q], c.z);
                    }
            }
        }

        // squared distance to the target
        if (prow < a.H) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (col + q < a.W) {
                    const size_t at = (static_cast<size_t>(prow) * a.W + col + q) * 3u;
                    const float d0 = cr[q] - __ldg(a.target + at), d1 = cg[q] - __ldg(a.target + at + 1), d2 = cb[q] - __ldg(a.target + at + 2);
                    sq += d0 * d0 + d1 * d1 + d2 * d2;
                    if (a.canvas) {
                        float* out = a.canvas + static_cast<size_t>(member) * a.W * a.H * 3u + at;
                        out[0] = cr[q]; out[1] = cg[q]; out[2] = cb[q];
                    }
                }
            }
        }
    }
    // fixed-order sum of the block
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
    if (lane == 0) warp_sum[warp] = sq;
    __syncthreads();
    if (tid == 0) {
        float total = 0.f;
        for (int w = 0; w < kPaintThreads / 32; ++w) total += warp_sum[w];
        a.partial[static_cast<size_t>(member) * gridDim.y + blockIdx.y] = total;
    }
}

__global__ void k_paint_finalize(const float* __restrict__ partial, uint32_t P, uint32_t tiles, float inv_count,
                                 float* __restrict__ fitness)
{
    dep_wait();
    dep_trigger();
    const uint32_t m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= P) return;
    float s = 0.f;
    for (uint32_t t = 0; t < tiles; ++t) s += partial[static_cast<size_t>(m) * tiles + t];
    fitness[m] = -s * inv_count;
}

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------
struct PaintSplit { uint32_t rects_x, rects, per_block, blocks; };

// A block builds the member's records, so it should have some rectangles to use them on; about 24 blocks per SM in all even
// out what the rectangles of a painting differ by.
static PaintSplit paint_split(uint32_t P, uint32_t W, uint32_t H)
{
    PaintSplit s;
    s.rects_x = (W + kRectW - 1u) / kRectW;
    s.rects = s.rects_x * ((H + kRectH - 1u) / kRectH);
    const uint64_t share = static_cast<uint64_t>(s.rects) * P / (kSms * 24u);
    s.per_block = share < 4u ? 4u : share > s.rects ? (s.rects + 3u) / 4u * 4u : static_cast<uint32_t>(share) / 4u * 4u;
    s.blocks = (s.rects + s.per_block - 1u) / s.per_block;
    return s;
}

bool paint_supported(uint32_t param_dim, uint32_t W, uint32_t H)
{
    return param_dim % 10u == 0 && param_dim / 10u >= 1 && param_dim / 10u <= kPaintMaxTriangles &&
           W >= 1 && H >= 1 && W <= 4096 && H <= 4096;
}

size_t paint_scratch_bytes(uint32_t P, uint32_t W, uint32_t H)
{
    return static_cast<size_t>(P) * paint_split(P, W, H).blocks * sizeof(float);
}

int launch_rollout_paint(cudaStream_t st, const float* theta, uint32_t ldD, uint32_t P, uint32_t param_dim,
                         uint32_t W, uint32_t H, float background, const float* target, void* scratch,
                         float* fitness, float* canvas)
{
    const PaintSplit s = paint_split(P, W, H);
    PaintArgs a;
    a.theta = theta; a.ldD = ldD; a.P = P; a.n_tri = param_dim / 10u; a.W = W; a.H = H;
    a.background = background; a.target = target; a.partial = static_cast<float*>(scratch); a.canvas = canvas;
    a.rects_x = s.rects_x; a.rects = s.rects; a.rects_per_block = s.per_block;
    const bool near = a.n_tri > 32u;
    const size_t smem = (sizeof(PaintTri) + (near ? kPaintThreads / 32 * sizeof(uint16_t) : 0u) + sizeof(uint8_t)) * a.n_tri;        // at most 45 KB
    if (launch_dependent(near ? k_paint<true> : k_paint<false>, dim3(P, s.blocks), dim3(kPaintThreads), smem, st, a) != cudaSuccess) return -1;
    const float inv = 1.0f / (3.0f * static_cast<float>(W) * static_cast<float>(H));
    if (launch_dependent(k_paint_finalize, dim3((P + 255u) / 256u), dim3(256), 0, st, a.partial, P, s.blocks, inv, fitness) != cudaSuccess)
        return -1;
    return 2;
}

}  // namespace evo
