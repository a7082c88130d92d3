// Front-to-back alpha compositing (Section 3.2, Eq. 4) and its reverse.  Both
// evaluate vertically adjacent pixels in pairs, in packed FP32, on a tile's
// depth-sorted records staged through shared memory.  The arithmetic of a
// pixel is written with explicit roundings so that both passes, and every
// way of cutting the work, take bit-identical decisions.
#include "common.cuh"

namespace gs3 {

constexpr int NT = 128;          // threads of a forward block (one 16x16 tile): two pixels each

struct RasterParams {
    const float2 *mean2d;
    const float4 *conic_op;
    const float *rgb;
    const int32_t *radius;
    const uint32_t *vals;
    const uint2 *ranges;
    int64_t n;
    int V, W, H, tx, ty, bin, bins_x, bins;
    float bg0, bg1, bg2;
    float *img;
    float *T_final;
    int32_t *last;
    // backward
    const float *d_img;
    float *grads;
    float *d_opacity;
    unsigned long long *stats;  // optional: [tested, contributing] (pixel, Gaussian) pairs
    // optional per-tile lists of staged records (Gaussian, list position):
    // written by the forward, read by the reverse
    uint2 *tl_rec;
    int32_t *tl_cnt;
    int tl_cap;
};

// Add this thread's pair counts to the optional statistics words.
__device__ __forceinline__ void flush_stats(unsigned long long *stats, uint32_t tested,
                                            uint32_t contrib)
{
    if (!stats) return;
    unsigned long long a = tested, b = contrib;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(stats, a);
        atomicAdd(stats + 1, b);
    }
}

// The staged conic is scaled by log2(e) (scale_conic), so the power comes in
// base-2 units and G = 2^power from one ex2.approx; alpha and dL/dpower keep
// their natural-unit meaning.
constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;

__device__ __forceinline__ float4 scale_conic(float4 co)
{
    return make_float4(co.x * kLog2e, co.y * kLog2e, co.z * kLog2e, co.w);
}

// G = 2^power.
__device__ __forceinline__ float pair_gauss(float power)
{
    float g;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(g) : "f"(power));
    return g;
}

constexpr float kAlphaCap = 0.99f;
constexpr float kTEps = 1e-4f;

// alpha >= 1/255 (Eq. 4's skip) is tested on the base-2 power, -power <=
// log2(255 o) staged with the record: forward and reverse take the same
// decision, which differs from the test on alpha only within the rounding of
// the exponential.  Only records with 255 o >= 1 are staged.  A logarithm
// that rounds below 0, or to -0, at 255 o = 1 counts as +0, so that the
// threshold's bit pattern is below those of every negative number and NaN.
__device__ __forceinline__ bool visible(float o) { return o * 255.f >= 1.f; }
__device__ __forceinline__ float staged_threshold(float o) { return fmaxf(__log2f(255.f * o), 0.f); }

// Can record (m, co) reach alpha >= 1/255 at some pixel centre of tile
// (tx_t, ty_t)?  alpha = o exp(-q/2) with q = A dx^2 + 2B dx dy + C dy^2, so
// it needs q <= 2 ln(255 o) somewhere in the tile.  The minimum of the convex
// q over the tile's rectangle of pixel centres is 0 when the mean lies inside,
// else it is on an edge, where q is a 1-D quadratic minimised in closed form.
// A margin of 0.01 in q (far above FP32 rounding) keeps the test
// conservative: a dropped record is one every pixel of the tile would skip,
// so images, gradients and list positions are unchanged.
__device__ __forceinline__ bool ellipse_hits_tile(float2 m, float4 co, int tx_t, int ty_t)
{
    if (!visible(co.w)) return false;
    const float tau = 2.f * __logf(255.f * co.w) + 0.01f;
    const float xa = (float)(tx_t * 16) + 0.5f - m.x, xb = xa + 15.f;
    const float ya = (float)(ty_t * 16) + 0.5f - m.y, yb = ya + 15.f;
    if (xa <= 0.f && xb >= 0.f && ya <= 0.f && yb >= 0.f) return true;
    const float A = co.x, B = co.y, C = co.z;
    // the 1-D minimisers need not be exact: q at any point of an edge bounds
    // its minimum from above, and a minimiser off by a rounding moves q by a
    // second-order amount, far inside the margin
    const float bA = B * __frcp_rn(A), bC = B * __frcp_rn(C);
    auto qx = [&](float dx) {  // min over dy in [ya, yb] at fixed dx
        float dy = fminf(fmaxf(-bC * dx, ya), yb);
        return A * dx * dx + 2.f * B * dx * dy + C * dy * dy;
    };
    auto qy = [&](float dy) {  // min over dx in [xa, xb] at fixed dy
        float dx = fminf(fmaxf(-bA * dy, xa), xb);
        return A * dx * dx + 2.f * B * dx * dy + C * dy * dy;
    };
    float q = fminf(fminf(qx(xa), qx(xb)), fminf(qy(ya), qy(yb)));
    return q <= tau;
}

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }

__device__ __forceinline__ void cp_async4(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Forward: one 16x16 tile per 128-thread block, two vertically adjacent pixels
// a thread evaluated as a pair in packed FP32.  It is bound by instruction
// issue (76 % of the slots, the ALU pipe busiest) where there are many tiles,
// and by the chain of a tile's batches where there are few.  The batches
// therefore run as a pipeline with one barrier each: while a batch of staged
// records is composited, the next batch's candidates are in flight to
// registers (their indices one batch earlier) and the colours of the records
// just kept to shared memory (cp.async).  250K Gaussians and four 1352x1014
// views / 50K and eight 480x360 / 49K and one 477x363 view: 523 / 189 / 67 us.
// Measured slower: a batch that waits for its indices, records and colours in
// turn, behind three barriers (575 / 235 / 94 us), four pixels a lane as in the
// reverse (676 / 272 / 95 us: it needs 120 registers, and fewer warps hide
// less), records culled per warp (576 / 204 / 65 us), two candidates a thread
// per batch (745 / 255 / 78 us at 64 registers), no per-lane skip of records
// (548 / 223 / 78 us).
constexpr int FWD_UNROLL = 4;

struct FwdBatch {
    float4 xyt[NT];    // mean, threshold power
    float4 co[NT];     // conic in base-2 units, opacity
    float4 rgbk[NT];   // colour and (bit pattern of) 1 + the list position
};

struct PixFwd2 {
    float2 y, T, C0, C1, C2;
    int last0, last1;
    int alive;   // bit k: pixel k has not stopped
    int stop;    // number of staged records up to the last stop
};

// One staged record (number `staged` of the tile's list) at the thread's two
// pixels; a pixel takes part when its negated power is in [0, threshold] (see
// bwd_chunk).
template <bool STATS>
__device__ __forceinline__ void fwd_record(PixFwd2 &P, float4 xyt, float4 co, const float4 &rgbk, float pxf, int staged,
                                           uint32_t &n_tested, uint32_t &n_contrib)
{
    const uint32_t thr = __float_as_uint(xyt.z);
    const float dx = __fsub_rn(pxf, xyt.x);
    const float axx = __fmul_rn(co.x, __fmul_rn(dx, dx));
    const float2 dy = __fadd2_rn(P.y, f2(-xyt.y));
    const float2 q = __ffma2_rn(f2(co.z), __fmul2_rn(dy, dy), f2(axx));
    const float2 np = __ffma2_rn(f2(0.5f), q, __fmul2_rn(f2(co.y), __fmul2_rn(f2(dx), dy)));
    bool in0 = __float_as_uint(np.x) <= thr, in1 = __float_as_uint(np.y) <= thr;
    if (STATS) n_tested += __popc(P.alive);
    if (!(in0 || in1)) return;
    float2 alpha = __fmul2_rn(f2(co.w), make_float2(pair_gauss(-np.x), pair_gauss(-np.y)));
    alpha.x = fminf(kAlphaCap, in0 ? alpha.x : 0.f);
    alpha.y = fminf(kAlphaCap, in1 ? alpha.y : 0.f);
    float2 T = __fmul2_rn(P.T, __ffma2_rn(alpha, f2(-1.f), f2(1.f)));
    if (fminf(T.x, T.y) < kTEps) {
        // a pixel stops before this record (its T stays >= 1e-4 otherwise, so
        // only a pixel that takes part can get here); its y becomes NaN, which
        // no later record passes.  The empty asm keeps this a branch.
        asm volatile("" ::: "memory");
        const float nan = __int_as_float(0x7fc00000);
        if (T.x < kTEps) {
            alpha.x = 0.f;
            T.x = P.T.x;
            P.y.x = nan;
            in0 = false;
            P.alive &= ~1;
        }
        if (T.y < kTEps) {
            alpha.y = 0.f;
            T.y = P.T.y;
            P.y.y = nan;
            in1 = false;
            P.alive &= ~2;
        }
        P.stop = staged;
    }
    const float2 w = __fmul2_rn(alpha, P.T);
    P.C0 = __ffma2_rn(f2(rgbk.x), w, P.C0);
    P.C1 = __ffma2_rn(f2(rgbk.y), w, P.C1);
    P.C2 = __ffma2_rn(f2(rgbk.z), w, P.C2);
    P.T = T;
    const int k1 = __float_as_int(rgbk.w);
    P.last0 = in0 ? k1 : P.last0;
    P.last1 = in1 ? k1 : P.last1;
    if (STATS) n_contrib += (uint32_t)in0 + (uint32_t)in1;
}

// 9 blocks per SM: 54 registers without spills (8: 529 / 200 us without the
// per-lane skip; 10: 48 registers, 562 us)
template <bool BINNED, bool STATS>
__global__ void __launch_bounds__(NT, 9) raster_fwd_kernel(RasterParams p)
{
    if (grid_wait()) return;
    __shared__ FwdBatch s_batch[2];
    __shared__ int s_wcnt[2][NT / 32];
    __shared__ int s_count;
    constexpr unsigned all = 0xffffffffu;
    const int tile = blockIdx.x, view = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx_t = tile % p.tx, ty_t = tile / p.tx;
    // a warp owns a compact 8x8 block, whose pixels tend to share records and list ends
    const int px = tx_t * 16 + (warp & 1) * 8 + (lane & 7), py0 = ty_t * 16 + (warp >> 1) * 8 + (lane >> 3) * 2;
    const bool pix0 = px < p.W && py0 < p.H, pix1 = px < p.W && py0 + 1 < p.H;
    const float pxf = (float)px + 0.5f;
    const int binid = (ty_t / p.bin) * p.bins_x + tx_t / p.bin;
    const uint2 range = p.ranges[(int64_t)view * p.bins + binid];
    const int total = (int)(range.y - range.x);
    const int64_t vb = (int64_t)view * p.n;
    const int64_t tg = (int64_t)view * gridDim.x + tile;   // the tile's list
    const float nan = __int_as_float(0x7fc00000);
    PixFwd2 P;
    P.y = make_float2(pix0 ? (float)py0 + 0.5f : nan, pix1 ? (float)py0 + 1.5f : nan);
    P.T = f2(1.f);
    P.C0 = P.C1 = P.C2 = f2(0.f);
    P.last0 = P.last1 = 0;
    P.alive = (int)pix0 | ((int)pix1 << 1);
    P.stop = 0;
    if (tid == 0) s_count = 0;
    uint32_t n_tested = 0, n_contrib = 0;
    // the thread's candidate of the batch to be tested, and the index of the one after
    uint32_t g = 0, g_next = 0;
    int r;
    float2 m;
    float4 co;
    auto load_index = [&](int k) { return k < total ? p.vals[range.x + k] : 0u; };
    auto load_record = [&](int k) {
        const bool ok = k < total;
        r = ok ? (BINNED ? p.radius[vb + g] : 1) : 0;
        m = ok ? p.mean2d[vb + g] : make_float2(0.f, 0.f);
        co = ok ? p.conic_op[vb + g] : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    auto composite = [&](const FwdBatch &B, int cnt, int first) {
        int j = 0;
        for (; j + FWD_UNROLL <= cnt && P.alive; j += FWD_UNROLL) {
#pragma unroll
            for (int i = 0; i < FWD_UNROLL; ++i)
                fwd_record<STATS>(P, B.xyt[j + i], B.co[j + i], B.rgbk[j + i], pxf, first + j + i + 1, n_tested,
                                  n_contrib);
        }
        for (; j < cnt && P.alive; ++j)
            fwd_record<STATS>(P, B.xyt[j], B.co[j], B.rgbk[j], pxf, first + j + 1, n_tested, n_contrib);
    };
    g = load_index(tid);
    load_record(tid);
    g_next = load_index(NT + tid);
    int staged = 0, prev = 0, buf = 0;   // records staged so far, those of the batch before
    bool open = true;
    for (int base = 0; base < total; base += NT, buf ^= 1) {
        const int k = base + tid;
        bool keep = r > 0;
        if (BINNED && keep) {
            int x0, y0, x1, y1;
            tile_rect(m.x, m.y, r, p.tx, p.ty, x0, y0, x1, y1);
            keep = tx_t >= x0 && tx_t < x1 && ty_t >= y0 && ty_t < y1;
        }
        keep = keep && ellipse_hits_tile(m, co, tx_t, ty_t);
        const unsigned kept = __ballot_sync(all, keep);
        if (lane == 0) s_wcnt[buf][warp] = __popc(kept);
        // the barrier of the batch: its counts and the batch before's records
        // and colours are there, and buffer `buf` (two batches ago) is free
        cp_async_wait();
        if (!__syncthreads_or(P.alive)) {
            open = false;
            break;
        }
        int off = 0, cnt = 0;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) {
            const int c = s_wcnt[buf][w];
            off += w < warp ? c : 0;
            cnt += c;
        }
        if (keep) {
            const int slot = off + __popc(kept & ((1u << lane) - 1u));
            if (p.tl_rec && staged + slot < p.tl_cap)
                p.tl_rec[tg * p.tl_cap + staged + slot] = make_uint2(g, (uint32_t)k);
            FwdBatch &B = s_batch[buf];
            B.xyt[slot] = make_float4(m.x, m.y, staged_threshold(co.w), 0.f);
            B.co[slot] = scale_conic(co);
            float *c = &B.rgbk[slot].x;
            const float *src = p.rgb + 3 * (vb + g);
            cp_async4(c, src);
            cp_async4(c + 1, src + 1);
            cp_async4(c + 2, src + 2);
            c[3] = __int_as_float(k + 1);
        }
        g = g_next;
        load_record(k + NT);
        g_next = load_index(k + 2 * NT);
        composite(s_batch[buf ^ 1], prev, staged - prev);
        prev = cnt;
        staged += cnt;
    }
    if (open) {
        cp_async_wait();
        __syncthreads();
        composite(s_batch[buf ^ 1], prev, staged - prev);
    }
    if (STATS) flush_stats(p.stats, n_tested, n_contrib);
    if (p.tl_rec) {
        // records past every pixel's stop took part at no pixel (their
        // positions are at or past every pixel's last): the list ends before
        // them
        const int mine = __reduce_max_sync(all, P.alive ? staged : P.stop);
        if (lane == 0 && mine > 0) atomicMax(&s_count, mine);
        __syncthreads();
        if (tid == 0) p.tl_cnt[tg] = s_count <= p.tl_cap ? s_count : -1;
    }
    const int64_t HW = (int64_t)p.H * p.W;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (!(q == 0 ? pix0 : pix1)) continue;
        const float T = q ? P.T.y : P.T.x;
        const int64_t pix = (int64_t)(py0 + q) * p.W + px;
        float *im = p.img + (int64_t)view * 3 * HW + pix;
        im[0] = fmaf(T, p.bg0, q ? P.C0.y : P.C0.x);
        im[HW] = fmaf(T, p.bg1, q ? P.C1.y : P.C1.x);
        im[2 * HW] = fmaf(T, p.bg2, q ? P.C2.y : P.C2.x);
        p.T_final[(int64_t)view * HW + pix] = T;
        p.last[(int64_t)view * HW + pix] = q ? P.last1 : P.last0;
    }
}

// ------------------------------------------------------------------ reverse
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Reverse: one warp per 8x16 half of a tile, four vertically adjacent pixels a
// lane as NP = 2 packed pairs (or 8x8 and NP = 1, see kFewTiles), no barrier
// anywhere; the warps of a block share nothing.  What bounds it is the pair
// arithmetic (FMA pipe 55 %, 62 % of the issue slots) and, at small images, the
// longest tile.  Why it is cut this way (250K Gaussians, four 1352x1014 views /
// 50K, eight 480x360 views, one launch, by CUPTI: 646 / 184 us):
//  - the sums over pixels are taken with the lanes turned.  While a chunk of
//    BWD_CHUNK records is walked, lane = pixel column, and each lane leaves
//    the sums over its own four pixels (of dL/dpower times 1, dy, dy^2 and of
//    the colour gradient) in shared memory; then lane = (record, pixels), and
//    four lanes add up a record's 32 columns.  A shuffle butterfly per record
//    for each pixel pair, summed over a tile's warps behind two barriers a
//    chunk, takes half of a kernel's instructions (922 / 293 us).
//  - each warp keeps, of the tile's list, the records that can reach its own
//    half (staged_hits).
//  - four pixels a lane share a record's loads and column offset: two pixels
//    a lane (8x8 per warp) run into the shared-memory pipe (79 % of its
//    wavefronts) where there are many tiles, 725 us against 640.
//  - no branch on "no lane takes part": the records of a chunk run as one
//    straight line, so that their independent parts overlap (715 -> 667 us).
//  - with NP = 1 a batch's list entries are loaded one batch ahead, and the
//    colours with the means instead of after the test (82 -> 76 us for 4K
//    Gaussians in four 128x96 views; nothing to gain with NP = 2).
//  - tiles whose list is long go first (kHeavyList).
constexpr int BWD_WARPS = 4;                 // warps of a block (two tiles); 1, 2 and 4 measured within 2 %
constexpr int BWD_CHUNK = 8;                 // records of a turned sum
constexpr int BWD_ROW = 36;                  // lanes' places of a record: two records of a quarter warp meet different banks
constexpr int BWD_QUEUE = 32 + BWD_CHUNK;    // staged records of a warp: a batch and what was left of the one before
constexpr int BWD_TEST = 128;                // records of a bin's list tested at a time (tiles without a list)
// A block that walks one long list alone at the end of the launch keeps the
// other SMs waiting, so the grid has two layers: the first takes the tiles
// with at least this many records (and those without a list), the second the
// others; a block of the other kind returns at once.  Lists of the headline
// workload: median 70, 90 % below 219, longest over 1 000.  50K Gaussians in
// 480x360 views 241 -> 205 us, the headline batch 666 -> 662 us (192: 218 /
// 665, 384: 212 / 685).
constexpr int kHeavyList = 256;

template <int NP>
struct PixBwd {
    int last[2 * NP];
    float2 T[NP], dC0[NP], dC1[NP], dC2[NP], nS[NP];   // nS: minus dL/dC . (colour behind)
};

// Up to this many tiles per SM, in all views, a warp takes 8x8 pixels: twice
// the warps with little more than half the instructions per record each, for
// launches that end with a few long lists on an idle chip.  4K Gaussians, four
// 128x96 views (192 tiles) 129 -> 76 us; 50K, eight 480x360 views (5 520) 207
// -> 184 us; 250K, one 1352x1014 view (5 440) 154 -> 158 us; 1M, one 1920x1080
// view (8 160) 262 -> 295 us; 250K, two 1352x1014 views (10 880) 352 -> 390 us;
// 50K, sixteen 480x360 views (11 040) 368 -> 348 us.  What decides is how long
// the longest lists are against the work of all, which the host does not know:
// by tiles alone one 1352x1014 view is on the wrong side by 4 us and sixteen
// 480x360 views by 20.
constexpr int kFewTiles = 40;

struct BwdWarp {
    float4 sum4[BWD_CHUNK][BWD_ROW];   // per record and lane, over its pixels: S, S_y, S_yy, red
    float2 sum2[BWD_CHUNK][BWD_ROW];   // green, blue
    float4 xyt[BWD_QUEUE];             // mean, threshold power, list position
    float4 co[BWD_QUEUE];              // conic in base-2 units, and minus the opacity
    float4 rgbg[BWD_QUEUE];            // colour, Gaussian
    uint2 cand[BWD_TEST + 32];         // tiles without a list: records whose rectangle holds the tile
};

// Can a staged record reach alpha >= 1/255 at some centre of the 8 x 8 NP
// pixels from (cx, cy) on?  As ellipse_hits_tile, in the staged units (the negated
// power, base 2), with the evaluation's rounding taken off the form:
// a record dropped here is one that every pixel of the warp skips.
template <int NP>
__device__ __forceinline__ bool staged_hits(float4 xyt, float4 co, float cx, float cy)
{
    const float tau = xyt.z + 0.0075f;
    const float xa = cx - xyt.x, xb = xa + 7.f, ya = cy - xyt.y, yb = ya + (8.f * NP - 1.f);
    if (xa <= 0.f && xb >= 0.f && ya <= 0.f && yb >= 0.f) return true;
    const float A = 0.5f * co.x, B = co.y, C = 0.5f * co.z;   // A dx^2 + B dx dy + C dy^2
    const float bA = 0.5f * B * __frcp_rn(A), bC = 0.5f * B * __frcp_rn(C);
    auto form = [&](float dx, float dy) {
        const float s = A * dx * dx + C * dy * dy;
        return fmaf(-1e-6f, s, fmaf(B * dx, dy, s));
    };
    auto qx = [&](float dx) { return form(dx, fminf(fmaxf(-bC * dx, ya), yb)); };
    auto qy = [&](float dy) { return form(fminf(fmaxf(-bA * dy, xa), xb), dy); };
    return fminf(fminf(qx(xa), qx(xb)), fminf(qy(ya), qy(yb))) <= tau;
}

// Weight times dL/dC.  GUARD: a pixel that takes no part (weight 0) gives 0
// even where its dL/dC is not finite.
template <bool GUARD>
__device__ __forceinline__ float2 weigh(float2 w, float2 d)
{
    return GUARD ? make_float2(w.x == 0.f ? 0.f : w.x * d.x, w.y == 0.f ? 0.f : w.y * d.y) : __fmul2_rn(w, d);
}
template <bool GUARD>
__device__ __forceinline__ float2 weigh(float2 w, float2 d, float2 a)
{
    return GUARD ? __fadd2_rn(a, weigh<true>(w, d)) : __ffma2_rn(w, d, a);
}

// The chunk's cnt records from slot `head` on at the warp's pixels, back to
// front (slots past cnt hold records that take part nowhere), and their
// gradients added to p.grads.
//
// power is carried negated, np = (A dx^2 + C dy^2) / 2 + B dx dy, with the
// forward's roundings (negation is exact; the sum is written as a fused
// multiply-add by 0.5 because the compiler contracts a packed product and a
// packed sum, which would round, and decide, differently).  A pixel takes part
// when np is in [0, threshold]: one unsigned comparison of the bit patterns,
// which a negative or NaN np fails.  A pixel that takes no part gets
// alpha = 0 and no difference, which leaves its transmittance, its
// colour-behind term and the sums exactly as they are.
//
// Record gradients from the moments: with power = -(A dx^2 + C dy^2) / 2 -
// B dx dy and dx = px - u,
//   dL/du = A S_x + B S_y,  dL/dv = C S_y + B S_x,
//   dL/dA = -S_xx / 2,  dL/dB = -S_xy,  dL/dC = -S_yy / 2,
// S_. = sum of dL/dpower times the offsets' monomials; the sums below are of
// -dL/dpower and of minus the weight.
template <int NP, bool WANT_OP, bool STATS, bool GUARD>
__device__ __forceinline__ void bwd_chunk(const RasterParams &p, BwdWarp &S, PixBwd<NP> &P, int head, int cnt, float pxf,
                                          const float2 (&pyf)[NP], float cx0, int64_t vb, uint32_t &n_contrib)
{
    constexpr unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31;
#pragma unroll 4
    for (int i = 0; i < BWD_CHUNK; ++i) {
        const float4 xyt = S.xyt[head + i];
        const float4 co = S.co[head + i];
        const float4 c = S.rgbg[head + i];
        const int pos = __float_as_int(xyt.w);
        const uint32_t thr = __float_as_uint(xyt.z);
        const float dx = __fsub_rn(pxf, xyt.x);
        const float axx = __fmul_rn(co.x, __fmul_rn(dx, dx));
        float2 dy[NP], dyy[NP], nd[NP], nw[NP];
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            dy[h] = __fadd2_rn(pyf[h], f2(-xyt.y));
            dyy[h] = __fmul2_rn(dy[h], dy[h]);
            const float2 q = __ffma2_rn(f2(co.z), dyy[h], f2(axx));
            const float2 np = __ffma2_rn(f2(0.5f), q, __fmul2_rn(f2(co.y), __fmul2_rn(f2(dx), dy[h])));
            const bool in0 = pos < P.last[2 * h] && __float_as_uint(np.x) <= thr;
            const bool in1 = pos < P.last[2 * h + 1] && __float_as_uint(np.y) <= thr;
            if (STATS) n_contrib += (uint32_t)in0 + (uint32_t)in1;
            // minus alpha, before and after the cap
            float2 raw = __fmul2_rn(f2(co.w), make_float2(pair_gauss(-np.x), pair_gauss(-np.y)));
            raw.x = in0 ? raw.x : 0.f;
            raw.y = in1 ? raw.y : 0.f;
            const float2 na = make_float2(fmaxf(-kAlphaCap, raw.x), fmaxf(-kAlphaCap, raw.y));
            const float2 om = __fadd2_rn(na, f2(1.f));
            P.T[h] = __fmul2_rn(P.T[h], make_float2(rcp_approx(om.x), rcp_approx(om.y)));
            nw[h] = __fmul2_rn(na, P.T[h]);
            float2 t = __fmul2_rn(P.dC0[h], f2(c.x));
            t = __ffma2_rn(P.dC1[h], f2(c.y), t);
            t = __ffma2_rn(P.dC2[h], f2(c.z), t);
            float2 diff = __fadd2_rn(t, P.nS[h]);   // dC . c - S
            diff.x = in0 ? diff.x : 0.f;
            diff.y = in1 ? diff.y : 0.f;
            P.nS[h] = __ffma2_rn(na, diff, P.nS[h]);
            nd[h] = __fmul2_rn(__fmul2_rn(P.T[h], diff), na);
            if (co.w <= -kAlphaCap) {   // no gradient through a capped alpha
                if (!(raw.x > -kAlphaCap)) nd[h].x = 0.f;
                if (!(raw.y > -kAlphaCap)) nd[h].y = 0.f;
            }
        }
        float2 s = nd[0], sy = __fmul2_rn(nd[0], dy[0]), syy = __fmul2_rn(nd[0], dyy[0]);
        float2 r = weigh<GUARD>(nw[0], P.dC0[0]), g = weigh<GUARD>(nw[0], P.dC1[0]), b = weigh<GUARD>(nw[0], P.dC2[0]);
        if (NP == 2) {
            constexpr int q = NP - 1;
            s = __fadd2_rn(s, nd[q]);
            sy = __ffma2_rn(nd[q], dy[q], sy);
            syy = __ffma2_rn(nd[q], dyy[q], syy);
            r = weigh<GUARD>(nw[q], P.dC0[q], r);
            g = weigh<GUARD>(nw[q], P.dC1[q], g);
            b = weigh<GUARD>(nw[q], P.dC2[q], b);
        }
        S.sum4[i][lane] = make_float4(s.x + s.y, sy.x + sy.y, syy.x + syy.y, r.x + r.y);
        S.sum2[i][lane] = make_float2(g.x + g.y, b.x + b.y);
    }
    __syncwarp();
    // lane = (record tr, columns th and th + 4)
    const int tr = lane >> 2, th = lane & 3, j = head + tr;
    const float4 xyt = S.xyt[j];
    const float4 co = S.co[j];
    float s0 = 0.f, sx = 0.f, sy = 0.f, sxx = 0.f, sxy = 0.f, syy = 0.f, r = 0.f;
    float2 gb = f2(0.f);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        float2 a = f2(0.f), y = f2(0.f);   // the column's (S, S_y) and (S_yy, red)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 e = S.sum4[tr][8 * q + 4 * i + th];
            a = __fadd2_rn(a, make_float2(e.x, e.y));
            y = __fadd2_rn(y, make_float2(e.z, e.w));
            gb = __fadd2_rn(gb, S.sum2[tr][8 * q + 4 * i + th]);
        }
        const float dx = __fsub_rn(cx0 + (float)(4 * i + th), xyt.x);
        const float adx = a.x * dx;
        s0 += a.x;
        sx += adx;
        sxx = fmaf(adx, dx, sxx);
        sy += a.y;
        sxy = fmaf(a.y, dx, sxy);
        syy += y.x;
        r += y.y;
    }
    // the record's four lanes exchange halves: lane th ends with two of the 8 sums
    float v[8] = {sx, sy, sxx, sxy, syy, r, gb.x, gb.y};
    const bool up = th & 2, up1 = th & 1;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float send = up ? v[q] : v[q + 4];
        v[q] = (up ? v[q + 4] : v[q]) + __shfl_xor_sync(all, send, 2);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const float send = up1 ? v[q] : v[q + 2];
        v[q] = (up1 ? v[q + 2] : v[q]) + __shfl_xor_sync(all, send, 1);
    }
    const float A = co.x * -kLn2, B = co.y * -kLn2, C = co.z * -kLn2;
    const int64_t gi = vb + __float_as_uint(S.rgbg[j].w);
    float2 gq = make_float2(th == 3 ? -v[0] : 0.5f * v[0], th == 1 ? v[1] : -v[1]);
    if (th == 0) gq = make_float2(fmaf(A, v[0], B * v[1]), fmaf(C, v[1], B * v[0]));
    if (tr < cnt && (v[0] != 0.f || v[1] != 0.f))
        atomicAdd(reinterpret_cast<float2 *>(p.grads + 8 * gi + 2 * th), gq);
    if (WANT_OP) {
        // sum of dL/dalpha G = (sum of dL/dpower) / o, as dL/dpower = dL/dalpha o G
        s0 += __shfl_xor_sync(all, s0, 1);
        s0 += __shfl_xor_sync(all, s0, 2);
        if (tr < cnt && th == 0 && s0 != 0.f) atomicAdd(p.d_opacity + gi, s0 / co.w);
    }
    __syncwarp();
}

template <int NP, bool WANT_OP, bool BINNED, bool STATS>
__global__ void __launch_bounds__(32 * BWD_WARPS) raster_bwd_kernel(RasterParams p)
{
    if (grid_wait()) return;
    __shared__ BwdWarp s_warp[BWD_WARPS];
    constexpr unsigned all = 0xffffffffu;
    BwdWarp &S = s_warp[threadIdx.x >> 5];
    const int view = blockIdx.y, lane = threadIdx.x & 31;
    const int unit = blockIdx.x * BWD_WARPS + (threadIdx.x >> 5);
    constexpr int UNITS = 4 / NP;   // warps of a tile
    constexpr bool AHEAD = NP == 1;
    const int tile = unit / UNITS, part = unit % UNITS;
    if (tile >= p.tx * p.ty) return;
    const int64_t tg = (int64_t)view * (p.tx * p.ty) + tile;
    // with the forward's list of the tile, its records are staged straight
    // from it (list order is position order); otherwise the bin's list is
    // tested again
    const int listed = p.tl_rec ? p.tl_cnt[tg] : -1;
    const bool heavy = listed < 0 || listed >= kHeavyList;
    if (listed == 0 || heavy != (blockIdx.z == 0)) return;
    const int tx_t = tile % p.tx, ty_t = tile / p.tx;
    const int wx = tx_t * 16 + (part & 1) * 8, wy = ty_t * 16 + (part >> 1) * 8;
    const int px = wx + (lane & 7), py0 = wy + (lane >> 3) * (2 * NP);
    const float cx0 = (float)wx + 0.5f, cy0 = (float)wy + 0.5f;   // centre of the warp's first pixel
    const float pxf = (float)px + 0.5f;
    float2 pyf[NP];
#pragma unroll
    for (int h = 0; h < NP; ++h) pyf[h] = make_float2((float)(py0 + 2 * h) + 0.5f, (float)(py0 + 2 * h) + 1.5f);
    const int64_t vb = (int64_t)view * p.n;
    const int64_t HW = (int64_t)p.H * p.W;
    PixBwd<NP> P;
    bool bad = false;
    {
        float T[2 * NP], d0[2 * NP], d1[2 * NP], d2[2 * NP], ns[2 * NP];
#pragma unroll
        for (int k = 0; k < 2 * NP; ++k) {
            const int py = py0 + k;
            P.last[k] = 0;
            T[k] = 1.f;
            d0[k] = d1[k] = d2[k] = 0.f;
            if (px < p.W && py < p.H) {
                const int64_t pix = (int64_t)view * HW + (int64_t)py * p.W + px;
                const float *di = p.d_img + (int64_t)view * 3 * HW + (int64_t)py * p.W + px;
                P.last[k] = p.last[pix];
                T[k] = p.T_final[pix];
                d0[k] = di[0];
                d1[k] = di[HW];
                d2[k] = di[2 * HW];
            }
            ns[k] = -fmaf(d2[k], p.bg2, fmaf(d1[k], p.bg1, d0[k] * p.bg0));
            bad |= !isfinite(d0[k] + d1[k] + d2[k]);
        }
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            P.T[h] = make_float2(T[2 * h], T[2 * h + 1]);
            P.dC0[h] = make_float2(d0[2 * h], d0[2 * h + 1]);
            P.dC1[h] = make_float2(d1[2 * h], d1[2 * h + 1]);
            P.dC2[h] = make_float2(d2[2 * h], d2[2 * h + 1]);
            P.nS[h] = make_float2(ns[2 * h], ns[2 * h + 1]);
        }
    }
    const bool guard = __any_sync(all, bad);
    const int wlast = __reduce_max_sync(all, max(max(P.last[0], P.last[1]), max(P.last[2 * NP - 2], P.last[2 * NP - 1])));
    if (wlast == 0) return;
    uint32_t n_tested = 0, n_contrib = 0;
    const uint2 *rec = p.tl_rec + tg * p.tl_cap;
    uint32_t first = 0;
    if (listed < 0) {
        const int binid = (ty_t / p.bin) * p.bins_x + tx_t / p.bin;
        first = p.ranges[(int64_t)view * p.bins + binid].x;
    }
    int head = 0, have = 0;     // the queue: its first record's slot (a multiple of BWD_CHUNK) and its length
    int cand0 = 0, cands = 0;   // tiles without a list: the candidates not yet staged
    int left = listed >= 0 ? listed : wlast;
    auto listed_entry = [&](int l) { return l - 1 - lane >= 0 ? rec[l - 1 - lane] : make_uint2(0u, 0x7fffffffu); };
    uint2 e_next = make_uint2(0u, 0x7fffffffu);
    if (AHEAD && listed >= 0) e_next = listed_entry(left);
    while (left > 0 || cands > 0 || have > 0) {
        // stage batches of 32 records, back to front, until a chunk is full
        while ((left > 0 || cands > 0) && have < BWD_CHUNK) {
            uint2 e = make_uint2(0u, 0x7fffffffu);   // (Gaussian, position)
            if (listed >= 0) {
                e = AHEAD ? e_next : listed_entry(left);
                left -= 32;
                if (AHEAD) e_next = listed_entry(left);
            } else {
                // a bin's list can hold tens of thousands of records, few of
                // them this tile's: their rectangles are tested BWD_TEST at a
                // time, every load of a test in flight at once (one test of
                // 32 after the other made a single such tile the launch's
                // longest: 832 -> 667 us)
                if (cands < 32 && left > 0) {
                    if (lane < cands) e = S.cand[cand0 + lane];
                    __syncwarp();
                    if (lane < cands) S.cand[lane] = e;
                    cand0 = 0;
                    while (cands < 32 && left > 0) {
                        constexpr int U = BWD_TEST / 32;
                        uint32_t g[U];
                        int r[U];
                        float2 m[U];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const int i = left - 1 - lane - 32 * u;
                            g[u] = i >= 0 ? p.vals[first + i] : 0u;
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const bool ok = left - 1 - lane - 32 * u >= 0;
                            r[u] = ok ? (BINNED ? p.radius[vb + g[u]] : 1) : 0;
                            m[u] = ok ? p.mean2d[vb + g[u]] : make_float2(0.f, 0.f);
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            bool in = r[u] > 0;
                            if (BINNED && in) {
                                int x0, y0, x1, y1;
                                tile_rect(m[u].x, m[u].y, r[u], p.tx, p.ty, x0, y0, x1, y1);
                                in = tx_t >= x0 && tx_t < x1 && ty_t >= y0 && ty_t < y1;
                            }
                            const unsigned b = __ballot_sync(all, in);
                            if (in)
                                S.cand[cands + __popc(b & ((1u << lane) - 1u))] =
                                    make_uint2(g[u], (uint32_t)(left - 1 - lane - 32 * u));
                            cands += __popc(b);
                        }
                        left -= BWD_TEST;
                    }
                    __syncwarp();
                }
                const int take = min(cands, 32);
                e = lane < take ? S.cand[cand0 + lane] : make_uint2(0u, 0x7fffffffu);
                cand0 += take;
                cands -= take;
            }
            bool keep = (int)e.y < wlast;
            int walked = 0x7fffffff;   // STATS: the position of a record of the tile's list
            float4 xyt, co;
            float c0 = 0.f, c1 = 0.f, c2 = 0.f;
            auto colour = [&]() {
                const float *c = p.rgb + 3 * (vb + e.x);
                c0 = c[0], c1 = c[1], c2 = c[2];
            };
            if (keep) {
                if (AHEAD) colour();
                const float2 m = p.mean2d[vb + e.x];
                co = p.conic_op[vb + e.x];
                if (STATS && (listed >= 0 || ellipse_hits_tile(m, co, tx_t, ty_t))) walked = (int)e.y;
                xyt = make_float4(m.x, m.y, staged_threshold(co.w), __uint_as_float(e.y));
                keep = visible(co.w);
                co = scale_conic(co);
                co.w = -co.w;
                keep = keep && staged_hits<NP>(xyt, co, cx0, cy0);
            }
            if (STATS) {
                for (int l = 0; l < 32; ++l) {
                    const int pos = __shfl_sync(all, walked, l);
#pragma unroll
                    for (int k = 0; k < 2 * NP; ++k) n_tested += pos < P.last[k];
                }
            }
            const unsigned kept = __ballot_sync(all, keep);
            if (keep) {
                int q = head + have + __popc(kept & ((1u << lane) - 1u));
                if (q >= BWD_QUEUE) q -= BWD_QUEUE;
                S.xyt[q] = xyt;
                S.co[q] = co;
                if (!AHEAD) colour();
                S.rgbg[q] = make_float4(c0, c1, c2, __uint_as_float(e.x));
            }
            have += __popc(kept);
        }
        if (have == 0) break;
        const int cnt = min(have, BWD_CHUNK);
        if (lane >= cnt && lane < BWD_CHUNK) {   // the last chunk's missing records take part nowhere
            S.xyt[head + lane] = make_float4(0.f, 0.f, 0.f, __int_as_float(0x7fffffff));
            S.co[head + lane] = S.rgbg[head + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncwarp();
        if (guard)
            bwd_chunk<NP, WANT_OP, STATS, true>(p, S, P, head, cnt, pxf, pyf, cx0, vb, n_contrib);
        else
            bwd_chunk<NP, WANT_OP, STATS, false>(p, S, P, head, cnt, pxf, pyf, cx0, vb, n_contrib);
        head += BWD_CHUNK;
        if (head == BWD_QUEUE) head = 0;
        have -= cnt;
    }
    if (STATS) flush_stats(p.stats, n_tested, n_contrib);
}

static gs_status fill(const gs_projected *proj, int64_t n, int V, int W, int H, int bin,
                      const float *bg, const uint32_t *vals, const uint32_t *ranges,
                      const gs_tile_lists *lists, RasterParams &p)
{
    if (lists) {
        GS_REQUIRE(lists->rec && lists->count && lists->cap >= 1 && lists->cap <= (1 << 20),
                   "raster: tile lists need rec, count and 1 <= cap <= 2^20");
        GS_REQUIRE(aligned(lists->rec, 8) && aligned(lists->count, 4), "raster: misaligned tile lists");
        p.tl_rec = reinterpret_cast<uint2 *>(lists->rec);
        p.tl_cnt = lists->count;
        p.tl_cap = lists->cap;
    }
    GS_REQUIRE(proj && vals && ranges, "raster: null argument");
    GS_REQUIRE(n >= 0 && V >= 1 && V <= GS_MAX_VIEWS, "raster: bad n or V");
    GS_REQUIRE(W > 0 && H > 0 && W <= 16384 && H <= 16384, "raster: bad image size");
    GS_REQUIRE(aligned(proj->mean2d, 8) && aligned(proj->conic_opacity, 16) && aligned(ranges, 8),
               "raster: misaligned input");
    p.mean2d = reinterpret_cast<const float2 *>(proj->mean2d);
    p.conic_op = reinterpret_cast<const float4 *>(proj->conic_opacity);
    p.rgb = proj->rgb;
    p.radius = proj->radius;
    GS_REQUIRE(bin >= 1 && bin <= 64, "raster: bin must be 1..64 tiles");
    GS_REQUIRE(bin == 1 || n == 0 || proj->radius, "raster: binned lists need the radius array");
    p.vals = vals;
    p.ranges = reinterpret_cast<const uint2 *>(ranges);
    p.n = n;
    p.V = V;
    p.W = W;
    p.H = H;
    p.tx = tiles_x_of(W);
    p.ty = tiles_y_of(H);
    p.bin = bin;
    p.bins_x = bins_x_of(W, bin);
    p.bins = p.bins_x * bins_y_of(H, bin);
    p.bg0 = bg ? bg[0] : 0.f;
    p.bg1 = bg ? bg[1] : 0.f;
    p.bg2 = bg ? bg[2] : 0.f;
    return GS_OK;
}

template <int NP, bool WANT_OP, bool BINNED>
static void launch_bwd(const RasterParams &p, cudaStream_t s)
{
    // 4 / NP warps a tile; the second layer takes the tiles with short lists
    // (without lists every tile is the first layer's)
    const dim3 grid((unsigned)ceil_div(4 / NP * p.tx * p.ty, BWD_WARPS), p.V, p.tl_rec ? 2 : 1);
    if (p.stats)
        launch_next(raster_bwd_kernel<NP, WANT_OP, BINNED, true>, grid, 32 * BWD_WARPS, 0, s, p);
    else
        launch_next(raster_bwd_kernel<NP, WANT_OP, BINNED, false>, grid, 32 * BWD_WARPS, 0, s, p);
}

template <bool WANT_OP, bool BINNED>
static void launch_bwd(const RasterParams &p, cudaStream_t s)
{
    if ((int64_t)p.tx * p.ty * p.V <= (int64_t)kFewTiles * num_sms())
        launch_bwd<1, WANT_OP, BINNED>(p, s);
    else
        launch_bwd<2, WANT_OP, BINNED>(p, s);
}

}  // namespace gs3

using namespace gs3;

extern "C" gs_status gs_raster_fwd(const gs_projected *proj, int64_t n, int V, int W, int H,
                                   int bin, const float *bg, const uint32_t *vals,
                                   const uint32_t *ranges, float *img, float *T_final,
                                   int32_t *last, uint64_t *d_stats, const gs_tile_lists *lists,
                                   gs_stream stream)
{
    RasterParams p{};
    gs_status st = fill(proj, n, V, W, H, bin, bg, vals, ranges, lists, p);
    if (st != GS_OK) return st;
    GS_REQUIRE(img && T_final && last, "gs_raster_fwd: null output");
    p.img = img;
    p.T_final = T_final;
    p.last = last;
    p.stats = reinterpret_cast<unsigned long long *>(d_stats);
    dim3 grid(p.tx * p.ty, V);
    note_launch();
    cudaStream_t s = as_stream(stream);
    if (bin > 1 && p.stats)
        launch_next(raster_fwd_kernel<true, true>, grid, NT, 0, s, p);
    else if (bin > 1)
        launch_next(raster_fwd_kernel<true, false>, grid, NT, 0, s, p);
    else if (p.stats)
        launch_next(raster_fwd_kernel<false, true>, grid, NT, 0, s, p);
    else
        launch_next(raster_fwd_kernel<false, false>, grid, NT, 0, s, p);
    return launch_status("gs_raster_fwd");
}

extern "C" gs_status gs_raster_bwd(const gs_projected *proj, int64_t n, int V, int W, int H,
                                   int bin, const float *bg, const uint32_t *vals,
                                   const uint32_t *ranges, const float *T_final,
                                   const int32_t *last, const float *d_img, float *grads,
                                   float *d_opacity, uint64_t *d_stats, const gs_tile_lists *lists,
                                   gs_stream stream)
{
    RasterParams p{};
    gs_status st = fill(proj, n, V, W, H, bin, bg, vals, ranges, lists, p);
    if (st != GS_OK) return st;
    GS_REQUIRE(T_final && last && d_img && (grads || n == 0), "gs_raster_bwd: null argument");
    GS_REQUIRE(aligned(grads, 16), "gs_raster_bwd: grads must be 16-byte aligned");
    cudaStream_t s = as_stream(stream);
    if (n > 0) {
        cudaMemsetAsync(grads, 0, sizeof(float) * 8 * n * V, s);
        if (d_opacity) cudaMemsetAsync(d_opacity, 0, sizeof(float) * n * V, s);
    }
    p.T_final = const_cast<float *>(T_final);
    p.last = const_cast<int32_t *>(last);
    p.d_img = d_img;
    p.grads = grads;
    p.d_opacity = d_opacity;
    p.stats = reinterpret_cast<unsigned long long *>(d_stats);
    note_launch();
    if (d_opacity && bin > 1)
        launch_bwd<true, true>(p, s);
    else if (d_opacity)
        launch_bwd<true, false>(p, s);
    else if (bin > 1)
        launch_bwd<false, true>(p, s);
    else
        launch_bwd<false, false>(p, s);
    return launch_status("gs_raster_bwd");
}
