// L1 + D-SSIM loss and its gradient (Section 4.1, Eq. 6).
// Pass 1 filters (x, y, (x - y)^2, xy) with the separable 11x11 Gaussian
// window, forms the SSIM map and the three per-pixel coefficients of its
// derivative wrt (mu_x, E[x^2], E[xy]); pass 2 filters those coefficients (the
// window is symmetric, so the adjoint is the same filter) and assembles
// dL/dI; pass 3 reduces the block partial sums (compensated FP32).
#include <math.h>

#include "common.cuh"

namespace gs3 {

// Both filtering passes work on tiles of LX x LY outputs, columns first.  In
// the column stage a thread walks down one of the LC = LX + 10 columns, its
// inputs read straight from global memory (a warp's lanes on one row, so
// coalesced at any width), and keeps LR outputs going; in the row stage a
// thread takes LO consecutive outputs of a row of the column-filtered maps in
// shared memory.  The passes are bound by instruction issue, so the shape is
// chosen for the fewest instructions a pixel: the maps go through both stages
// in pairs, in packed FP32 with one weight for both halves, as one 16-byte
// shared-memory access a pixel; 64 columns and LR = 8 rows make 256 column
// items, 32 rows and LO = 7 outputs make 256 row items.  A row stage whose
// lanes stand on eight rows of an odd stride meets no bank conflict; its
// results go through the same buffer once more to be written row by row.
// Of the squares only (x - y)^2 is filtered: sigma_x^2 + sigma_y^2 is its
// variance plus twice the covariance, and written so the map's numerator and
// denominator share the covariance's rounding.
// Four planes of three channels, 1352x1014: 191 us for the whole call (pass 1
// 99, pass 2 90, pass 3 5 us); one 479x361 image 17 us, sixteen 1920x1080 images
// 1 050 us; the gradient's error against 64 bits 6.1e-6 relative.  Rows first
// with pairs along the row (extra additions, and twice the weights, fetched
// again at each use), staged by TMA where W is a multiple of 4: 277, 26 and
// 1 500 us, 6.6e-6.  Both passes on chunks of planes whose coefficients stay in
// L2: 222 us (the chunks' last waves cost more).
constexpr int LX = 54, LY = 32;      // outputs of a tile
constexpr int LH = 5;                // window half-width
constexpr int LC = LX + 2 * LH;      // columns of the column stage
constexpr int LR = 8;                // rows of one column item
constexpr int LO = 7;                // outputs of one row item
constexpr int LTHREADS = 256;
constexpr int LS = 67, LS2 = 66, LS1 = 68;   // row strides of the shared maps (float4, float2, float)
static_assert(LC * (LY / LR) == LTHREADS, "one column item a thread");
static_assert(LY * 8 == LTHREADS && 8 * LO >= LX && 7 * LO + LO + 2 * LH <= LS, "one row item a thread");
static_assert(LS % 2 == 1, "eight rows meet eight bank groups");

struct LossParams {
    float w[6];           // the normalised 11-tap Gaussian window (sigma 1.5): taps 0..5, symmetric; set on the host
    const float *x, *y;
    int H, W;
    float lam;
    float invM;           // 1 / (planes H W), the mean's weight (set on the host)
    float *ca, *cb, *cc;  // per-pixel derivative coefficients
    float2 *partial;      // [blocks]: (sum of SSIM map, sum |x - y|)
    float *d_img;
    float *d_loss, *d_ssim;
    int nblocks;
};

__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }

// The six taps in registers (the empty asm keeps the compiler from fetching
// them again at every use).
struct Taps {
    float w[6];
    __device__ __forceinline__ explicit Taps(const LossParams &p)
    {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            w[k] = p.w[k];
            asm volatile("" : "+f"(w[k]));
        }
    }
    __device__ __forceinline__ float operator[](int k) const { return w[k <= 5 ? k : 10 - k]; }
};

// The order of a window's inputs, from its two ends inwards: the largest
// weights come last for most outputs, when the sums have their size, which
// keeps the filters' rounding error down (the gradient's 8.2e-6 -> 7.4e-6
// relative, before (x - y)^2 took the squares' place).
__device__ __forceinline__ constexpr int inwards(int i, int n) { return i & 1 ? n - 1 - (i >> 1) : i >> 1; }

// One column item's inputs: f(k, values at input row k) for the LR + 10 rows
// from gy0 on of column gx of N planes; 0 outside the image.  A block whose
// whole window lies inside takes the path without tests, on 32-bit offsets.
template <int N, typename F>
__device__ __forceinline__ void walk_column(const float *const (&base)[N], int gx, int gy0, int H, int W, bool inside,
                                            F &&f)
{
    constexpr int ROWS = LR + 2 * LH;
    if (inside) {
        const uint32_t step = 4u * (uint32_t)W;
        uint32_t top = 4u * ((uint32_t)gy0 * (uint32_t)W + (uint32_t)gx), bottom = top + (ROWS - 1) * step;
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            float v[N];
#pragma unroll
            for (int m = 0; m < N; ++m)
                v[m] = *reinterpret_cast<const float *>(reinterpret_cast<const char *>(base[m]) +
                                                        (i & 1 ? bottom : top));
            if (i & 1) bottom -= step;
            else top += step;
            f(inwards(i, ROWS), v);
        }
    } else {
        const bool okx = gx >= 0 && gx < W;
        const int64_t at0 = (int64_t)gy0 * W + gx;
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            const int k = inwards(i, ROWS);
            const bool ok = okx && gy0 + k >= 0 && gy0 + k < H;
            float v[N];
#pragma unroll
            for (int m = 0; m < N; ++m) v[m] = ok ? base[m][at0 + (int64_t)k * W] : 0.f;
            f(k, v);
        }
    }
}

// The row stage's place: a warp's lanes are eight rows x four groups of LO
// columns.
__device__ __forceinline__ void row_item(int &row, int &c0)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    row = (warp >> 1) * 8 + (lane & 7);
    c0 = ((warp & 1) * 4 + (lane >> 3)) * LO;
}

template <typename I>
__global__ void __launch_bounds__(LTHREADS, 3) ssim_fwd_kernel(LossParams p)
{
    if (grid_wait()) return;
    __shared__ float4 s_map[LY][LS];
    __shared__ float red[2][LTHREADS / 32];
    const int tid = threadIdx.x;
    const int x0 = blockIdx.x * LX, y0 = blockIdx.y * LY;
    const int64_t HW = (int64_t)p.H * p.W;
    const int64_t plane = (int64_t)blockIdx.z * HW;
    const int col = tid % LC, r0 = tid / LC * LR;
    const Taps w(p);
    const bool inside = x0 >= LH && x0 + LX + LH <= p.W && y0 >= LH && y0 + LY + LH <= p.H && sizeof(I) == 4;
    float lsum = 0.f;
    {
        const bool own = col >= LH && col < LH + LX;
        float2 axy[LR], adp[LR];   // filtered (x, y) and ((x - y)^2, xy)
#pragma unroll
        for (int o = 0; o < LR; ++o) axy[o] = adp[o] = dup(0.f);
        const float *const base[2] = {p.x + plane, p.y + plane};
        walk_column<2>(base, x0 - LH + col, y0 + r0 - LH, p.H, p.W, inside, [&](int k, const float (&v)[2]) {
            const float d = v[0] - v[1];
            const float2 xy = make_float2(v[0], v[1]), dp = make_float2(d * d, v[0] * v[1]);
            if (k >= LH && k < LH + LR) lsum += own ? fabsf(d) : 0.f;
#pragma unroll
            for (int o = 0; o < LR; ++o) {
                if (k - o < 0 || k - o > 2 * LH) continue;
                axy[o] = __ffma2_rn(dup(w[k - o]), xy, axy[o]);
                adp[o] = __ffma2_rn(dup(w[k - o]), dp, adp[o]);
            }
        });
#pragma unroll
        for (int o = 0; o < LR; ++o) s_map[r0 + o][col] = make_float4(axy[o].x, axy[o].y, adp[o].x, adp[o].y);
    }
    __syncthreads();
    int row, c0;
    row_item(row, c0);
    float2 fxy[LO], fdp[LO];
#pragma unroll
    for (int o = 0; o < LO; ++o) fxy[o] = fdp[o] = dup(0.f);
#pragma unroll
    for (int i = 0; i < LO + 2 * LH; ++i) {
        const int j = inwards(i, LO + 2 * LH);
        const float4 v = s_map[row][c0 + j];
#pragma unroll
        for (int o = 0; o < LO; ++o) {
            if (j - o < 0 || j - o > 2 * LH) continue;
            fxy[o] = __ffma2_rn(dup(w[j - o]), make_float2(v.x, v.y), fxy[o]);
            fdp[o] = __ffma2_rn(dup(w[j - o]), make_float2(v.z, v.w), fdp[o]);
        }
    }
    __syncthreads();
    // per-thread and per-warp sums in FP32 (at most LO * 32 terms)
    const float C1 = 0.01f * 0.01f, C2 = 0.03f * 0.03f;
    float ssum = 0.f;
    const bool oky = y0 + row < p.H;
#pragma unroll
    for (int o = 0; o < LO; ++o) {
        const float mx = fxy[o].x, my = fxy[o].y;
        const float dm = mx - my, vd = fdp[o].x - dm * dm, sxy = fdp[o].y - mx * my;
        const float n1 = 2.f * mx * my + C1, n2 = 2.f * sxy + C2;
        // d1 = mx^2 + my^2 + C1 and d2 = sigma_x^2 + sigma_y^2 + C2
        const float d1 = dm * dm + n1, d2 = vd + n2;
        const float idd = 1.f / (d1 * d2);
        const float sv = n1 * n2 * idd;
        // 1 / d1 = d2 idd and 1 / d2 = d1 idd
        const float ds_dmx = 2.f * my * n2 * idd - sv * 2.f * mx * (d2 * idd);
        const float ds_dsxx = -sv * (d1 * idd);
        const float ds_dsxy = 2.f * n1 * idd;
        s_map[row][c0 + o] = make_float4(ds_dmx - 2.f * mx * ds_dsxx - my * ds_dsxy, ds_dsxx, ds_dsxy, 0.f);
        if (oky && c0 + o < LX && x0 + c0 + o < p.W) ssum += sv;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ssum += __shfl_xor_sync(0xffffffffu, ssum, o);
        lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    }
    if ((tid & 31) == 0) {
        red[0][tid >> 5] = ssum;
        red[1][tid >> 5] = lsum;
    }
    __syncthreads();
    if (col < LX && x0 + col < p.W) {
        float *ca = p.ca + plane, *cb = p.cb + plane, *cc = p.cc + plane;
#pragma unroll
        for (int i = 0; i < LR; ++i) {
            const int r = tid / LC + i * (LTHREADS / LC);
            if (y0 + r >= p.H) continue;
            const float4 v = s_map[r][col];
            const I at = (I)(y0 + r) * (I)p.W + (I)(x0 + col);
            ca[at] = v.x;
            cb[at] = v.y;
            cc[at] = v.z;
        }
    }
    if (tid == 0) {
        float a = 0.f, b = 0.f;
        for (int ww = 0; ww < LTHREADS / 32; ++ww) {
            a += red[0][ww];
            b += red[1][ww];
        }
        p.partial[((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = make_float2(a, b);
    }
}

template <typename I>
__global__ void __launch_bounds__(LTHREADS, 4) ssim_bwd_kernel(LossParams p)
{
    if (grid_wait()) return;
    __shared__ float2 s_ab[LY][LS2];   // filtered (ca, cb)
    __shared__ float s_c[LY][LS1];     // filtered cc
    const int tid = threadIdx.x;
    const int x0 = blockIdx.x * LX, y0 = blockIdx.y * LY;
    const int64_t HW = (int64_t)p.H * p.W;
    const int64_t plane = (int64_t)blockIdx.z * HW;
    const int col = tid % LC, r0 = tid / LC * LR;
    const Taps w(p);
    const bool inside = x0 >= LH && x0 + LX + LH <= p.W && y0 >= LH && y0 + LY + LH <= p.H && sizeof(I) == 4;
    {
        float2 aab[LR];
        float ac[LR];
#pragma unroll
        for (int o = 0; o < LR; ++o) {
            aab[o] = dup(0.f);
            ac[o] = 0.f;
        }
        const float *const base[3] = {p.ca + plane, p.cb + plane, p.cc + plane};
        walk_column<3>(base, x0 - LH + col, y0 + r0 - LH, p.H, p.W, inside, [&](int k, const float (&v)[3]) {
#pragma unroll
            for (int o = 0; o < LR; ++o) {
                if (k - o < 0 || k - o > 2 * LH) continue;
                aab[o] = __ffma2_rn(dup(w[k - o]), make_float2(v[0], v[1]), aab[o]);
                ac[o] = fmaf(w[k - o], v[2], ac[o]);
            }
        });
#pragma unroll
        for (int o = 0; o < LR; ++o) {
            s_ab[r0 + o][col] = aab[o];
            s_c[r0 + o][col] = ac[o];
        }
    }
    __syncthreads();
    int row, c0;
    row_item(row, c0);
    {
        float2 fab[LO];
        float fc[LO];
#pragma unroll
        for (int o = 0; o < LO; ++o) {
            fab[o] = dup(0.f);
            fc[o] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < LO + 2 * LH; ++i) {
            const int j = inwards(i, LO + 2 * LH);
            const float2 ab = s_ab[row][c0 + j];
            const float c = s_c[row][c0 + j];
#pragma unroll
            for (int o = 0; o < LO; ++o) {
                if (j - o < 0 || j - o > 2 * LH) continue;
                fab[o] = __ffma2_rn(dup(w[j - o]), ab, fab[o]);
                fc[o] = fmaf(w[j - o], c, fc[o]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int o = 0; o < LO; ++o) {
            s_ab[row][c0 + o] = fab[o];
            s_c[row][c0 + o] = fc[o];
        }
    }
    const bool okx = col < LX && x0 + col < p.W;
    constexpr int RSTEP = LTHREADS / LC;
    const I first = (I)(y0 + tid / LC) * (I)p.W + (I)(x0 + col);
    const float *X = p.x + plane, *Y = p.y + plane;
    float *D = p.d_img + plane;
    float xv[LR], yv[LR];
#pragma unroll
    for (int i = 0; i < LR; ++i) {
        const bool ok = okx && y0 + tid / LC + i * RSTEP < p.H;
        const I at = first + (I)(i * RSTEP) * (I)p.W;
        xv[i] = ok ? X[at] : 0.f;
        yv[i] = ok ? Y[at] : 0.f;
    }
    __syncthreads();
    if (!okx) return;
#pragma unroll
    for (int i = 0; i < LR; ++i) {
        const int r = tid / LC + i * RSTEP;
        if (y0 + r >= p.H) continue;
        const float2 ab = s_ab[r][col];
        const float diff = xv[i] - yv[i];
        const float sgn = diff > 0.f ? 1.f : (diff < 0.f ? -1.f : 0.f);
        const float dssim = ab.x + 2.f * xv[i] * ab.y + yv[i] * s_c[r][col];
        D[first + (I)(i * RSTEP) * (I)p.W] = ((1.f - p.lam) * sgn - p.lam * dssim) * p.invM;
    }
}

// Compensated (Kahan) accumulation: s + (-c) carries the sum to about one
// rounding, independent of the number of terms.
__device__ __forceinline__ void kahan_add(float &s, float &c, float x)
{
    const float y = x - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
}

// Pass 3: the block partial sums in FP32, each thread's share compensated,
// the 1024 shares added in a tree (error about log2(1024) roundings).
__global__ void __launch_bounds__(1024) loss_final_kernel(LossParams p)
{
    if (grid_wait()) return;
    __shared__ float red[2][32];
    float sa = 0.f, ca = 0.f, sb = 0.f, cb = 0.f;
    // eight loads in flight a step
    for (int i0 = threadIdx.x; i0 < p.nblocks; i0 += 8 * blockDim.x) {
        float2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * (int)blockDim.x;
            v[u] = i < p.nblocks ? p.partial[i] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            kahan_add(sa, ca, v[u].x);
            kahan_add(sb, cb, v[u].y);
        }
    }
    float a = sa - ca, b = sb - cb;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = a;
        red[1][threadIdx.x >> 5] = b;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int nw = (int)(blockDim.x >> 5);
        a = threadIdx.x < nw ? red[0][threadIdx.x] : 0.f;
        b = threadIdx.x < nw ? red[1][threadIdx.x] : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
        }
        if (threadIdx.x == 0) {
            const float ssim = a * p.invM;
            *p.d_loss = (1.f - p.lam) * (b * p.invM) + p.lam * (1.f - ssim);
            if (p.d_ssim) *p.d_ssim = ssim;
        }
    }
}

static size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace gs3

using namespace gs3;

extern "C" size_t gs_loss_workspace_size(int planes, int H, int W)
{
    if (planes <= 0 || H <= 0 || W <= 0) return 0;
    size_t px = (size_t)planes * H * W;
    size_t nb = (size_t)ceil_div(W, LX) * ceil_div(H, LY) * planes;
    return 3 * a256(4 * px) + a256(16 * nb);
}

extern "C" gs_status gs_loss_l1_dssim(const float *img, const float *target, int planes, int H,
                                      int W, float lambda, float *d_img, float *d_loss,
                                      float *d_ssim, void *ws, size_t ws_bytes, gs_stream stream)
{
    GS_REQUIRE(img && target && d_img && d_loss && ws, "gs_loss_l1_dssim: null argument");
    GS_REQUIRE(planes > 0 && H > 0 && W > 0 && planes <= 65535, "gs_loss_l1_dssim: bad shape");
    GS_REQUIRE(ws_bytes >= gs_loss_workspace_size(planes, H, W),
               "gs_loss_l1_dssim: workspace too small");
    GS_REQUIRE(aligned(ws, 256), "gs_loss_l1_dssim: workspace must be 256-byte aligned");
    LossParams p{};
    {
        double w[11], sum = 0.0;
        for (int i = 0; i < 11; ++i) sum += (w[i] = exp(-(double)((i - 5) * (i - 5)) / 4.5));
        for (int i = 0; i < 6; ++i) p.w[i] = (float)(w[i] / sum);
    }
    p.H = H;
    p.W = W;
    p.lam = lambda;
    p.invM = (float)(1.0 / ((double)planes * (double)H * (double)W));
    const size_t px = (size_t)planes * H * W;
    char *b = reinterpret_cast<char *>(ws);
    p.ca = reinterpret_cast<float *>(b);
    p.cb = reinterpret_cast<float *>(b + a256(4 * px));
    p.cc = reinterpret_cast<float *>(b + 2 * a256(4 * px));
    float2 *partial = reinterpret_cast<float2 *>(b + 3 * a256(4 * px));
    p.d_loss = d_loss;
    p.d_ssim = d_ssim;
    const unsigned gx = (unsigned)ceil_div(W, LX), gy = (unsigned)ceil_div(H, LY);
    const dim3 grid(gx, gy, (unsigned)planes);
    cudaStream_t s = as_stream(stream);
    p.x = img;
    p.y = target;
    p.d_img = d_img;
    p.partial = partial;
    p.nblocks = (int)(gx * gy * (unsigned)planes);
    // 32-bit offsets within a plane while its bytes fit (the 64-bit ones made
    // the call 219 us where these make it 198)
    const bool small = (uint64_t)H * W < (uint64_t(1) << 30);
    note_launch();
    if (small) launch_next(ssim_fwd_kernel<uint32_t>, grid, LTHREADS, 0, s, p);
    else launch_next(ssim_fwd_kernel<int64_t>, grid, LTHREADS, 0, s, p);
    note_launch();
    if (small) launch_next(ssim_bwd_kernel<uint32_t>, grid, LTHREADS, 0, s, p);
    else launch_next(ssim_bwd_kernel<int64_t>, grid, LTHREADS, 0, s, p);
    note_launch();
    launch_next(loss_final_kernel, 1, 1024, 0, s, p);
    return launch_status("gs_loss_l1_dssim");
}
