// FP32 MLP of the transformation cache, 32-64-64-7 with ReLU and no bias, and
// its reverse, on the FP32 pipes.
//
// A block takes chunks of 64 rows; every product of a chunk is a small matrix
// product out of shared memory in which a thread owns a tile of 4 rows x 4
// features.  Activations lie [feature][row], so that one float4 holds four
// rows: the products of the layers take it as two packed operands against one
// weight, the weight gradients contract over it.  Per 64 multiply-adds a
// thread reads 8 float4, whose 32 lanes touch one or two wavefronts, so the
// FMA pipes and not shared memory are the bound.  (One thread per row, with
// the whole row's activations in its registers or its own shared-memory
// column, reads a weight or an activation per multiply-add: 44 us forward and
// 237 us reverse at 50 000 rows, against 25 and 65 us.  At 80 TFLOP/s they
// would take 8 and 24 us: the barriers between a chunk's products and the last,
// partly filled round of 782 chunks over the resident blocks are the rest.)
//
// Every activation, gate and row gradient is one ascending chain of fused
// multiply-adds, in the forward pass and where the reverse forms it again, so
// both see the same gates.
#include <algorithm>

#include "common.cuh"
#include "ntc.cuh"

namespace gs3 {

constexpr int MF_ROWS = 64, MF_THREADS = 256;
constexpr int MF_LD = MF_ROWS + 4;  // float4-aligned; eight features' float4 lie in eight bank groups
constexpr int MF_W1 = 36, MF_W2 = 68, MF_W3 = 68;
constexpr int MF_WSIZE = 64 * MF_W1 + 64 * MF_W2 + 7 * MF_W3;
constexpr size_t MF_BWD_SMEM = sizeof(float) * (MF_WSIZE + (32 + 4 * 64 + 8) * MF_LD);

struct MfWeights {
    const float *w1, *w2, *w3;
};

__device__ __forceinline__ MfWeights mf_load_weights(float *s, const float *W)
{
    float *w1 = s, *w2 = w1 + 64 * MF_W1, *w3 = w2 + 64 * MF_W2;
    for (int k = threadIdx.x; k < 64 * 32; k += MF_THREADS) w1[(k >> 5) * MF_W1 + (k & 31)] = W[k];
    for (int k = threadIdx.x; k < 64 * 64; k += MF_THREADS) w2[(k >> 6) * MF_W2 + (k & 63)] = W[64 * 32 + k];
    for (int k = threadIdx.x; k < 7 * 64; k += MF_THREADS) w3[(k >> 6) * MF_W3 + (k & 63)] = W[64 * 32 + 64 * 64 + k];
    return {w1, w2, w3};
}

__device__ __forceinline__ float4 mf_ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void mf_st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }

// four values of a row; `vec` says that rows start on a boundary of four values
__device__ __forceinline__ float4 mf_enc4(const float *p, bool vec)
{
    return vec ? *reinterpret_cast<const float4 *>(p) : make_float4(p[0], p[1], p[2], p[3]);
}
__device__ __forceinline__ float4 mf_enc4(const __nv_bfloat16 *p, bool vec)
{
    if (!vec) return make_float4(to_f32(p[0]), to_f32(p[1]), to_f32(p[2]), to_f32(p[3]));
    const uint2 u = *reinterpret_cast<const uint2 *>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
}

// slot k of the work is row k, or rows[k] of a list; -1 past the end
__device__ __forceinline__ int64_t mf_row(const uint32_t *rows, int64_t k, int64_t nslots, int64_t n)
{
    if (k >= nslots) return -1;
    const int64_t i = rows ? (int64_t)rows[k] : k;
    return i < n ? i : -1;
}

template <typename ET>
__device__ __forceinline__ void mf_load_x(float *sX, const ET *enc, bool vec, const uint32_t *rows, int64_t k0,
                                          int64_t nslots, int64_t n)
{
#pragma unroll
    for (int u = 0; u < MF_ROWS * 8 / MF_THREADS; ++u) {
        const int r = (threadIdx.x >> 3) + u * (MF_THREADS / 8), p = 4 * (threadIdx.x & 7);
        const int64_t i = mf_row(rows, k0 + r, nslots, n);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i >= 0) v = mf_enc4(enc + i * 32 + p, vec);
        sX[(p + 0) * MF_LD + r] = v.x;
        sX[(p + 1) * MF_LD + r] = v.y;
        sX[(p + 2) * MF_LD + r] = v.z;
        sX[(p + 3) * MF_LD + r] = v.w;
    }
}

// acc[i] (rows 4 tr .. + 3) = sum_k W[tc + 16 i][k] A[k][row], k ascending
template <int K, int LDW>
__device__ __forceinline__ void mf_layer(float2 (&acc)[4][2], const float *W, const float *A, int tr, int tc)
{
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
        float4 w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = mf_ld4(W + (tc + 16 * i) * LDW + k);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float4 a = mf_ld4(A + (k + u) * MF_LD + 4 * tr);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float wu = u == 0 ? w[i].x : u == 1 ? w[i].y : u == 2 ? w[i].z : w[i].w;
                acc[i][0] = __ffma2_rn(make_float2(wu, wu), make_float2(a.x, a.y), acc[i][0]);
                acc[i][1] = __ffma2_rn(make_float2(wu, wu), make_float2(a.z, a.w), acc[i][1]);
            }
        }
    }
}

__device__ __forceinline__ float4 mf_relu(const float2 (&a)[2])
{
    return make_float4(fmaxf(a[0].x, 0.f), fmaxf(a[0].y, 0.f), fmaxf(a[1].x, 0.f), fmaxf(a[1].y, 0.f));
}

// w[i][j] += sum over the chunk's rows of A[tr + 16 i][row] B[tc + 16 j][row]
template <int NB>
__device__ __forceinline__ void mf_contract(float (&w)[4][NB], const float *A, const float *B, int tr, int tc)
{
    float2 s[4][NB];   // over the even and the odd rows
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < NB; ++j) s[i][j] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int r = 0; r < MF_ROWS; r += 4) {
        float4 a[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = mf_ld4(A + (tr + 16 * i) * MF_LD + r);
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            const float4 b = mf_ld4(B + (tc + 16 * j) * MF_LD + r);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                s[i][j] = __ffma2_rn(make_float2(a[i].x, a[i].y), make_float2(b.x, b.y), s[i][j]);
                s[i][j] = __ffma2_rn(make_float2(a[i].z, a[i].w), make_float2(b.z, b.w), s[i][j]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < NB; ++j) w[i][j] += s[i][j].x + s[i][j].y;
}

// The activations of all layers share one buffer: with the weights it stays
// below the 48 KB that a kernel has without asking, and four blocks fit an SM.
template <typename ET>
__global__ void __launch_bounds__(MF_THREADS, 4) mlp_f32_fwd_kernel(const ET *enc, bool vec, int64_t n,
                                                                    const float *W, float *raw7)
{
    __shared__ __align__(16) float smem[MF_WSIZE + 64 * MF_LD];
    const MfWeights w = mf_load_weights(smem, W);
    float *sA = smem + MF_WSIZE;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // a warp covers 4 row groups x 8 features of the 16 x 16 threads
    const int tr = (warp >> 1) * 4 + (lane >> 3), tc = (warp & 1) * 8 + (lane & 7);
    const int64_t nchunks = (n + MF_ROWS - 1) / MF_ROWS;
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const int64_t k0 = ch * MF_ROWS;
        mf_load_x(sA, enc, vec, nullptr, k0, n, n);
        __syncthreads();
        float2 acc[4][2];
        mf_layer<32, MF_W1>(acc, w.w1, sA, tr, tc);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) mf_st4(sA + (tc + 16 * i) * MF_LD + 4 * tr, mf_relu(acc[i]));
        __syncthreads();
        mf_layer<64, MF_W2>(acc, w.w2, sA, tr, tc);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) mf_st4(sA + (tc + 16 * i) * MF_LD + 4 * tr, mf_relu(acc[i]));
        __syncthreads();
        // one row a thread, outputs q and q + 4
        const int r = t & 63, q = t >> 6, q4 = min(q + 4, 6);
        float o0 = 0.f, o1 = 0.f;
#pragma unroll 4
        for (int j = 0; j < 64; j += 4) {
            const float4 a = mf_ld4(w.w3 + q * MF_W3 + j), b = mf_ld4(w.w3 + q4 * MF_W3 + j);
            const float *h = sA + j * MF_LD + r;
            o0 = fmaf(a.x, h[0], o0), o1 = fmaf(b.x, h[0], o1);
            o0 = fmaf(a.y, h[MF_LD], o0), o1 = fmaf(b.y, h[MF_LD], o1);
            o0 = fmaf(a.z, h[2 * MF_LD], o0), o1 = fmaf(b.z, h[2 * MF_LD], o1);
            o0 = fmaf(a.w, h[3 * MF_LD], o0), o1 = fmaf(b.w, h[3 * MF_LD], o1);
        }
        if (k0 + r < n) {
            raw7[(k0 + r) * 7 + q] = o0;
            if (q < 3) raw7[(k0 + r) * 7 + q + 4] = o1;
        }
        __syncthreads();
    }
}

// One block runs the forward pass of a chunk again, then the row gradients
// and the weight gradients.  These are summed in three levels, so that no chain
// of additions runs over all rows of a block: a chunk's rows (the even and the
// odd ones, 32 each; 8 a warp for the last layer), the chunks in registers that
// live over all of them, and the blocks by one atomic a weight and block at the
// end (the last layer's warps are added up before).
template <typename ET>
__global__ void __launch_bounds__(MF_THREADS, 2)
    mlp_f32_bwd_kernel(const ET *enc, bool vec, int64_t n, const float *W, const float *d_raw7, const float *d_scale,
                       float *dW, float *d_enc, bool vec_out, const uint32_t *rows, const int64_t *d_rows)
{
    extern __shared__ __align__(16) float smem[];
    const MfWeights w = mf_load_weights(smem, W);
    float *sX = smem + MF_WSIZE, *sH1 = sX + 32 * MF_LD, *sH2 = sH1 + 64 * MF_LD, *sG2 = sH2 + 64 * MF_LD;
    float *sG1 = sG2 + 64 * MF_LD, *sGO = sG1 + 64 * MF_LD;
    const float scale = d_scale ? *d_scale : 1.f;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int tr = (warp >> 1) * 4 + (lane >> 3), tc = (warp & 1) * 8 + (lane & 7);
    float dw1[4][2], dw2[4][4], dw3[4][4];   // sums over the chunks so far
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j < 2) dw1[i][j] = 0.f;
            dw2[i][j] = dw3[i][j] = 0.f;
        }
    const int64_t nslots = d_rows ? *d_rows : n;
    const int64_t nchunks = (nslots + MF_ROWS - 1) / MF_ROWS;
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const int64_t k0 = ch * MF_ROWS;
        mf_load_x(sX, enc, vec, rows, k0, nslots, n);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int r = t & 63, q = (t >> 6) + 4 * u;
            const int64_t i = mf_row(rows, k0 + r, nslots, n);
            sGO[q * MF_LD + r] = i >= 0 && q < 7 ? d_raw7[i * 7 + q] * scale : 0.f;
        }
        __syncthreads();
        float2 acc[4][2];
        mf_layer<32, MF_W1>(acc, w.w1, sX, tr, tc);
#pragma unroll
        for (int i = 0; i < 4; ++i) mf_st4(sH1 + (tc + 16 * i) * MF_LD + 4 * tr, mf_relu(acc[i]));
        __syncthreads();
        mf_layer<64, MF_W2>(acc, w.w2, sH1, tr, tc);
        {
            float2 g[4][2];
#pragma unroll
            for (int i = 0; i < 4; ++i) g[i][0] = g[i][1] = make_float2(0.f, 0.f);
#pragma unroll
            for (int q = 0; q < 7; ++q) {
                const float4 a = mf_ld4(sGO + q * MF_LD + 4 * tr);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float wu = w.w3[q * MF_W3 + tc + 16 * i];
                    g[i][0] = __ffma2_rn(make_float2(wu, wu), make_float2(a.x, a.y), g[i][0]);
                    g[i][1] = __ffma2_rn(make_float2(wu, wu), make_float2(a.z, a.w), g[i][1]);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 h = mf_relu(acc[i]);
                const int at = (tc + 16 * i) * MF_LD + 4 * tr;
                mf_st4(sH2 + at, h);
                mf_st4(sG2 + at, make_float4(h.x > 0.f ? g[i][0].x : 0.f, h.y > 0.f ? g[i][0].y : 0.f,
                                             h.z > 0.f ? g[i][1].x : 0.f, h.w > 0.f ? g[i][1].y : 0.f));
            }
        }
        __syncthreads();
        // G1[row][k] = sum_j G2[row][j] W2[j][k] behind H1's gate, k = 4 tc .. + 3
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int j = 0; j < 64; ++j) {
            const float4 a = mf_ld4(sG2 + j * MF_LD + 4 * tr), b = mf_ld4(w.w2 + j * MF_W2 + 4 * tc);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float wu = i == 0 ? b.x : i == 1 ? b.y : i == 2 ? b.z : b.w;
                acc[i][0] = __ffma2_rn(make_float2(wu, wu), make_float2(a.x, a.y), acc[i][0]);
                acc[i][1] = __ffma2_rn(make_float2(wu, wu), make_float2(a.z, a.w), acc[i][1]);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int at = (4 * tc + i) * MF_LD + 4 * tr;
            const float4 h = mf_ld4(sH1 + at);
            mf_st4(sG1 + at, make_float4(h.x > 0.f ? acc[i][0].x : 0.f, h.y > 0.f ? acc[i][0].y : 0.f,
                                         h.z > 0.f ? acc[i][1].x : 0.f, h.w > 0.f ? acc[i][1].y : 0.f));
        }
        __syncthreads();
        if (d_enc) {  // sum_k W1[k][m] G1[row][k], m = 2 tc, 2 tc + 1
            float2 e[2][2];
            e[0][0] = e[0][1] = e[1][0] = e[1][1] = make_float2(0.f, 0.f);
#pragma unroll 4
            for (int k = 0; k < 64; ++k) {
                const float4 a = mf_ld4(sG1 + k * MF_LD + 4 * tr);
                const float2 b = *reinterpret_cast<const float2 *>(w.w1 + k * MF_W1 + 2 * tc);
                e[0][0] = __ffma2_rn(make_float2(b.x, b.x), make_float2(a.x, a.y), e[0][0]);
                e[0][1] = __ffma2_rn(make_float2(b.x, b.x), make_float2(a.z, a.w), e[0][1]);
                e[1][0] = __ffma2_rn(make_float2(b.y, b.y), make_float2(a.x, a.y), e[1][0]);
                e[1][1] = __ffma2_rn(make_float2(b.y, b.y), make_float2(a.z, a.w), e[1][1]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t i = mf_row(rows, k0 + 4 * tr + u, nslots, n);
                if (i < 0) continue;
                const float a = u & 1 ? e[0][u >> 1].y : e[0][u >> 1].x, b = u & 1 ? e[1][u >> 1].y : e[1][u >> 1].x;
                float *o = d_enc + i * 32 + 2 * tc;
                if (vec_out) *reinterpret_cast<float2 *>(o) = make_float2(a, b);
                else o[0] = a, o[1] = b;
            }
        }
        // dW1[j][m] and dW2[j][k]: j = tr + 16 i, m and k = tc + 16 i
        mf_contract<2>(dw1, sG1, sX, tr, tc);
        mf_contract<4>(dw2, sG2, sH1, tr, tc);
        // dW3[q][j]: each warp takes 8 of the rows, q = 4 (lane / 16) + i, j = lane % 16 + 16 i
        {
            float d[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) d[i][j] = 0.f;
#pragma unroll 1
            for (int r = 8 * warp; r < 8 * warp + 8; r += 4) {
                float4 a[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) a[i] = mf_ld4(sGO + (4 * (lane >> 4) + i) * MF_LD + r);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 b = mf_ld4(sH2 + ((lane & 15) + 16 * j) * MF_LD + r);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        d[i][j] = fmaf(a[i].x, b.x, d[i][j]);
                        d[i][j] = fmaf(a[i].y, b.y, d[i][j]);
                        d[i][j] = fmaf(a[i].z, b.z, d[i][j]);
                        d[i][j] = fmaf(a[i].w, b.w, d[i][j]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) dw3[i][j] += d[i][j];
        }
        __syncthreads();
    }
    float *sW3 = sX;   // the warps' sums of the last layer, [warp][8][64]; every chunk is done with sX to sH2
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            sW3[(warp * 8 + 4 * (lane >> 4) + i) * 64 + (lane & 15) + 16 * j] = dw3[i][j];
    __syncthreads();
    for (int k = t; k < 7 * 64; k += MF_THREADS) {
        float s = 0.f;
#pragma unroll
        for (int w8 = 0; w8 < MF_THREADS / 32; ++w8) s += sW3[w8 * 8 * 64 + k];
        if (s != 0.f) atomicAdd(dW + 64 * 32 + 64 * 64 + k, s);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int j = tr + 16 * i;
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (dw1[i][k] != 0.f) atomicAdd(dW + j * 32 + tc + 16 * k, dw1[i][k]);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (dw2[i][k] != 0.f) atomicAdd(dW + 64 * 32 + j * 64 + tc + 16 * k, dw2[i][k]);
    }
}

template <typename ET>
static void launch_fwd(const void *enc, int64_t n, const gs_mlp *w, float *raw7, cudaStream_t s)
{
    const int blocks = (int)std::min<int64_t>(ceil_div(n, MF_ROWS), 4 * num_sms());
    note_launch();
    mlp_f32_fwd_kernel<ET><<<blocks, MF_THREADS, 0, s>>>((const ET *)enc, aligned(enc, 4 * sizeof(ET)), n, w->w_f32,
                                                        raw7);
}

template <typename ET>
static void launch_bwd(const void *enc, int64_t n, const gs_mlp *w, const float *d_raw7, const float *d_scale,
                       float *dW, float *d_enc, const uint32_t *rows, const int64_t *d_rows, cudaStream_t s)
{
    set_smem_limit((const void *)mlp_f32_bwd_kernel<ET>, MF_BWD_SMEM);
    const int blocks = (int)std::min<int64_t>(ceil_div(n, MF_ROWS), 2 * num_sms());
    note_launch();
    mlp_f32_bwd_kernel<ET><<<blocks, MF_THREADS, MF_BWD_SMEM, s>>>((const ET *)enc, aligned(enc, 4 * sizeof(ET)), n,
                                                                  w->w_f32, d_raw7, d_scale, dW, d_enc,
                                                                  aligned(d_enc, 8), rows, d_rows);
}

gs_status mlp_f32_fwd(const void *enc, int enc_dtype, int64_t n, const gs_mlp *w, float *raw7, cudaStream_t s)
{
    if (enc_dtype == GS_F32) launch_fwd<float>(enc, n, w, raw7, s);
    else launch_fwd<__nv_bfloat16>(enc, n, w, raw7, s);
    return launch_status("ntc_mlp_fwd");
}

gs_status mlp_f32_bwd(const void *enc, int enc_dtype, int64_t n, const gs_mlp *w, const float *d_raw7,
                      const float *d_scale, float *dW, float *d_enc, const uint32_t *rows, const int64_t *d_rows,
                      cudaStream_t s)
{
    if (enc_dtype == GS_F32) launch_bwd<float>(enc, n, w, d_raw7, d_scale, dW, d_enc, rows, d_rows, s);
    else launch_bwd<__nv_bfloat16>(enc, n, w, d_raw7, d_scale, dW, d_enc, rows, d_rows, s);
    return launch_status("ntc_mlp_bwd");
}

}  // namespace gs3
