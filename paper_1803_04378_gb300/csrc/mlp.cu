// mlp.cu -- the learned warm start's network (lp_mlp_* in include/lpgb.h).
//
// A 3-layer perceptron  in -> H -> H -> out  with ReLU, trained with the
// binary cross-entropy on logits against the 0/1 "basic at the optimum"
// labels of a family of LPs, and Adam.  Weights are used in FP16 with FP32
// accumulation on the tensor cores (tcgen05.mma through tc_gemm: TMA-staged
// tiles, accumulators in TMEM); FP32 master weights and Adam moments are kept
// for the update.
//
// Loss (per batch of B samples):  L = (1/B) sum_b sum_o [softplus(z_bo) - t_bo z_bo]
// so dL/dz = (sigmoid(z) - t) / B, small enough and large enough for FP16.
//
// Every product is D = X Y^T with both operands K-major (tc_gemm), so each
// FP16 operand is kept in the layout its GEMM reads: activations row-major
// [B x features] and, for the weight gradients, transposed [features x B];
// the weights as W^T (forward) and W (the input gradients of the backward
// pass).  FP16 rows are padded with zeros to a multiple of 64 elements (whole K
// blocks); FP32 results keep the logical widths.  Parameters are packed
// W1, b1, W2, b2, W3, b3 with W_l row-major [in_l x out_l].
//
// Bias, ReLU and its backward ride in the GEMMs' epilogues: a lane of an epilogue
// warp holds 32 columns of one row, so the row-major copy leaves in 16-byte
// stores and the transposed copy in 64-byte rows of a warp.  (As kernels of
// their own, with the transposed copy written element by element, they took
// 220 of a training step's 324 us at batch 256 and 6144 -> 512 -> 512 -> 3072.)
// Every sum keeps its order -- K by K in the MMA, row by row in the bias
// gradients -- whatever the tile width, so the results do not depend on it:
// products with few tiles take 32 columns per CTA (z1 at batch 256: 8 CTAs of 128
// columns 32 us).  The chain is programmatic dependent launches.
#include "../../include/lpgb.h"
#include "lpgb_internal.cuh"
#include "tc_gemm.cuh"

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <vector>

using lpgb::launch_k;
using lpgb::pdl_enter;

namespace {

// FP16 row strides: whole K blocks of the GEMMs, the padding zero
inline int pad64(int v) { return (v + 63) & ~63; }

// 32 consecutive halves of row `row` from column c0 (row stride ld, a multiple
// of 8, base 16-byte aligned): 16-byte stores where all columns exist
__device__ __forceinline__ void store_row16(__half* a, int ld, int row, int c0, int N, const __half (&h)[32]) {
    __half* p = a + (size_t)row * ld + c0;
    if (c0 + 32 <= N) {
#pragma unroll
        for (int i = 0; i < 32; i += 8) *reinterpret_cast<uint4*>(p + i) = *reinterpret_cast<const uint4*>(&h[i]);
    } else {
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (c0 + i < N) p[i] = h[i];
    }
}
// the same as column `row` of the transposed copy: a warp's rows side by side; the
// rows between M and the next multiple of 64 are zero (K of the weight gradients)
__device__ __forceinline__ void store_col16(__half* aT, int ldt, int row, int M, int c0, int N, const __half (&h)[32]) {
    if (row >= ((M + 63) & ~63)) return;
#pragma unroll
    for (int i = 0; i < 32; ++i)
        if (c0 + i < N) aT[(size_t)(c0 + i) * ldt + row] = row < M ? h[i] : __float2half_rn(0.f);
}
__device__ __forceinline__ void load_row32(const float* z, int ld, int row, int c0, int N, float (&v)[32]) {
    const float* p = z + (size_t)row * ld + c0;
    if (c0 + 32 <= N && (ld & 3) == 0 && (reinterpret_cast<uintptr_t>(z) & 15) == 0) {
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
            const float4 q = *reinterpret_cast<const float4*>(p + i);
            v[i] = q.x; v[i + 1] = q.y; v[i + 2] = q.z; v[i + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = c0 + i < N ? p[i] : 0.f;
    }
}
__device__ __forceinline__ void store_row32(float* z, int ld, int row, int c0, int N, const float (&v)[32]) {
    float* p = z + (size_t)row * ld + c0;
    if (c0 + 32 <= N && (ld & 3) == 0 && (reinterpret_cast<uintptr_t>(z) & 15) == 0) {
#pragma unroll
        for (int i = 0; i < 32; i += 4) *reinterpret_cast<float4*>(p + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (c0 + i < N) p[i] = v[i];
    }
}

// D = acc (the weight gradients)
struct EpiStore {
    float* D;
    int M, N;
    __device__ void operator()(int trow, int m0, int n0, int c0, const float (&v)[32]) const {
        if (m0 + trow < M) store_row32(D, N, m0 + trow, n0 + c0, N, v);
    }
};

// z = acc + bias; with a: a = relu(z) in FP16, and with aT its transpose; z itself
// where it is asked for
struct EpiAct {
    const float* bias;
    float* z;
    __half *a, *aT;
    int lda, ldt, M, N;
    __device__ void operator()(int trow, int m0, int n0, int c0, const float (&v)[32]) const {
        const int row = m0 + trow, c = n0 + c0;
        float x[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) x[i] = v[i] + (c + i < N ? __ldg(bias + c + i) : 0.f);
        if (z && row < M) store_row32(z, N, row, c, N, x);
        if (a) {
            __align__(16) __half h[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) h[i] = __float2half_rn(fmaxf(x[i], 0.f));
            if (row < M) store_row16(a, lda, row, c, N, h);
            if (aT) store_col16(aT, ldt, row, M, c, N, h);
        }
    }
};

// dz = acc * (z > 0), FP16 (row-major and transposed)
struct EpiReluBack {
    const float* z;
    __half *dz, *dzT;
    int ld, ldt, M, N;
    __device__ void operator()(int trow, int m0, int n0, int c0, const float (&v)[32]) const {
        const int row = m0 + trow, c = n0 + c0;
        __align__(16) __half h[32];
        if (row < M) {
            float zz[32];
            load_row32(z, N, row, c, N, zz);
#pragma unroll
            for (int i = 0; i < 32; ++i) h[i] = __float2half_rn(zz[i] > 0.f ? v[i] : 0.f);
            store_row16(dz, ld, row, c, N, h);
        }
        store_col16(dzT, ldt, row, M, c, N, h);
    }
};

// X (rows x cols, FP32) -> x16 (row stride ld) and, where asked for, xT (cols x
// rows, row stride ldt, zero up to the next multiple of 64 rows), FP16, by 32 x 32
// tiles through shared memory
constexpr int kTile = 32;
__global__ void __launch_bounds__(256) k_input16(const float* __restrict__ X, int rows, int cols,
                                                 __half* __restrict__ x16, int ld, __half* __restrict__ xT, int ldt) {
    pdl_enter();
    __shared__ __half tile[kTile][kTile + 2];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int tc = (cols + kTile - 1) / kTile;  // tiles in a row of them: one grid dimension, for any batch
    const int c0 = blockIdx.x % tc * kTile, r0 = blockIdx.x / tc * kTile;
#pragma unroll
    for (int i = 0; i < kTile; i += 8) {
        const int r = r0 + ty + i, c = c0 + tx;
        __half h = __float2half_rn(0.f);
        if (r < rows && c < cols) {
            h = __float2half_rn(X[(size_t)r * cols + c]);
            x16[(size_t)r * ld + c] = h;
        }
        tile[ty + i][tx] = h;
    }
    if (!xT) return;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kTile; i += 8) {
        const int c = c0 + ty + i, r = r0 + tx;
        if (c < cols) xT[(size_t)c * ldt + r] = tile[tx][ty + i];  // (zero past the batch)
    }
}

// dz = (sigmoid(z) - t) / B in FP16 (row-major, and transposed with zeros up to the
// next multiple of 64 rows); a partial sum per block of (softplus(z) - t z) / B.  32 x 32
// tiles through shared memory; in the GEMM's epilogue the exponentials of 64 elements
// per lane ran on four warps per SM and took 25 us at 256 x 3072, here 5.
__global__ void __launch_bounds__(256) k_bce(const float* __restrict__ z, const float* __restrict__ t, int rows, int cols,
                                             __half* __restrict__ dz, int ld, __half* __restrict__ dzT, int ldt,
                                             float* __restrict__ part) {
    pdl_enter();
    __shared__ __half tile[kTile][kTile + 2];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int tc = (cols + kTile - 1) / kTile;  // tiles in a row of them: one grid dimension, for any batch
    const int c0 = blockIdx.x % tc * kTile, r0 = blockIdx.x / tc * kTile;
    const float inv = 1.f / (float)rows;
    float l = 0.f;
#pragma unroll
    for (int i = 0; i < kTile; i += 8) {
        const int r = r0 + ty + i, c = c0 + tx;
        __half h = __float2half_rn(0.f);
        if (r < rows && c < cols) {
            const float v = z[(size_t)r * cols + c], tt = t[(size_t)r * cols + c];
            const float sp = v > 0.f ? v + log1pf(expf(-v)) : log1pf(expf(v));
            l += (sp - tt * v) * inv;
            const float sg = 1.f / (1.f + expf(-v));
            h = __float2half_rn((sg - tt) * inv);
            dz[(size_t)r * ld + c] = h;
        }
        tile[ty + i][tx] = h;
    }
    __shared__ float wl[8];
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (tx == 0) wl[ty] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) l += wl[w];
        part[blockIdx.x] = l;
    }
#pragma unroll
    for (int i = 0; i < kTile; i += 8) {
        const int c = c0 + ty + i, r = r0 + tx;
        if (c < cols) dzT[(size_t)c * ldt + r] = tile[tx][ty + i];
    }
}

// db[c] = sum_r dz[r][c], row by row, of the three layers' dz at once: a block
// loads 64 columns of 128 rows at a time and 64 of its threads add them (one
// row's load in flight per column took the three sums 55 us, 32 rows 14)
// The first block also adds the loss's partial sums, in a fixed order.
struct ColSum {
    const __half* dz[3];
    float* db[3];
    int ld[3], cols[3];
    const float* part;
    int nparts;
    float* loss;
};
constexpr int kSumRows = 128, kSumCols = 64;
__global__ void __launch_bounds__(256) k_colsum(ColSum q, int rows) {
    pdl_enter();
    __shared__ __half tile[kSumRows][kSumCols];
    const int l = blockIdx.y, c0 = blockIdx.x * kSumCols, tid = threadIdx.x;
    if (l == 0 && c0 == 0 && tid < 32) {
        double v = 0.0;
        for (int e = tid; e < q.nparts; e += 32) v += (double)q.part[e];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (tid == 0) *q.loss = (float)v;
    }
    if (c0 >= q.cols[l]) return;
    float s = 0.f;
    for (int r0 = 0; r0 < rows; r0 += kSumRows) {
        const int nr = min(kSumRows, rows - r0);
        // (rows are padded to 64 columns: whole 16-byte pieces)
        for (int e = tid; e < nr * (kSumCols / 8); e += 256) {
            const int r = e / (kSumCols / 8), c = 8 * (e % (kSumCols / 8));
            *reinterpret_cast<uint4*>(&tile[r][c]) =
                *reinterpret_cast<const uint4*>(q.dz[l] + (size_t)(r0 + r) * q.ld[l] + c0 + c);
        }
        __syncthreads();
        if (tid < kSumCols) {
            int r = 0;
#pragma unroll 16
            for (; r < nr; ++r) s += __half2float(tile[r][tid]);
        }
        __syncthreads();
    }
    if (tid < kSumCols && c0 + tid < q.cols[l]) q.db[l][c0 + tid] = s;
}

// One Adam step on every parameter (kAdam) and the FP16 copies of the weights from
// the FP32 masters: W itself (row stride ldn, where asked for) and W^T, by 64 x 32
// tiles through shared memory.  The blocks past the matrices' tiles take the biases.
struct Mats {
    int rows[3], cols[3], tiles_c[3], first[4];  // first tile of each matrix; first[3]: their number
    size_t off[6];                               // W1 b1 W2 b2 W3 b3
    int nbias[3];
    __half *wn[3], *wt[3];
    int ldn[3], ldt[3];
};
struct Adam {
    float *p, *m1, *m2;
    const float* g;
    float lr, b1, b2, eps, c1, c2;
};
template <bool kAdam>
__device__ __forceinline__ float adam_one(const Adam& q, size_t e) {
    if (!kAdam) return q.p[e];
    const float gg = q.g[e];
    const float a = q.b1 * q.m1[e] + (1.f - q.b1) * gg;
    const float v = q.b2 * q.m2[e] + (1.f - q.b2) * gg * gg;
    q.m1[e] = a;
    q.m2[e] = v;
    const float w = q.p[e] - q.lr * (a / q.c1) / (sqrtf(v / q.c2) + q.eps);
    q.p[e] = w;
    return w;
}
constexpr int kWR = 64, kWC = 32;
template <bool kAdam>
__global__ void __launch_bounds__(256) k_weights(Adam q, Mats w) {
    pdl_enter();
    __shared__ __half tile[kWC][kWR + 2];
    const int t = blockIdx.x;
    if (t >= w.first[3]) {
        if (!kAdam) return;
        int e = (t - w.first[3]) * 256 + threadIdx.x;
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            if (e >= 0 && e < w.nbias[l]) adam_one<kAdam>(q, w.off[2 * l + 1] + e);
            e -= w.nbias[l];
        }
        return;
    }
    const int l = t >= w.first[2] ? 2 : (t >= w.first[1] ? 1 : 0);
    const int rows = w.rows[l], cols = w.cols[l];
    const int r0 = (t - w.first[l]) / w.tiles_c[l] * kWR, c0 = (t - w.first[l]) % w.tiles_c[l] * kWC;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < kWR; i += 8) {
        const int r = r0 + ty + i, c = c0 + tx;
        if (r < rows && c < cols) {
            const __half h = __float2half_rn(adam_one<kAdam>(q, w.off[2 * l] + (size_t)r * cols + c));
            if (w.wn[l]) w.wn[l][(size_t)r * w.ldn[l] + c] = h;
            tile[tx][ty + i] = h;
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kWC; i += 8) {
        const int c = c0 + ty + i, r = r0 + 2 * tx;
        if (c >= cols || r >= rows) continue;
        __half* d = w.wt[l] + (size_t)c * w.ldt[l] + r;
        if (r + 1 < rows) *reinterpret_cast<__half2*>(d) = *reinterpret_cast<const __half2*>(&tile[ty + i][2 * tx]);
        else *d = tile[ty + i][2 * tx];
    }
}

}  // namespace

struct lp_mlp {
    int in = 0, hid = 0, out = 0, maxb = 0;
    int in_p = 0, hid_p = 0, out_p = 0, b_p = 0;  // FP16 row strides (multiples of 64)
    size_t np = 0;
    size_t off[6] = {};  // W1 b1 W2 b2 W3 b3 offsets into the packed vectors
    cudaStream_t stream = nullptr;
    std::vector<void*> allocs;
    float *p = nullptr, *g = nullptr, *m1 = nullptr, *m2 = nullptr;  // packed fp32
    __half *w1t = nullptr, *w2t = nullptr, *w3t = nullptr;           // W^T: [hid x in], [hid x hid], [out x hid]
    __half *w2n = nullptr, *w3n = nullptr;                           // W:   [hid x hid], [hid x out]
    __half *x16 = nullptr, *xT = nullptr;                            // [maxb x in], [in x maxb]
    float *z1 = nullptr, *z2 = nullptr, *z3 = nullptr;               // pre-activations
    __half *a1 = nullptr, *a2 = nullptr, *a1T = nullptr, *a2T = nullptr;
    __half *dz3 = nullptr, *dz2 = nullptr, *dz1 = nullptr;
    __half *dz3T = nullptr, *dz2T = nullptr, *dz1T = nullptr;
    float* loss = nullptr;
    float* part = nullptr;   // its partial sums, one per block of k_bce
    int32_t* err = nullptr;  // bounded-wait flag of the tensor-core GEMMs
    int64_t steps = 0;
    int sms = 1;
};

namespace {

int mfail(cudaError_t e) { return e == cudaErrorMemoryAllocation ? LP_ERR_OOM : LP_ERR_CUDA; }

#define MCK(x)                                   \
    do {                                         \
        cudaError_t e_ = (x);                    \
        if (e_ != cudaSuccess) return mfail(e_); \
    } while (0)

template <typename T>
int malloc_t(lp_mlp* h, T** p, size_t n) {
    void* v = nullptr;
    cudaError_t e = cudaMalloc(&v, std::max<size_t>(n, 1) * sizeof(T));
    if (e != cudaSuccess) return mfail(e);
    h->allocs.push_back(v);
    *p = static_cast<T*>(v);
    return LP_OK;
}

// epi(X Y^T): X is M x K (row stride ldx), Y N x K (row stride ldy), both FP16.
// Tiles of 32 columns while the chip holds them at once, else 64, else 128; the
// deeper rings of the narrow tiles keep as many bytes in flight.
template <class Epi>
int gemm(const lp_mlp* h, int M, int N, int K, const __half* X, int ldx, const __half* Y, int ldy, const Epi& epi) {
    using namespace lpgb;
    const int mt = (M + tcg::kTM - 1) / tcg::kTM;
    const int bn = mt * ((N + 31) / 32) <= h->sms ? 32 : (mt * ((N + 63) / 64) <= h->sms ? 64 : 128);
    const int ar = M >= tcg::kTM ? tcg::kTM : (M + 7) & ~7;  // whole 8-row swizzle atoms
    CUtensorMap ma, mb;
    const int kb = bn == 32 ? tcg::GemmStage<32>::KB : (bn == 64 ? tcg::GemmStage<64>::KB : tcg::GemmStage<128>::KB);
    if (!tc_make_map_16bit_k(&ma, X, M, K, ldx, ar, kb, false) || !tc_make_map_16bit_k(&mb, Y, N, K, ldy, bn, kb, false))
        return LP_ERR_CUDA;
    cudaError_t e;
    if (bn == 32) e = tcg::launch_tc_gemm<32, false, true>(ma, mb, epi, M, N, K, ar, h->err, h->stream, true);
    else if (bn == 64) e = tcg::launch_tc_gemm<64, false, true>(ma, mb, epi, M, N, K, ar, h->err, h->stream, true);
    else e = tcg::launch_tc_gemm<128, false, true>(ma, mb, epi, M, N, K, ar, h->err, h->stream, true);
    MCK(e);
    return LP_OK;
}

// One Adam step with the gradients in h->g (lr > 0) and the FP16 weights, or the weights alone
int refresh_weights(lp_mlp* h, float lr = 0.f) {
    Mats w{};
    const int in[3] = {h->in, h->hid, h->hid}, out[3] = {h->hid, h->hid, h->out};
    __half* wn[3] = {nullptr, h->w2n, h->w3n};
    __half* wt[3] = {h->w1t, h->w2t, h->w3t};
    int biases = 0;
    for (int l = 0; l < 3; ++l) {
        w.rows[l] = in[l];
        w.cols[l] = out[l];
        w.tiles_c[l] = (out[l] + kWC - 1) / kWC;
        w.first[l + 1] = w.first[l] + w.tiles_c[l] * ((in[l] + kWR - 1) / kWR);
        w.off[2 * l] = h->off[2 * l];
        w.off[2 * l + 1] = h->off[2 * l + 1];
        w.nbias[l] = out[l];
        w.wn[l] = wn[l];
        w.wt[l] = wt[l];
        w.ldn[l] = l == 2 ? h->out_p : h->hid_p;
        w.ldt[l] = l == 0 ? h->in_p : h->hid_p;
        biases += out[l];
    }
    Adam q{h->p, h->m1, h->m2, h->g, lr, 0.9f, 0.999f, 1e-8f, 1.f, 1.f};
    if (lr > 0.f) {
        q.c1 = 1.f - powf(q.b1, (float)h->steps);
        q.c2 = 1.f - powf(q.b2, (float)h->steps);
        MCK(launch_k(k_weights<true>, dim3(w.first[3] + (biases + 255) / 256), dim3(256), 0, h->stream, true, q, w));
    } else {
        MCK(launch_k(k_weights<false>, dim3(w.first[3]), dim3(256), 0, h->stream, false, q, w));
    }
    return LP_OK;
}

// 32 x 32 tiles of a batch's rows, padded to 64, by `cols` columns
unsigned tiles(int cols, int B) { return (unsigned)((cols + kTile - 1) / kTile) * (unsigned)(pad64(B) / kTile); }

// the hidden layers for a batch already in x16; back: what the backward pass reads is kept too
int hidden_layers(lp_mlp* h, int B, bool back) {
    const float *b1 = h->p + h->off[1], *b2 = h->p + h->off[3];
    int rc;
    if ((rc = gemm(h, B, h->hid, h->in, h->x16, h->in_p, h->w1t, h->in_p,
                   EpiAct{b1, back ? h->z1 : nullptr, h->a1, back ? h->a1T : nullptr, h->hid_p, h->b_p, B, h->hid})))
        return rc;
    return gemm(h, B, h->hid, h->hid, h->a1, h->hid_p, h->w2t, h->hid_p,
                EpiAct{b2, back ? h->z2 : nullptr, h->a2, back ? h->a2T : nullptr, h->hid_p, h->b_p, B, h->hid});
}

// loss and gradients into h->g for targets t (fp32, device, [B x out])
int forward_backward(lp_mlp* h, int B, const float* t) {
    int rc;
    if ((rc = hidden_layers(h, B, true))) return rc;
    // layer 3: logits, dz3 and the loss; da2 = dz3 W3^T, dz2; da1 = dz2 W2^T, dz1
    if ((rc = gemm(h, B, h->out, h->hid, h->a2, h->hid_p, h->w3t, h->hid_p,
                   EpiAct{h->p + h->off[5], h->z3, nullptr, nullptr, 0, 0, B, h->out})))
        return rc;
    MCK(launch_k(k_bce, dim3(tiles(h->out, B)), dim3(256), 0, h->stream, true,
                 (const float*)h->z3, t, B, h->out, h->dz3, h->out_p, h->dz3T, h->b_p, h->part));
    if ((rc = gemm(h, B, h->hid, h->out, h->dz3, h->out_p, h->w3n, h->out_p,
                   EpiReluBack{h->z2, h->dz2, h->dz2T, h->hid_p, h->b_p, B, h->hid})))
        return rc;
    if ((rc = gemm(h, B, h->hid, h->hid, h->dz2, h->hid_p, h->w2n, h->hid_p,
                   EpiReluBack{h->z1, h->dz1, h->dz1T, h->hid_p, h->b_p, B, h->hid})))
        return rc;
    // gW3 = a2^T dz3, gW2 = a1^T dz2, gW1 = x^T dz1
    if ((rc = gemm(h, h->hid, h->out, B, h->a2T, h->b_p, h->dz3T, h->b_p, EpiStore{h->g + h->off[4], h->hid, h->out})))
        return rc;
    if ((rc = gemm(h, h->hid, h->hid, B, h->a1T, h->b_p, h->dz2T, h->b_p, EpiStore{h->g + h->off[2], h->hid, h->hid})))
        return rc;
    if ((rc = gemm(h, h->in, h->hid, B, h->xT, h->b_p, h->dz1T, h->b_p, EpiStore{h->g + h->off[0], h->in, h->hid})))
        return rc;
    const ColSum q{{h->dz3, h->dz2, h->dz1}, {h->g + h->off[5], h->g + h->off[3], h->g + h->off[1]},
                   {h->out_p, h->hid_p, h->hid_p}, {h->out, h->hid, h->hid}, h->part,
                   (int)tiles(h->out, B), h->loss};
    MCK(launch_k(k_colsum, dim3((std::max(h->out, h->hid) + kSumCols - 1) / kSumCols, 3), dim3(256), 0, h->stream, true, q, B));
    return LP_OK;
}

int load_x(lp_mlp* h, const float* X, int B, bool back) {
    if (B < 1 || B > h->maxb || !X) return LP_ERR_INVALID_ARG;
    MCK(launch_k(k_input16, dim3(tiles(h->in, B)), dim3(256), 0, h->stream, false, X,
                 B, h->in, h->x16, h->in_p, back ? h->xT : (__half*)nullptr, h->b_p));
    return LP_OK;
}

// the GEMMs' bounded waits: LP_ERR_TIMEOUT if one gave up
int check_err(lp_mlp* h) {
    int32_t e = 0;
    MCK(cudaMemcpyAsync(&e, h->err, sizeof(int32_t), cudaMemcpyDeviceToHost, h->stream));
    MCK(cudaStreamSynchronize(h->stream));
    return e ? LP_ERR_TIMEOUT : LP_OK;
}

}  // namespace

extern "C" {

int lp_mlp_create(lp_mlp** out, int32_t in_dim, int32_t hidden, int32_t out_dim, int32_t max_batch,
                  void* cuda_stream) {
    if (!out || in_dim < 1 || hidden < 1 || out_dim < 1 || max_batch < 1) return LP_ERR_INVALID_ARG;
    *out = nullptr;
    lp_mlp* h = new (std::nothrow) lp_mlp();
    if (!h) return LP_ERR_OOM;
    h->in = in_dim; h->hid = hidden; h->out = out_dim; h->maxb = max_batch;
    h->in_p = pad64(in_dim); h->hid_p = pad64(hidden); h->out_p = pad64(out_dim); h->b_p = pad64(max_batch);
    h->stream = static_cast<cudaStream_t>(cuda_stream);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&h->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        delete h;
        return LP_ERR_CUDA;
    }
    const size_t sz[6] = {(size_t)in_dim * hidden, (size_t)hidden, (size_t)hidden * hidden, (size_t)hidden,
                          (size_t)hidden * out_dim, (size_t)out_dim};
    size_t o = 0;
    for (int i = 0; i < 6; ++i) { h->off[i] = o; o += sz[i]; }
    h->np = o;
    const size_t B = max_batch, I = in_dim, H = hidden, O = out_dim;
    int rc = LP_OK;
    if ((rc = malloc_t(h, &h->p, o)) || (rc = malloc_t(h, &h->g, o)) || (rc = malloc_t(h, &h->m1, o)) ||
        (rc = malloc_t(h, &h->m2, o)) || (rc = malloc_t(h, &h->w1t, H * h->in_p)) ||
        (rc = malloc_t(h, &h->w2t, H * h->hid_p)) || (rc = malloc_t(h, &h->w3t, O * h->hid_p)) ||
        (rc = malloc_t(h, &h->w2n, H * h->hid_p)) || (rc = malloc_t(h, &h->w3n, H * h->out_p)) ||
        (rc = malloc_t(h, &h->x16, B * h->in_p)) || (rc = malloc_t(h, &h->xT, I * h->b_p)) ||
        (rc = malloc_t(h, &h->z1, B * H)) || (rc = malloc_t(h, &h->z2, B * H)) || (rc = malloc_t(h, &h->z3, B * O)) ||
        (rc = malloc_t(h, &h->a1, B * h->hid_p)) || (rc = malloc_t(h, &h->a2, B * h->hid_p)) ||
        (rc = malloc_t(h, &h->a1T, H * h->b_p)) || (rc = malloc_t(h, &h->a2T, H * h->b_p)) ||
        (rc = malloc_t(h, &h->dz3, B * h->out_p)) || (rc = malloc_t(h, &h->dz2, B * h->hid_p)) ||
        (rc = malloc_t(h, &h->dz1, B * h->hid_p)) || (rc = malloc_t(h, &h->dz3T, O * h->b_p)) ||
        (rc = malloc_t(h, &h->dz2T, H * h->b_p)) || (rc = malloc_t(h, &h->dz1T, H * h->b_p)) ||
        (rc = malloc_t(h, &h->part, ((O + kTile - 1) / kTile) * (h->b_p / kTile))) ||
        (rc = malloc_t(h, &h->loss, 1)) || (rc = malloc_t(h, &h->err, 1))) {
        lp_mlp_destroy(h);
        return rc;
    }
    bool ok = cudaMemsetAsync(h->p, 0, o * sizeof(float), h->stream) == cudaSuccess &&
              cudaMemsetAsync(h->m1, 0, o * sizeof(float), h->stream) == cudaSuccess &&
              cudaMemsetAsync(h->m2, 0, o * sizeof(float), h->stream) == cudaSuccess &&
              cudaMemsetAsync(h->err, 0, sizeof(int32_t), h->stream) == cudaSuccess;
    // the padding of the FP16 rows stays zero from here on
    const struct { __half* p; size_t n; } padded[] = {
        {h->w1t, H * h->in_p}, {h->w2t, H * h->hid_p}, {h->w3t, O * h->hid_p}, {h->w2n, H * h->hid_p},
        {h->w3n, H * h->out_p}, {h->x16, B * h->in_p}, {h->xT, I * h->b_p}, {h->a1, B * h->hid_p},
        {h->a2, B * h->hid_p}, {h->a1T, H * h->b_p}, {h->a2T, H * h->b_p}, {h->dz3, B * h->out_p},
        {h->dz2, B * h->hid_p}, {h->dz1, B * h->hid_p}, {h->dz3T, O * h->b_p}, {h->dz2T, H * h->b_p},
        {h->dz1T, H * h->b_p}};
    for (const auto& q : padded) ok = ok && cudaMemsetAsync(q.p, 0, q.n * sizeof(__half), h->stream) == cudaSuccess;
    if (!ok || refresh_weights(h) != LP_OK) {
        lp_mlp_destroy(h);
        return LP_ERR_CUDA;
    }
    *out = h;
    return LP_OK;
}

int64_t lp_mlp_num_params(const lp_mlp* h) { return h ? (int64_t)h->np : -1; }

int lp_mlp_set_params(lp_mlp* h, const float* params) {
    if (!h || !params) return LP_ERR_INVALID_ARG;
    MCK(cudaMemcpyAsync(h->p, params, h->np * sizeof(float), cudaMemcpyHostToDevice, h->stream));
    int rc = refresh_weights(h);
    if (rc != LP_OK) return rc;
    MCK(cudaMemsetAsync(h->m1, 0, h->np * sizeof(float), h->stream));
    MCK(cudaMemsetAsync(h->m2, 0, h->np * sizeof(float), h->stream));
    h->steps = 0;
    MCK(cudaStreamSynchronize(h->stream));
    return LP_OK;
}

int lp_mlp_get_params(const lp_mlp* h, float* params) {
    if (!h || !params) return LP_ERR_INVALID_ARG;
    MCK(cudaMemcpyAsync(params, h->p, h->np * sizeof(float), cudaMemcpyDeviceToHost, h->stream));
    MCK(cudaStreamSynchronize(h->stream));
    return LP_OK;
}

int lp_mlp_forward(lp_mlp* h, const float* X, int32_t batch, float* logits) {
    if (!h || !logits) return LP_ERR_INVALID_ARG;
    int rc = load_x(h, X, batch, false);
    if (rc != LP_OK) return rc;
    if ((rc = hidden_layers(h, batch, false)) != LP_OK) return rc;
    return gemm(h, batch, h->out, h->hid, h->a2, h->hid_p, h->w3t, h->hid_p,
                EpiAct{h->p + h->off[5], logits, nullptr, nullptr, 0, 0, batch, h->out});
}

int lp_mlp_gradients(lp_mlp* h, const float* X, const float* T, int32_t batch, float* grads, float* loss) {
    if (!h || !T) return LP_ERR_INVALID_ARG;
    int rc = load_x(h, X, batch, true);
    if (rc != LP_OK) return rc;
    if ((rc = forward_backward(h, batch, T)) != LP_OK) return rc;
    if (grads) MCK(cudaMemcpyAsync(grads, h->g, h->np * sizeof(float), cudaMemcpyDeviceToHost, h->stream));
    if (loss) MCK(cudaMemcpyAsync(loss, h->loss, sizeof(float), cudaMemcpyDeviceToHost, h->stream));
    return check_err(h);
}

int lp_mlp_train_step(lp_mlp* h, const float* X, const float* T, int32_t batch, float lr, float* loss) {
    if (!h || !T || !(lr > 0.f)) return LP_ERR_INVALID_ARG;
    int rc = load_x(h, X, batch, true);
    if (rc != LP_OK) return rc;
    if ((rc = forward_backward(h, batch, T)) != LP_OK) return rc;
    h->steps++;
    if ((rc = refresh_weights(h, lr)) != LP_OK) return rc;
    if (loss) {
        MCK(cudaMemcpyAsync(loss, h->loss, sizeof(float), cudaMemcpyDeviceToHost, h->stream));
        return check_err(h);
    }
    return LP_OK;
}

void lp_mlp_destroy(lp_mlp* h) {
    if (!h) return;
    if (h->stream) cudaStreamSynchronize(h->stream);
    for (void* p : h->allocs) cudaFree(p);
    delete h;
}

}  // extern "C"
