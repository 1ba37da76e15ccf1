// price_static.cu -- reduced costs and Dantzig's entering choice without any
// allocation (lp_price_static in include/lpgb.h).
//
// Some callers cannot allocate device memory: code running inside a CUDA
// graph they capture themselves, allocator-free embedded runtimes, or hosts
// whose memory budget is fixed up front.  This entry point takes only the
// caller's buffers.  The one piece of scratch the kernel needs -- a partial
// best candidate per block plus the last-block ticket -- lives in a
// file-scope __device__ array, so every GPU that loads the library holds it
// (about 17 KB) until the process exits.
//
// Host code must not hand the array's name to a kernel: in host code the name
// is only a host-side stand-in.  The device address is fetched once per
// device context with cudaGetSymbolAddress (with that device current) and
// passed in; a call that finds a different context on its device than the
// one the address was fetched in (after cudaDeviceReset, say) fetches it again.
#include "../../include/lpgb.h"

#include <cuda.h>
#include <cuda_runtime.h>

#include <cfloat>
#include <cstdint>
#include <mutex>

namespace {

constexpr int kThreads = 512;
constexpr int kMaxBlocks = 1024;   // partial slots in the static scratch
constexpr int kMaxDevices = 64;

struct Best {
    double d;
    int32_t j;
    int32_t pad;
};

struct Scratch {
    Best part[kMaxBlocks];
    int32_t ticket;  // must be zero when a launch starts
    int32_t pad[63];
};

static __device__ __align__(256) Scratch g_price_scratch;

struct DeviceSetup {
    bool ready = false;
    unsigned long long ctx_id = 0;  // the context the address below belongs to
    Scratch* scratch = nullptr;     // device address of g_price_scratch
    int sms = 0;
};
DeviceSetup g_setup[kMaxDevices];
std::mutex g_setup_mutex;

__device__ __forceinline__ bool better(double da, int ja, double db, int jb) {
    if (ja < 0) return false;
    if (jb < 0) return true;
    return da > db || (da == db && ja < jb);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// v != 0 (a NaN is), by its bits: an FP64 compare costs the pipe as much as an FMA.
__device__ __forceinline__ bool nonzero(double v) {
    return ((unsigned long long)__double_as_longlong(v) << 1) != 0;
}

// Block-wide best (d, j); valid in thread 0.
__device__ void block_best(double& d, int& j) {
    __shared__ double sd[32];
    __shared__ int sj[32];
    for (int o = 16; o > 0; o >>= 1) {
        const double od = __shfl_xor_sync(0xffffffffu, d, o);
        const int oj = __shfl_xor_sync(0xffffffffu, j, o);
        if (better(od, oj, d, j)) { d = od; j = oj; }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) { sd[w] = d; sj[w] = j; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < (int)(blockDim.x >> 5); ++i)
            if (better(sd[i], sj[i], d, j)) { d = sd[i]; j = sj[i]; }
    }
}

// At the duals of a solve under way y_i is zero on every row with a basic slack, so
// only the rows with a nonzero y_i are read when they are few.  The dense pass is
// bound by the FP64 pipe (an FMA per 8 bytes): 82 us a call at 4096 x 8192.  With one
// row in twelve the list takes a twelfth of the FMAs and, in 128-byte pieces, 202 of
// A's 268 MB: 49 us, bound by DRAM.  From a cold L2 the two take 84 and 64, and one row
// in four 76; one in three would read nearly every piece and gains nothing (dense again).
// Where no warp has a second column, each waits for its chain of gathers: 12288 x 700
// takes 66 us dense, 57 with one row in twelve and 85 with one in four, so the line is
// one in eight there.  Below kSparseMin rows there is nothing to gain, and the duals are
// not even counted (100 x 200, its memset included: 10.4 us, 11.1 with the list).
constexpr int kSparse = 4, kSparseFew = 8, kSparseMin = 512;

// The best of the block's columns from the rows with a dual alone (nz of them).  A function of its own: inlined beside it, the dense
// pass's loop is scheduled worse (82 us instead of 66 at 12288 x 700).
__device__ __noinline__ Best sparse_columns(int m, int nz, const double* __restrict__ A, int lda,
                                            const double* __restrict__ c,
                                            const int32_t* __restrict__ pos, int owned) {
    extern __shared__ __align__(16) double ysh[];
    __shared__ int wn[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int G = gridDim.x, me = (m + 1) & ~1;
    double best_d = -DBL_MAX;
    int best_j = -1;
    // the rows with a dual, in increasing order: each warp counts and then writes
    // those of its run of rows
    uint16_t* nzi = reinterpret_cast<uint16_t*>(ysh + me);
    const int run = ((m + nw - 1) / nw + 31) & ~31;
    const int r0 = min(m, warp * run), r1 = min(m, r0 + run);
    int mine = 0;
    for (int k = r0; k < r1; k += 32)
        mine += __popc(__ballot_sync(0xffffffffu, k + lane < r1 && nonzero(ysh[k + lane])));
    __syncthreads();
    if (lane == 0) wn[warp] = mine;
    __syncthreads();
    int at = 0;
    for (int w = 0; w < warp; ++w) at += wn[w];
    for (int k = r0; k < r1; k += 32) {
        const bool in = k + lane < r1 && nonzero(ysh[k + lane]);
        const unsigned bal = __ballot_sync(0xffffffffu, in);
        if (in) nzi[at + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(k + lane);
        at += __popc(bal);
    }
    __syncthreads();
    // two columns per warp at a time, eight gathers in flight per lane
    for (int l = warp; l < owned; l += 2 * nw) {
        const int j0 = blockIdx.x + G * l, j1 = j0 + G * nw;
        const bool in0 = pos[j0] < 0, in1 = l + nw < owned && pos[j1] < 0;
        const double* c0 = A + (size_t)j0 * lda;
        const double* c1 = A + (size_t)(in1 ? j1 : j0) * lda;
        double a0 = 0.0, a1 = 0.0;
#pragma unroll 8
        for (int t = lane; t < nz; t += 32) {
            const int i = nzi[t];
            const double v = ysh[i], u0 = __ldg(c0 + i), u1 = __ldg(c1 + i);
            a0 = fma(u0, v, a0);
            a1 = fma(u1, v, a1);
        }
        const double d0 = c[j0] - warp_sum(a0);
        if (in0 && better(d0, j0, best_d, best_j)) { best_d = d0; best_j = j0; }
        if (in1) {  // (uniform over the warp)
            const double d1 = c[j1] - warp_sum(a1);
            if (better(d1, j1, best_d, best_j)) { best_d = d1; best_j = j1; }
        }
    }
    return {best_d, best_j, 0};
}

// d_j = c_j - y^T a_j for nonbasic j (d_{n+i} = -y_i for slacks); the block
// that finishes last writes the largest d_j > tol_d (exact ties to the
// smallest j) to q_out / dq_out, or q_out = -1 when none exceeds tol_d.
// kList: m >= kSparseMin.
template <bool kList>
__global__ void __launch_bounds__(kThreads) k_price_static(int m, int n, const double* __restrict__ A, int lda,
                                                           const double* __restrict__ c,
                                                           const double* __restrict__ y,
                                                           const int32_t* __restrict__ pos, double tol_d,
                                                           int32_t* q_out, double* dq_out, Scratch* sc) {
    extern __shared__ __align__(16) double ysh[];  // read as double2 below
    const int me = (m + 1) & ~1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __shared__ int wn[kThreads / 32];
    int duals = 0;
#pragma unroll 4
    for (int k = threadIdx.x; k < me; k += blockDim.x) {
        const double v = k < m ? y[k] : 0.0;
        ysh[k] = v;
        if (kList) duals += nonzero(v);
    }
    if (kList) {
        duals = __reduce_add_sync(0xffffffffu, duals);
        if (lane == 0) wn[warp] = duals;
    }
    __syncthreads();
    int nz = 0;
    if (kList)
        for (int w = 0; w < nw; ++w) nz += wn[w];
    const int half = m >> 1;
    const double2* y2 = reinterpret_cast<const double2*>(ysh);
    double best_d = -DBL_MAX;
    int best_j = -1;
    const int G = gridDim.x;
    const int owned = (n - (int)blockIdx.x + G - 1) / G;
    const bool sparse = kList && nz <= m / (owned > nw ? kSparse : kSparseFew);
    if (sparse) {
        const Best b = sparse_columns(m, nz, A, lda, c, pos, owned);
        best_d = b.d;
        best_j = b.j;
    }
    for (int l = warp; l < owned && !sparse; l += nw) {
        const int j = blockIdx.x + G * l;
        if (pos[j] >= 0) continue;
        const double* colp = A + (size_t)j * lda;
        const double2* col = reinterpret_cast<const double2*>(colp);
        double a0 = 0.0, a1 = 0.0;
#pragma unroll 4
        for (int k = lane; k < half; k += 32) {
            const double2 u = __ldg(col + k), w = y2[k];
            a0 = fma(u.x, w.x, a0);
            a1 = fma(u.y, w.y, a1);
        }
        if ((m & 1) && lane == 0) a0 = fma(__ldg(colp + m - 1), ysh[m - 1], a0);
        const double d = c[j] - warp_sum(a0 + a1);
        if (better(d, j, best_d, best_j)) { best_d = d; best_j = j; }
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
        const int j = n + i;
        if (pos[j] >= 0) continue;
        const double d = -ysh[i];
        if (better(d, j, best_d, best_j)) { best_d = d; best_j = j; }
    }
    block_best(best_d, best_j);
    __shared__ int last;
    if (threadIdx.x == 0) {
        sc->part[blockIdx.x].d = best_d;
        sc->part[blockIdx.x].j = best_j;
        __threadfence();
        last = atomicAdd(&sc->ticket, 1) == G - 1;
    }
    __syncthreads();
    if (!last) return;
    double d = -DBL_MAX;
    int j = -1;
    for (int b = threadIdx.x; b < G; b += blockDim.x) {
        const double od = __ldcg(&sc->part[b].d);
        const int oj = __ldcg(&sc->part[b].j);
        if (better(od, oj, d, j)) { d = od; j = oj; }
    }
    block_best(d, j);
    if (threadIdx.x == 0) {
        *q_out = (j >= 0 && d > tol_d) ? j : -1;
        *dq_out = j >= 0 ? d : 0.0;
        sc->ticket = 0;
    }
}

// y, and the rows of its nonzeros: 8.5 m bytes, two blocks per SM up to the largest m (with
// their values and 32-bit rows, 11 m bytes, one block above 10,400 rows: 12288 x 4096
// took 171 us dense instead of 123)
size_t price_smem(int m) {
    return (size_t)((m + 1) & ~1) * sizeof(double) + (size_t)(m / kSparse) * sizeof(uint16_t);
}

// Identity of the calling thread's current context (driver entry points
// looked up through the runtime, so the library needs no libcuda at link
// time).  Host-only queries: they enqueue nothing and allocate nothing.
typedef CUresult (*CtxGetCurrentFn)(CUcontext*);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long*);

int current_ctx_id(unsigned long long* id) {
    static CtxGetCurrentFn get_current = nullptr;
    static CtxGetIdFn get_id = nullptr;
    if (!get_current || !get_id) {
        void* f0 = nullptr;
        void* f1 = nullptr;
        cudaDriverEntryPointQueryResult q0, q1;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f0, 12000, cudaEnableDefault, &q0) != cudaSuccess ||
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &f1, 12000, cudaEnableDefault, &q1) != cudaSuccess ||
            q0 != cudaDriverEntryPointSuccess || q1 != cudaDriverEntryPointSuccess || !f0 || !f1)
            return LP_ERR_CUDA;
        get_current = reinterpret_cast<CtxGetCurrentFn>(f0);
        get_id = reinterpret_cast<CtxGetIdFn>(f1);
    }
    CUcontext ctx = nullptr;
    if (get_current(&ctx) != CUDA_SUCCESS || ctx == nullptr) return LP_ERR_CUDA;
    if (get_id(ctx, id) != CUDA_SUCCESS) return LP_ERR_CUDA;
    return LP_OK;
}

// Once per device context, with that device current: the scratch's device
// address, the shared-memory opt-in and the SM count.
int setup_device(int dev, DeviceSetup** out) {
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    DeviceSetup& s = g_setup[dev];
    unsigned long long ctx_id = 0;
    if (current_ctx_id(&ctx_id) != LP_OK) return LP_ERR_CUDA;
    if (s.ready && s.ctx_id != ctx_id) s.ready = false;  // a new context: the old address is void
    if (!s.ready) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_price_scratch) != cudaSuccess || ptr == nullptr) return LP_ERR_CUDA;
        if (cudaFuncSetAttribute(k_price_static<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)price_smem(LP_PRICE_STATIC_MAX_M)) != cudaSuccess)
            return LP_ERR_CUDA;
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
            return LP_ERR_CUDA;
        s.scratch = static_cast<Scratch*>(ptr);
        s.sms = sms;
        s.ctx_id = ctx_id;
        s.ready = true;
    }
    *out = &s;
    return LP_OK;
}

}  // namespace

extern "C" int lp_price_static(int32_t m, int32_t n, const double* A_colmajor, int32_t lda, const double* c,
                               const double* y, const int32_t* pos, double tol_d, int32_t* q_out,
                               double* dq_out, void* cuda_stream) {
    if (m < 1 || n < 1 || m > LP_PRICE_STATIC_MAX_M || (int64_t)n + m > ((int64_t)1 << 30)) return LP_ERR_INVALID_ARG;
    if (lda < m || (lda & 1)) return LP_ERR_INVALID_ARG;
    if (!A_colmajor || !c || !y || !pos || !q_out || !dq_out) return LP_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(A_colmajor) & 15) != 0 || !(tol_d >= 0)) return LP_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return LP_ERR_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return LP_ERR_INVALID_ARG;
    DeviceSetup* s = nullptr;
    int rc = setup_device(dev, &s);
    if (rc != LP_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    int blocks = 2 * s->sms;
    if (blocks > kMaxBlocks) blocks = kMaxBlocks;
    if (blocks > n) blocks = n;
    if (cudaMemsetAsync(&s->scratch->ticket, 0, sizeof(int32_t), st) != cudaSuccess) return LP_ERR_CUDA;
    const size_t smem = price_smem(m);
    const auto kernel = m >= kSparseMin ? k_price_static<true> : k_price_static<false>;
    kernel<<<blocks, kThreads, smem, st>>>(m, n, A_colmajor, lda, c, y, pos, tol_d, q_out, dq_out, s->scratch);
    if (cudaGetLastError() != cudaSuccess) return LP_ERR_CUDA;
    return LP_OK;
}
