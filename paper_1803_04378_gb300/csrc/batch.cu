// batch.cu -- many small LPs in persistent launches (lp_batch_* in include/lpgb.h).
//
// Each CTA solves whole LPs, one at a time, taking the next one from an atomic
// work queue: the full revised simplex of Section 2.1 (Steps 3-8, Figure 1
// tableau with the explicit B^-1), the tabu rule of Sections 2.2/3.4 with the
// same aspiration and Bland safety net as the single-LP solver, and
// structure-aware reinversion every `reinvert_every` pivots.  LPs are grouped
// into size buckets (m <= 64, 128, 192, 256); every bucket has its own
// persistent kernel whose thread count and B^-1 residency (shared memory or
// an L2-resident global slot per CTA) come from the autotuner.  The bucket
// kernels run side by side on forked streams, captured together as one CUDA
// graph, so the tail of one bucket overlaps the others.  Inside a bucket the
// largest LPs go first so the tail is made of small ones.
//
// PRICE (price_mode 1, the default for batches): a BF16 copy of A screens the
// columns with FP32 FMAs, the top k are re-priced in FP64, and the full FP64
// PRICE runs whenever no candidate improves or Bland's rule is on.  FTRAN, the
// ratio test, the B^-1 update and reinversion are FP64.
//
// B^-1 is kept in slack-structured form: only the columns of rows whose slack is
// nonbasic, column-major, so that a thread per row reads consecutive addresses.
#include "iter_common.cuh"
#include "lpgb_internal.cuh"
#include "../../include/lpgb.h"

#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

namespace lpgb {

struct BatchLP {
    int32_t m, n;
    int64_t a_off;   // into A (row-major m x n) and A_lp
    int32_t r_off;   // into b / y (m values)
    int32_t c_off;   // into c / x (n values)
};

struct BatchParams {
    int32_t reinvert_every, tabu_tenure, max_iters, bland_after, price_mode, topk, trace_cap;
    double tol_d, tol_piv, tol_tie;
};

struct BatchState {
    BatchParams p;
    const BatchLP* lps;
    const int32_t* order;       // LP indices, bucket by bucket, largest first
    const double* A;
    const uint16_t* A_lp;       // BF16 copy (price_mode 1)
    const double* b;
    const double* c;
    int32_t* status;
    int32_t* iters;
    double* obj;
    double* x;
    double* y;
    int32_t* queue;             // one counter per bucket
    double* scratch[4];         // per bucket, per-CTA slots: [B^-1 if global] [reinversion block]
    int64_t slot_doubles[4];    // 2 * (bucket's largest m)^2
    int32_t* trace_q;
    int32_t* trace_r;
};

constexpr int kBuckets = 4;
static_assert(sizeof(BatchState::scratch) / sizeof(double*) == kBuckets, "one scratch area per bucket");
constexpr int kBucketM[kBuckets] = {64, 128, 192, 256};
constexpr int kBatchMaxM = 256;
constexpr int kBatchMaxN = 512;
constexpr int kBatchTopk = 8;
constexpr int kSlotsPerSm = 8;  // scratch slots per SM and bucket (CTAs per SM at most)
constexpr int kSmemCols = 16;   // live columns of B^-1 in shared memory where the tuning asks for it

namespace {

__device__ __forceinline__ float bf16f(uint16_t v) { return __uint_as_float((uint32_t)v << 16); }

// order-preserving integer image of a float (no NaN; -0 and +0 share one key)
__device__ __forceinline__ int fkey(float x) {
    int b = __float_as_int(x);
    if ((b & 0x7fffffff) == 0) b = 0;
    return b >= 0 ? b : (b ^ 0x7fffffff);
}

// Scalars of the LP being solved and the block's reduction scratch (shared memory).
struct LPScal {
    int status, it, degen_run, bland, flags, k, err;
    double z;
};
struct Red {
    int gmax[32];              // screen: the largest key of each lane's columns over all warps
    int lcount, lkey[32], lj[32];  // columns at or above the top-K threshold
    int sel[16][kBatchTopk];   // per warp: the top K of the list, best first
    double cd[kBatchTopk];     // their exact reduced costs
    int cj[kBatchTopk];
    long long wk[16];          // per warp: a key,
    int wj[16], wv[16], wc[16];  // an index, a variable, a count
    double wa[16], wt[16];
    double dq;
};

// Argmax of (key, j) over the block's valid candidates, exact ties to the smallest j
// (j = -1 when there is none); every thread gets the result.
template <int T>
__device__ __forceinline__ void block_best(long long key, int j, Red& R, long long& kbest, int& jbest) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long kb;
    const int win = warp_argmax_key(key, j, j >= 0, kb);
    if (lane == (win < 0 ? 0 : win)) { R.wk[w] = kb; R.wj[w] = win < 0 ? -1 : j; }
    __syncthreads();
    kbest = R.wk[0];
    jbest = R.wj[0];
#pragma unroll
    for (int i = 1; i < T / 32; ++i)
        if (beats(R.wk[i], R.wj[i], kbest, jbest)) { kbest = R.wk[i]; jbest = R.wj[i]; }
    __syncthreads();
}

// ---------------------------------------------------------------- one LP
// The method on the slack-structured inverse (kernels_struct.cu): only the k columns
// of B^-1 that belong to rows with a nonbasic slack differ from unit columns and
// only their duals from zero, so PRICE, FTRAN and the update work on k rows or
// columns and the slack basis needs no initialisation.  The batch's LPs end
// after 30 pivots on average, so k is far below m.
//
// Threads own rows (i = tid, tid + T, ..) through FTRAN, the ratio test and the update
// -- alpha, the ratio and the row's entries never leave the thread -- and columns
// (j = tid, tid + T, ..) through the screen, which then reads a live row of A
// coalesced.  Live column t lies in shared memory for t < ks, else in the CTA's
// L2-resident slot.
//
// What bounds it: the FP64 pipe (2 k m FMAs and m divisions a pivot, about 4 us of an
// SM at m = 225, k = 25; 65% of the time on 4096 LPs) and, with few LPs, the latency of
// a pivot (7.8 us at m <= 128).  Against the dense m x m inverse: 4096 LPs
// of m 16..256 30.6 -> 3.3 ms, 48 LPs of m 16..128 1.04 -> 0.39 ms, the same pivots.
// LPs whose rows all become live (k = m), the dense inverse's best case: 1024 of
// m 128..256 114 -> 78 ms, 48 of m 100..128 4.0 -> 3.7, 48 of m 60..64 1.10 -> 0.98.
//
// kPair (2 m <= T): two lanes per row, lane 2 i for the even live columns of row i and lane
// 2 i + 1 for the odd ones, which are FTRAN's two sums anyway; a thread per row
// leaves half of the warps idle (the 48 LPs of m 60..64: 1.14 ms).
template <int T, bool kPair>
__device__ void solve_one(const BatchState& s, int lp, unsigned char* smem, double* slot, int mmax, int nmax, int ks) {
    const BatchParams& P = s.p;
    const BatchLP L = s.lps[lp];
    const int m = L.m, n = L.n, N = n + m;
    const double* A = s.A + L.a_off;
    const uint16_t* Alp = s.A_lp ? s.A_lp + L.a_off : nullptr;
    const double* b = s.b + L.r_off;
    const double* c = s.c + L.c_off;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int W = T / 32;
    constexpr int VR = kPair ? 1 : (kBatchMaxM + T - 1) / T;  // rows and columns per thread
    constexpr int VC = (kBatchMaxN + T - 1) / T;

    // shared-memory carve-up (sizes by the bucket's largest LP)
    double* cs = reinterpret_cast<double*>(smem);  // live columns 0 .. ks - 1
    double* dp = cs + (size_t)ks * mmax;
    double* y = dp; dp += mmax;      // duals of the live rows, slot order
    double* rho = dp; dp += mmax;    // rho / alpha_r, slot order
    double* aq = dp; dp += mmax;     // the entering column on the live rows, slot order
    double* au = dp; dp += mmax;     // and on the row of position i's basic slack (zero: structural)
    double* bbar = dp; dp += mmax;
    float* y32 = reinterpret_cast<float*>(dp);
    float* cf = y32 + mmax;
    int* tabu = reinterpret_cast<int*>(cf + nmax);
    int16_t* basis = reinterpret_cast<int16_t*>(tabu + nmax + mmax);
    int16_t* pos = basis + mmax;
    int16_t* srow = pos + nmax + mmax;   // slot -> row
    int16_t* rslot = srow + mmax;        // row -> slot, -1: basic slack
    int16_t* lstP = rslot + mmax;
    int16_t* lstR = lstP + mmax;
    int16_t* pivrow = lstR + mmax;
    int16_t* pinv = pivrow + mmax;
    double* gcol = slot;                              // live columns ks ..
    double* Wm = slot + (size_t)mmax * mmax;          // reinversion block, k x k column-major
    auto col = [&](int t) -> double* { return t < ks ? cs + (size_t)t * m : gcol + (size_t)(t - ks) * m; };

    __shared__ LPScal S;
    __shared__ Red R;
    const int half = kPair ? tid & 1 : 0;
    auto row_of = [&](int v) { return kPair ? tid >> 1 : tid + T * v; };
    const long long ktol = dkey(P.tol_d), kpiv = dkey(P.tol_piv), kbig = dkey(DBL_MAX);

    // Step 1: slack basis
    for (int i = tid; i < m; i += T) {
        bbar[i] = b[i];
        basis[i] = (int16_t)(n + i);
        rslot[i] = -1;
        au[i] = 0.0;
    }
    for (int j = tid; j < N; j += T) {
        pos[j] = (int16_t)(j < n ? -1 : j - n);
        tabu[j] = 0;
        if (j < n) cf[j] = (float)c[j];
    }
    if (tid < 32) R.gmax[tid] = INT_MIN;
    if (tid == 0) {
        R.lcount = 0;
        S.status = kRunning; S.it = 0; S.degen_run = 0; S.bland = 0; S.flags = 0; S.err = 0; S.k = 0; S.z = 0.0;
    }
    __syncthreads();

    for (;;) {
        const int it = S.it, k = S.k;
        if (it >= P.max_iters) {
            if (tid == 0) S.status = kIterLimit;
            __syncthreads();
            break;
        }
        const bool bland = S.bland != 0;
        int q = -1;
        double dq = 0.0;
        // ---- Step 3/4: PRICE + CHUZC
        if (P.price_mode == 1 && !bland && Alp != nullptr) {
            // BF16 screen over nonbasic, non-tabu structural columns
            float acc[VC];
            bool live[VC];
#pragma unroll
            for (int v = 0; v < VC; ++v) {
                const int j = tid + T * v;
                live[v] = j < n && pos[j] < 0 && tabu[j] <= it;
                acc[v] = 0.f;
            }
#pragma unroll 4
            for (int t = 0; t < k; ++t) {
                const float yt = y32[t];
                const uint16_t* row = Alp + (size_t)srow[t] * n;
#pragma unroll
                for (int v = 0; v < VC; ++v)
                    if (live[v]) acc[v] = fmaf(yt, bf16f(__ldg(row + tid + T * v)), acc[v]);
            }
            int key[VC], top = INT_MIN;
#pragma unroll
            for (int v = 0; v < VC; ++v) {
                key[v] = live[v] ? fkey(cf[tid + T * v] - acc[v]) : INT_MIN;
                top = max(top, key[v]);
            }
            if (top != INT_MIN) atomicMax(&R.gmax[lane], top);
            __syncthreads();
            // The K-th largest of the 32 lanes' maxima is at most the K-th largest
            // column: the columns at or above it hold the top K (about 10 of them).
            const int K = P.topk < kBatchTopk ? P.topk : kBatchTopk;
            const int g = R.gmax[lane];
            int rank = 0;
#pragma unroll 8
            for (int o = 0; o < 32; ++o) {
                const int x = __shfl_sync(0xffffffffu, g, o);
                rank += x > g || (x == g && o < lane);
            }
            const int tau = max(__shfl_sync(0xffffffffu, g, __ffs(__ballot_sync(0xffffffffu, rank == K - 1)) - 1),
                                INT_MIN + 1);
#pragma unroll
            for (int v = 0; v < VC; ++v)
                if (key[v] >= tau) {
                    const int e = atomicAdd(&R.lcount, 1);
                    if (e < 32) { R.lkey[e] = key[v]; R.lj[e] = tid + T * v; }
                }
            __syncthreads();
            int cnt = R.lcount;
            if (cnt <= 32) {
                // rank the list (larger key, then smaller index); every warp alike
                const int lk = lane < cnt ? R.lkey[lane] : INT_MIN, lj = lane < cnt ? R.lj[lane] : INT_MAX;
                int lr = lane;
                if (cnt > K) {
                    lr = 0;
                    for (int o = 0; o < cnt; ++o) {
                        const int ok = __shfl_sync(0xffffffffu, lk, o), oj = __shfl_sync(0xffffffffu, lj, o);
                        lr += ok > lk || (ok == lk && oj < lj);
                    }
                }
                if (lane < cnt && lr < K) R.sel[warp][lr] = lj;
                __syncwarp();
            } else {
                // more equal columns than the list holds: K rounds of block argmax
                bool taken[VC];
#pragma unroll
                for (int v = 0; v < VC; ++v) taken[v] = key[v] < tau;
                for (int x = 0; x < K; ++x) {
                    long long bk = LLONG_MIN;
                    int bj = -1;
#pragma unroll
                    for (int v = 0; v < VC; ++v)
                        if (!taken[v] && beats(key[v], tid + T * v, bk, bj)) { bk = key[v]; bj = tid + T * v; }
                    block_best<T>(bk, bj, R, bk, bj);
#pragma unroll
                    for (int v = 0; v < VC; ++v) taken[v] |= bj == tid + T * v;
                    if (lane == 0) R.sel[warp][x] = bj;
                }
                __syncwarp();
                cnt = K;
            }
            cnt = min(cnt, K);
            // exact FP64 re-price: eight lanes per candidate
            const int id = tid >> 3, g8 = tid & 7;
            {
                const bool mine = id < cnt;
                const int j = mine ? R.sel[warp][id] : 0;
                double a = 0.0;
                if (4 * warp < cnt) {
                    if (mine)
                        for (int t = g8; t < k; t += 8) a = fma(y[t], __ldg(A + (size_t)srow[t] * n + j), a);
                    a += __shfl_xor_sync(0xffffffffu, a, 4);
                    a += __shfl_xor_sync(0xffffffffu, a, 2);
                    a += __shfl_xor_sync(0xffffffffu, a, 1);
                    if (mine && g8 == 0) { R.cd[id] = c[j] - a; R.cj[id] = j; }
                }
            }
            __syncthreads();
            // the best of them and of the non-tabu slacks (d = -y), every warp alike
            long long bk = LLONG_MIN;
            int bj = -1;
            if (lane < cnt) { bk = dkey(R.cd[lane]); bj = R.cj[lane]; }
            for (int t = lane; t < k; t += 32) {
                const int j = n + srow[t];
                const long long kd = dkey(-y[t]);
                if (tabu[j] <= it && beats(kd, j, bk, bj)) { bk = kd; bj = j; }
            }
            long long kb;
            const int win = warp_argmax_key(bk, bj, bj >= 0, kb);
            if (win >= 0 && kb > ktol) {
                q = __shfl_sync(0xffffffffu, bj, win);
                dq = kdouble(kb);
            }
        }
        if (q < 0) {
            // full FP64 PRICE (the oracle's rule, tabu and aspiration included)
            double d[VC];
#pragma unroll
            for (int v = 0; v < VC; ++v) d[v] = 0.0;
            for (int t = 0; t < k; ++t) {
                const double yt = y[t];
                const double* row = A + (size_t)srow[t] * n;
#pragma unroll
                for (int v = 0; v < VC; ++v)
                    if (tid + T * v < n) d[v] = fma(yt, __ldg(row + tid + T * v), d[v]);
            }
            long long ka = LLONG_MIN, kn = LLONG_MIN, km = LLONG_MIN;
            int ja = -1, jn = -1, jm = -1;
            auto offer = [&](double dv, int j) {
                const long long kd = dkey(dv);
                if (beats(kd, j, ka, ja)) { ka = kd; ja = j; }
                if (tabu[j] <= it && beats(kd, j, kn, jn)) { kn = kd; jn = j; }
                if (kd > ktol && (jm < 0 || j < jm)) jm = j;
            };
#pragma unroll
            for (int v = 0; v < VC; ++v) {
                const int j = tid + T * v;
                if (j < n) d[v] = c[j] - d[v];
                if (j < n && pos[j] < 0) offer(d[v], j);
            }
            for (int t = tid; t < k; t += T) offer(-y[t], n + srow[t]);
            block_best<T>(ka, ja, R, ka, ja);
            block_best<T>(kn, jn, R, kn, jn);
            if (bland) {
                // smallest improving index: argmax of -j
                km = jm >= 0 ? -(long long)jm : LLONG_MIN;
                block_best<T>(km, jm, R, km, jm);
            }
            if (ja < 0 || !(ka > ktol)) {
                if (tid == 0) S.status = kOptimal;
                __syncthreads();
                break;
            }
            if (bland) {
                q = jm;
#pragma unroll
                for (int v = 0; v < VC; ++v)
                    if (tid + T * v == q) R.dq = d[v];
                if (q >= n && tid == 0) R.dq = -y[rslot[q - n]];
                __syncthreads();
                dq = R.dq;
                if (tid == 0) S.flags |= kTfBland;
            } else if (jn >= 0 && kn > ktol) {
                q = jn;
                dq = kdouble(kn);
            } else {
                q = ja;
                dq = kdouble(ka);
                if (tid == 0) S.flags |= kTfAspiration;
            }
        }
        // ---- Step 5: FTRAN alpha = B^-1 a_q
        if (q < n) {
            for (int i = tid; i < m; i += T) {
                const double v = __ldg(A + (size_t)i * n + q);
                if (rslot[i] >= 0) aq[rslot[i]] = v;
                else au[pos[n + i]] = v;
            }
        } else {
            const int unit = rslot[q - n];
            for (int t = tid; t < k; t += T) aq[t] = t == unit ? 1.0 : 0.0;
        }
        __syncthreads();
        double al[VR], th[VR];
        long long kth[VR], kmin = kbig;
#pragma unroll
        for (int v = 0; v < VR; ++v) {
            const int i = row_of(v);
            double a0 = 0.0, a1 = 0.0;
            kth[v] = kbig;
            al[v] = th[v] = 0.0;
            if (i < m) {
                const double unit = q < n && basis[i] >= n ? au[i] : 0.0;
                if (kPair) {
#pragma unroll 4
                    for (int t = half; t < k; t += 2) a0 = fma(col(t)[i], aq[t], a0);
                    if (half) a0 += unit;
                } else {
                    int t = 0;
#pragma unroll 4
                    for (; t + 1 < k; t += 2) {
                        a0 = fma(col(t)[i], aq[t], a0);
                        a1 = fma(col(t + 1)[i], aq[t + 1], a1);
                    }
                    if (t < k) a0 = fma(col(t)[i], aq[t], a0);
                    a1 += unit;
                }
            }
            if (kPair) a1 = __shfl_xor_sync(0xffffffffu, a0, 1);
            if (i < m) {
                al[v] = a0 + a1;
                // ratios one row per lane: a warp-wide division covers its rows
                if (!half && dkey(al[v]) > kpiv) {
                    th[v] = bbar[i] / al[v];
                    kth[v] = dkey(th[v]);
                }
            }
            kmin = min(kmin, kth[v]);
        }
        // ---- Step 6: CHUZR with the tie set (on integer keys)
        kmin = warp_min_key(kmin);
        if (lane == 0) R.wk[warp] = kmin;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < W; ++w) kmin = min(kmin, R.wk[w]);
        if (kmin == kbig) {
            if (tid == 0) S.status = kUnbounded;
            __syncthreads();
            break;
        }
        // (max(1, |t|) by its bits: FP64 compares would cost the pipe as much as the FMA)
        const double tmin = kdouble(kmin);
        const long long mag = __double_as_longlong(tmin) & 0x7fffffffffffffffLL;
        const long long kthr = dkey(tmin + P.tol_tie * __longlong_as_double(max(mag, __double_as_longlong(1.0))));
        {
            // the warp's best tied row: largest alpha, exact ties to the smallest basic
            // variable (Bland: the smallest basic variable)
            long long ka = LLONG_MIN;
            int var = INT_MAX, row = -1, cnt = 0;
            double bt = 0.0, ba = 0.0;
#pragma unroll
            for (int v = 0; v < VR; ++v)
                if (kth[v] <= kthr && kth[v] != kbig) {
                    const int x = basis[row_of(v)];
                    const long long kv = dkey(al[v]);
                    ++cnt;
                    if (row < 0 || (bland ? x < var : (kv > ka || (kv == ka && x < var)))) {
                        ka = kv; var = x; row = row_of(v); bt = th[v]; ba = al[v];
                    }
                }
            const unsigned bal = __ballot_sync(0xffffffffu, row >= 0);
            int win = bal ? __ffs(bal) - 1 : 0;
            if (bal && (__popc(bal) > 1 || __any_sync(0xffffffffu, cnt > 1))) {
                long long kb;
                win = bland ? warp_argmin_index(var, row >= 0) : warp_argmax_key(ka, var, row >= 0, kb);
                cnt = __reduce_add_sync(0xffffffffu, cnt);
            }
            if (lane == win) { R.wj[warp] = row; R.wv[warp] = var; R.wc[warp] = cnt; R.wa[warp] = ba; R.wt[warp] = bt; }
        }
        __syncthreads();
        int r = -1, leave = 0, ties = 0, bw = 0;
        {
            long long ka = LLONG_MIN;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                if (R.wj[w] < 0) continue;
                const long long kv = dkey(R.wa[w]);
                ties += R.wc[w];
                if (r < 0 || (bland ? R.wv[w] < leave : (kv > ka || (kv == ka && R.wv[w] < leave)))) {
                    ka = kv; leave = R.wv[w]; r = R.wj[w]; bw = w;
                }
            }
        }
        const double ar = R.wa[bw], theta = R.wt[bw];
        // ---- Step 7/8: the slots after the pivot, rho and y (in the new slot order)
        const int join = leave >= n ? leave - n : -1, ent = q >= n ? q - n : -1;
        const int te = ent >= 0 ? rslot[ent] : -1;
        const int J = join >= 0 ? (ent >= 0 ? te : k) : -1;             // the joining row's slot
        const int src = ent >= 0 && join < 0 && te != k - 1 ? k - 1 : -1;  // slot that moves to te
        const int kn = k + (join >= 0) - (ent >= 0);
        const int srcrow = src >= 0 ? srow[src] : -1;
        for (int t = tid; t < kn; t += T) {
            const int o = t == te && src >= 0 ? src : t;
            const double rn = (t == J ? 1.0 : col(o)[r]) / ar;
            const double yo = t == J ? 0.0 : y[o];
            rho[t] = rn;
            const double yn = __dadd_rn(yo, __dmul_rn(dq, rn));
            y[t] = yn;
            y32[t] = (float)yn;
        }
        __syncthreads();
        // bookkeeping (tabu, trace, objective, basis, slots)
        if (tid == T - 1) {
            int flags = S.flags;
            const bool degenerate = theta <= P.tol_tie;
            if (degenerate) flags |= kTfDegenerate;
            if (P.tabu_tenure > 0 && (ties > 1 || degenerate)) {
                tabu[leave] = it + 1 + P.tabu_tenure;
                flags |= kTfTabuPush;
            }
            if (ties > 1) flags |= kTfTieSet;
            if (s.trace_q && it < P.trace_cap) {
                s.trace_q[(size_t)lp * P.trace_cap + it] = q;
                s.trace_r[(size_t)lp * P.trace_cap + it] = r;
            }
            S.z = __dadd_rn(S.z, __dmul_rn(dq, theta));
            pos[leave] = -1;
            basis[r] = (int16_t)q;
            pos[q] = (int16_t)r;
            if (ent >= 0) rslot[ent] = -1;
            if (src >= 0) { srow[te] = (int16_t)srcrow; rslot[srcrow] = (int16_t)te; }
            if (join >= 0) { srow[J] = (int16_t)join; rslot[join] = (int16_t)J; }
            S.k = kn;
            S.it = it + 1;
            S.degen_run = degenerate ? S.degen_run + 1 : 0;
            if (S.bland && !degenerate) S.bland = 0;
            if (!S.bland && P.bland_after > 0 && S.degen_run >= P.bland_after) S.bland = 1;
            S.flags = 0;
            R.lcount = 0;
        }
        if (tid < 32) R.gmax[tid] = INT_MIN;
        // ---- Step 8: own rows of bbar and of the live columns
#pragma unroll
        for (int v = 0; v < VR; ++v) {
            const int i = row_of(v);
            if (i >= m) continue;
            const double na = -al[v];
            if (!half) bbar[i] = i == r ? theta : __dsub_rn(bbar[i], __dmul_rn(al[v], theta));
            const double moved = src >= 0 ? col(src)[i] : 0.0;  // goes to slot te
            auto next = [&](int t, double o) {
                const double old = t == J ? 0.0 : (t == te && src >= 0 ? moved : o);
                col(t)[i] = i == r ? rho[t] : fma(na, rho[t], old);
            };
            // Four loads ahead of their stores: one by one each waits for the store before it,
            // which may alias it for all the compiler knows (1024 LPs of m 128..256, k = m:
            // 87 -> 78 ms; eight loads spill, 81).
            constexpr int st = kPair ? 2 : 1;
            int t = half;
            for (; t + 3 * st < kn; t += 4 * st) {
                double o[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) o[u] = col(t + u * st)[i];
#pragma unroll
                for (int u = 0; u < 4; ++u) next(t + u * st, o[u]);
            }
            for (; t < kn; t += st) next(t, col(t)[i]);
        }
        __syncthreads();
        // ---- periodic reinversion (structure-aware, as in the single-LP solver)
        if (P.reinvert_every > 0 && (it + 1) % P.reinvert_every == 0) {
            if (tid == 0) {
                int kp = 0, kr = 0;
                for (int p = 0; p < m; ++p)
                    if (basis[p] < n) lstP[kp++] = (int16_t)p;
                for (int i = 0; i < m; ++i)
                    if (rslot[i] >= 0) lstR[kr++] = (int16_t)i;
                if (kp != kn || kr != kn) S.err = 1;
            }
            __syncthreads();
            const int kk = kn;
            if (S.err) { if (tid == 0) S.status = -1; __syncthreads(); break; }
            for (int e = tid; e < kk * kk; e += T) {
                const int t = e / kk, a = e - t * kk;
                Wm[e] = __ldg(A + (size_t)lstR[a] * n + basis[lstP[t]]);
            }
            for (int a = tid; a < kk; a += T) { pinv[a] = 0; pivrow[a] = -1; }  // pinv doubles as "row used"
            __syncthreads();
            for (int j = 0; j < kk; ++j) {
                long long pk = LLONG_MIN;
                int p = -1;
                for (int a = tid; a < kk; a += T)
                    if (!pinv[a]) {
                        const long long v = dkey(fabs(Wm[(size_t)j * kk + a]));
                        if (beats(v, a, pk, p)) { pk = v; p = a; }
                    }
                block_best<T>(pk, p, R, pk, p);
                if (p < 0 || !(pk > 0)) {
                    if (tid == 0) S.err = 2;
                    __syncthreads();
                    break;
                }
                for (int a = tid; a < kk; a += T) rho[a] = Wm[(size_t)j * kk + a];  // pivot column f
                __syncthreads();
                const double pv = rho[p];
                for (int t = tid; t < kk; t += T) aq[t] = Wm[(size_t)t * kk + p] / pv;  // g_t (row p / pivot)
                if (tid == 0) { pivrow[j] = (int16_t)p; pinv[p] = 1; }
                __syncthreads();
                for (int e = tid; e < kk * kk; e += T) {
                    const int t = e / kk, a = e - t * kk;
                    if (t == j) Wm[e] = (a == p) ? 1.0 / pv : -rho[a] / pv;
                    else Wm[e] = (a == p) ? aq[t] : fma(-rho[a], aq[t], Wm[e]);
                }
                __syncthreads();
            }
            if (S.err) { if (tid == 0) S.status = -1; __syncthreads(); break; }
            for (int t = tid; t < kk; t += T) {
                pinv[pivrow[t]] = (int16_t)t;
                srow[t] = lstR[t];
                rslot[lstR[t]] = (int16_t)t;
            }
            __syncthreads();
            // B11^-1[bb][a] = Wm[pinv[a]*kk + pivrow[bb]]
            for (int e = tid; e < kk * kk; e += T) {
                const int bb = e / kk, a = e - bb * kk;
                col(a)[lstP[bb]] = Wm[(size_t)pinv[a] * kk + pivrow[bb]];
            }
            // slack positions: B^-1[p, R[a]] = -sum_b A[s, J[b]] B11^-1[b][a]
            for (int e = tid; e < m * kk; e += T) {
                const int p = e / (kk > 0 ? kk : 1), a = e - p * kk;
                if (kk == 0 || basis[p] < n) continue;
                const int sr = basis[p] - n;
                double acc = 0.0;
                for (int bb = 0; bb < kk; ++bb)
                    acc = fma(__ldg(A + (size_t)sr * n + basis[lstP[bb]]), Wm[(size_t)pinv[a] * kk + pivrow[bb]], acc);
                col(a)[p] = -acc;
            }
            __syncthreads();
            for (int p = tid; p < m; p += T) {
                double acc = basis[p] >= n ? b[basis[p] - n] : 0.0;
                for (int t = 0; t < kk; ++t) acc = fma(col(t)[p], b[srow[t]], acc);
                bbar[p] = acc;
            }
            for (int t = tid; t < kk; t += T) {
                double acc = 0.0;
                for (int bb = 0; bb < kk; ++bb) acc = fma(c[basis[lstP[bb]]], col(t)[lstP[bb]], acc);
                y[t] = acc;
                y32[t] = (float)acc;
            }
            __syncthreads();
            if (warp == 0) {
                double zz = 0.0;
                for (int bb = lane; bb < kk; bb += 32) zz = fma(c[basis[lstP[bb]]], bbar[lstP[bb]], zz);
                zz = warp_sum(zz);
                if (lane == 0) S.z = zz;
            }
            __syncthreads();
        }
    }
    // ---- outputs
    double* xo = s.x + L.c_off;
    double* yo = s.y + L.r_off;
    for (int j = tid; j < n; j += T) xo[j] = pos[j] >= 0 ? bbar[pos[j]] : 0.0;
    for (int i = tid; i < m; i += T) yo[i] = rslot[i] >= 0 ? y[rslot[i]] : 0.0;
    if (tid == 0) {
        s.status[lp] = S.status;
        s.iters[lp] = S.it;
        s.obj[lp] = S.z;
    }
    __syncthreads();
}

template <int T, bool kPair>
__global__ void __launch_bounds__(T, 1024 / T) k_batch(BatchState s, int bucket, int begin, int count, int mmax, int nmax,
                                                       int ks) {
    extern __shared__ __align__(16) unsigned char smem[];
    double* slot = s.scratch[bucket] + (size_t)blockIdx.x * s.slot_doubles[bucket];
    __shared__ int next;
    for (;;) {
        if (threadIdx.x == 0) next = atomicAdd(s.queue + bucket, 1);
        __syncthreads();
        const int k = next;
        __syncthreads();
        if (k >= count) break;
        solve_one<T, kPair>(s, s.order[begin + k], smem, slot, mmax, nmax, ks);
    }
}

}  // namespace

// ks live columns in shared memory beside the vectors
size_t batch_smem_bytes(int mmax, int nmax, int ks) {
    const size_t d = (size_t)ks * mmax + 5 * (size_t)mmax;
    const size_t f = (size_t)mmax + nmax;
    const size_t i = (size_t)nmax + mmax;
    const size_t h = 7 * (size_t)mmax + nmax + mmax;
    return d * 8 + f * 4 + i * 4 + h * 2;
}

using BatchKernel = void (*)(BatchState, int, int, int, int, int, int);

// m: the largest of the launch
BatchKernel batch_kernel(int threads, int m) {
    const bool pair = 2 * m <= threads;
    switch (threads) {
        case 128: return pair ? k_batch<128, true> : k_batch<128, false>;
        case 256: return pair ? k_batch<256, true> : k_batch<256, false>;
        default: return pair ? k_batch<512, true> : k_batch<512, false>;
    }
}

}  // namespace lpgb

using namespace lpgb;

// ---------------------------------------------------------------- host side
struct lp_batch {
    int device = 0;
    int count = 0;
    lp_options opt{};
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int sms = 0;
    size_t smem_optin = 0;
    std::vector<void*> allocs;
    std::vector<BatchLP> lps;
    std::vector<int32_t> order;
    int bucket_begin[kBuckets + 1] = {};
    int bucket_m[kBuckets] = {}, bucket_n[kBuckets] = {};  // the largest m and n in each bucket
    // 4096 LPs of m 16..256: 3.31 ms (3.35 with 256 threads throughout, 4.05 with 128, 5.2
    // with 512; shared-memory columns 3.43); m 16..64 alone 0.44 ms (0.65 with 256).
    // These are for k far below m.  Rows that all become live want more threads (1024 LPs
    // of m 65..128 11.6 ms with 128, 7.7 with 256, 8.8 with 512; 512 of m 193..256 119, 74,
    // 51): lp_batch_tune finds them on the batch itself.
    int cfg_threads[kBuckets] = {128, 128, 256, 256};
    int cfg_smem[kBuckets] = {0, 0, 0, 0};
    int64_t sum_m = 0, sum_n = 0;
    BatchState st{};
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    // the buckets run side by side on their own streams, forked from and
    // joined back into `stream`; the whole solve is one captured CUDA graph
    cudaStream_t bstream[kBuckets] = {};
    cudaEvent_t fork = nullptr, join[kBuckets] = {};
    cudaGraphExec_t graph = nullptr;
    bool solved = false;
    double fp64_flops_per_iter_avg = 0.0;
};

namespace {

int bfail(cudaError_t e) { return e == cudaErrorMemoryAllocation ? LP_ERR_OOM : LP_ERR_CUDA; }

#define BCK(x)                                     \
    do {                                           \
        cudaError_t e_ = (x);                      \
        if (e_ != cudaSuccess) return bfail(e_);   \
    } while (0)

template <typename T>
int balloc(lp_batch* h, T** p, size_t count) {
    void* v = nullptr;
    cudaError_t e = cudaMalloc(&v, std::max<size_t>(count, 1) * sizeof(T));
    if (e != cudaSuccess) return bfail(e);
    h->allocs.push_back(v);
    *p = static_cast<T*>(v);
    return LP_OK;
}

void bfree(lp_batch* h) {
    for (void* p : h->allocs) cudaFree(p);
    h->allocs.clear();
    if (h->e0) cudaEventDestroy(h->e0);
    if (h->e1) cudaEventDestroy(h->e1);
    if (h->graph) cudaGraphExecDestroy(h->graph);
    if (h->fork) cudaEventDestroy(h->fork);
    for (int bk = 0; bk < kBuckets; ++bk) {
        if (h->join[bk]) cudaEventDestroy(h->join[bk]);
        if (h->bstream[bk]) cudaStreamDestroy(h->bstream[bk]);
    }
    if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
}

bool cfg_valid(const lp_batch* h, int bucket, int threads, int smem) {
    if (threads != 128 && threads != 256 && threads != 512) return false;
    // (the flag stays tied to sizes whose whole inverse would fit)
    const size_t need = batch_smem_bytes(kBucketM[bucket], kBatchMaxN, smem ? kBucketM[bucket] : 0);
    return need <= h->smem_optin;
}

int grid_for(const lp_batch* h, int bucket, int* grid, size_t* smem) {
    const int T = h->cfg_threads[bucket];
    const bool sm = h->cfg_smem[bucket] != 0;
    *smem = batch_smem_bytes(h->bucket_m[bucket], h->bucket_n[bucket], sm ? kSmemCols : 0);
    BatchKernel k = batch_kernel(T, h->bucket_m[bucket]);
    // (one limit for every bucket: buckets with the same thread count share a kernel)
    BCK(cudaFuncSetAttribute(reinterpret_cast<const void*>(k), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)batch_smem_bytes(kBatchMaxM, kBatchMaxN, kSmemCols)));
    int occ = 0;
    BCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, T, *smem));
    *grid = h->sms * std::max(1, occ);
    return LP_OK;
}

struct BucketLaunch {
    int grid = 0;
    size_t smem = 0;
};

// Grid and shared memory of every non-empty bucket in [b0, b1).
int plan_buckets(lp_batch* h, int b0, int b1, BucketLaunch* out) {
    for (int bk = b0; bk < b1; ++bk) {
        const int cnt = h->bucket_begin[bk + 1] - h->bucket_begin[bk];
        out[bk] = BucketLaunch{};
        if (cnt == 0) continue;
        int rc = grid_for(h, bk, &out[bk].grid, &out[bk].smem);
        if (rc != LP_OK) return rc;
        out[bk].grid = std::min(std::min(out[bk].grid, h->sms * kSlotsPerSm), cnt);
    }
    return LP_OK;
}

// Launch the buckets in [b0, b1), largest first: one after another on
// `stream`, or (concurrent) each on its own stream between a fork and a join,
// so that a bucket's tail overlaps the next bucket.  Every bucket has its own
// scratch slots, so concurrent buckets never share one.
int launch_buckets(lp_batch* h, int b0, int b1, const BucketLaunch* plan, bool concurrent) {
    BCK(cudaMemsetAsync(h->st.queue, 0, sizeof(int32_t) * kBuckets, h->stream));
    if (concurrent) BCK(cudaEventRecord(h->fork, h->stream));
    for (int bk = b1 - 1; bk >= b0; --bk) {
        const int begin = h->bucket_begin[bk], cnt = h->bucket_begin[bk + 1] - begin;
        if (cnt == 0 || plan[bk].grid == 0) continue;
        cudaStream_t st = h->stream;
        if (concurrent) {
            st = h->bstream[bk];
            BCK(cudaStreamWaitEvent(st, h->fork, 0));
        }
        BatchKernel k = batch_kernel(h->cfg_threads[bk], h->bucket_m[bk]);
        k<<<plan[bk].grid, h->cfg_threads[bk], plan[bk].smem, st>>>(h->st, bk, begin, cnt, h->bucket_m[bk], h->bucket_n[bk],
                                                                    h->cfg_smem[bk] ? kSmemCols : 0);
        BCK(cudaGetLastError());
        if (concurrent) {
            BCK(cudaEventRecord(h->join[bk], st));
            BCK(cudaStreamWaitEvent(h->stream, h->join[bk], 0));
        }
    }
    return LP_OK;
}

// (Re)capture the whole solve as one graph after a change of the tuning.
int capture_batch_graph(lp_batch* h) {
    if (h->graph) {
        cudaGraphExecDestroy(h->graph);
        h->graph = nullptr;
    }
    BucketLaunch plan[kBuckets];
    int rc = plan_buckets(h, 0, kBuckets, plan);
    if (rc != LP_OK) return rc;
    cudaGraph_t g = nullptr;
    BCK(cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
    rc = launch_buckets(h, 0, kBuckets, plan, true);
    cudaError_t e = cudaStreamEndCapture(h->stream, &g);
    if (rc != LP_OK) {
        if (g) cudaGraphDestroy(g);
        return rc;
    }
    BCK(e);
    e = cudaGraphInstantiate(&h->graph, g, 0);
    cudaGraphDestroy(g);
    BCK(e);
    return LP_OK;
}

}  // namespace

extern "C" {

int lp_batch_create(lp_batch** out, int32_t count, const int32_t* m, const int32_t* n, const double* A,
                    const double* b, const double* c, int32_t on_device, const lp_options* opt) {
    if (!out) return LP_ERR_INVALID_ARG;
    *out = nullptr;
    if (count < 1 || !m || !n || !A || !b || !c) return LP_ERR_INVALID_ARG;
    lp_options o;
    lp_default_options(&o);
    o.price_mode = 1;
    o.topk = kBatchTopk;
    if (opt) o = *opt;
    if (o.price_mode < 0 || o.price_mode > 1 || o.topk < 1 || o.max_iters < 0 || o.reinvert_every < 0 ||
        o.tabu_tenure < 0 || o.bland_after < 0 || o.trace_cap < 0)
        return LP_ERR_INVALID_ARG;
    lp_batch* h = new (std::nothrow) lp_batch();
    if (!h) return LP_ERR_OOM;
    h->opt = o;
    h->count = count;
    int rc = LP_OK;
    auto fail = [&](int code) {
        bfree(h);
        delete h;
        return code;
    };
    h->lps.resize(count);
    int64_t aoff = 0, roff = 0, coff = 0;
    for (int k = 0; k < count; ++k) {
        if (m[k] < 1 || m[k] > kBatchMaxM || n[k] < 1 || n[k] > kBatchMaxN) return fail(LP_ERR_INVALID_ARG);
        h->lps[k] = {m[k], n[k], aoff, (int32_t)roff, (int32_t)coff};
        aoff += (int64_t)m[k] * n[k];
        roff += m[k];
        coff += n[k];
        if (roff > INT32_MAX || coff > INT32_MAX) return fail(LP_ERR_INVALID_ARG);
    }
    h->sum_m = roff;
    h->sum_n = coff;
    if (cudaGetDevice(&h->device) != cudaSuccess) return fail(LP_ERR_CUDA);
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, h->device) != cudaSuccess) return fail(LP_ERR_CUDA);
    h->sms = prop.multiProcessorCount;
    h->smem_optin = prop.sharedMemPerBlockOptin;
    if (o.cuda_stream) {
        h->stream = static_cast<cudaStream_t>(o.cuda_stream);
    } else {
        if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) return fail(LP_ERR_CUDA);
        h->own_stream = true;
    }
    if (cudaEventCreate(&h->e0) != cudaSuccess || cudaEventCreate(&h->e1) != cudaSuccess) return fail(LP_ERR_CUDA);
    if (cudaEventCreateWithFlags(&h->fork, cudaEventDisableTiming) != cudaSuccess) return fail(LP_ERR_CUDA);
    for (int bk = 0; bk < kBuckets; ++bk)
        if (cudaStreamCreateWithFlags(&h->bstream[bk], cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&h->join[bk], cudaEventDisableTiming) != cudaSuccess)
            return fail(LP_ERR_CUDA);
    // host-side validation of host inputs
    if (!on_device) {
        for (int64_t e = 0; e < aoff; ++e)
            if (!std::isfinite(A[e])) return fail(LP_ERR_INVALID_ARG);
        for (int64_t e = 0; e < roff; ++e)
            if (!std::isfinite(b[e]) || b[e] < 0) return fail(LP_ERR_INVALID_ARG);
        for (int64_t e = 0; e < coff; ++e)
            if (!std::isfinite(c[e])) return fail(LP_ERR_INVALID_ARG);
    }
    // buckets by m, largest work first inside a bucket
    std::vector<int> idx(count);
    for (int k = 0; k < count; ++k) idx[k] = k;
    auto bucket_of = [&](int k) {
        for (int bk = 0; bk < kBuckets; ++bk)
            if (h->lps[k].m <= kBucketM[bk]) return bk;
        return kBuckets - 1;
    };
    std::stable_sort(idx.begin(), idx.end(), [&](int a, int bb) {
        const int ba = bucket_of(a), bb2 = bucket_of(bb);
        if (ba != bb2) return ba < bb2;
        const int64_t wa = (int64_t)h->lps[a].m * (h->lps[a].m + h->lps[a].n);
        const int64_t wb = (int64_t)h->lps[bb].m * (h->lps[bb].m + h->lps[bb].n);
        return wa > wb;
    });
    h->order = idx;
    {
        int k = 0;
        for (int bk = 0; bk < kBuckets; ++bk) {
            h->bucket_begin[bk] = k;
            while (k < count && bucket_of(idx[k]) == bk) {
                h->bucket_m[bk] = std::max(h->bucket_m[bk], h->lps[idx[k]].m);
                h->bucket_n[bk] = std::max(h->bucket_n[bk], h->lps[idx[k]].n);
                ++k;
            }
        }
        h->bucket_begin[kBuckets] = count;
    }
    for (int bk = 0; bk < kBuckets; ++bk)
        if (!cfg_valid(h, bk, h->cfg_threads[bk], h->cfg_smem[bk])) h->cfg_smem[bk] = 0;
    // device buffers
    BatchState& S = h->st;
    S.p = {o.reinvert_every, o.tabu_tenure, o.max_iters, o.bland_after, o.price_mode, o.topk, o.trace_cap,
           o.tol_d, o.tol_piv, o.tol_tie};
    BatchLP* dl;
    int32_t *dord, *dst, *dit, *dq;
    double *dA, *db, *dc, *dob, *dx, *dy, *dscr;
    if ((rc = balloc(h, &dl, count)) || (rc = balloc(h, &dord, count)) || (rc = balloc(h, &dst, count)) ||
        (rc = balloc(h, &dit, count)) || (rc = balloc(h, &dq, kBuckets)) || (rc = balloc(h, &dA, aoff)) ||
        (rc = balloc(h, &db, roff)) || (rc = balloc(h, &dc, coff)) || (rc = balloc(h, &dob, count)) ||
        (rc = balloc(h, &dx, coff)) || (rc = balloc(h, &dy, roff)))
        return fail(rc);
    // per-CTA slots of each non-empty bucket: B^-1 (global residency) + reinversion block
    for (int bk = 0; bk < kBuckets; ++bk) {
        S.slot_doubles[bk] = 2 * (int64_t)kBucketM[bk] * kBucketM[bk];
        S.scratch[bk] = nullptr;
        if (h->bucket_begin[bk + 1] == h->bucket_begin[bk]) continue;
        if ((rc = balloc(h, &dscr, (size_t)S.slot_doubles[bk] * h->sms * kSlotsPerSm))) return fail(rc);
        S.scratch[bk] = dscr;
    }
    S.lps = dl; S.order = dord; S.status = dst; S.iters = dit; S.queue = dq;
    S.A = dA; S.b = db; S.c = dc; S.obj = dob; S.x = dx; S.y = dy;
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
    if (cudaMemcpyAsync(dl, h->lps.data(), sizeof(BatchLP) * count, cudaMemcpyHostToDevice, h->stream) ||
        cudaMemcpyAsync(dord, idx.data(), sizeof(int32_t) * count, cudaMemcpyHostToDevice, h->stream) ||
        cudaMemcpyAsync(dA, A, sizeof(double) * aoff, kind, h->stream) ||
        cudaMemcpyAsync(db, b, sizeof(double) * roff, kind, h->stream) ||
        cudaMemcpyAsync(dc, c, sizeof(double) * coff, kind, h->stream))
        return fail(LP_ERR_CUDA);
    if (o.price_mode == 1) {
        uint16_t* lp16;
        if ((rc = balloc(h, &lp16, aoff))) return fail(rc);
        launch_to_bf16(dA, lp16, (size_t)aoff, h->stream);
        S.A_lp = lp16;
    }
    if (o.trace_cap > 0) {
        int32_t *tq, *tr;
        if ((rc = balloc(h, &tq, (size_t)count * o.trace_cap)) || (rc = balloc(h, &tr, (size_t)count * o.trace_cap)))
            return fail(rc);
        S.trace_q = tq;
        S.trace_r = tr;
    }
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) return fail(LP_ERR_CUDA);
    if (on_device) {
        // device inputs: validate with the same rules on a host copy of b (small)
        std::vector<double> hb(roff);
        if (cudaMemcpy(hb.data(), db, sizeof(double) * roff, cudaMemcpyDeviceToHost)) return fail(LP_ERR_CUDA);
        for (double v : hb)
            if (!std::isfinite(v) || v < 0) return fail(LP_ERR_INVALID_ARG);
    }
    *out = h;
    return LP_OK;
}

int lp_batch_solve(lp_batch* h, lp_batch_result* res) {
    if (!h) return LP_ERR_INVALID_ARG;
    if (!h->graph) {
        int rc = capture_batch_graph(h);
        if (rc != LP_OK) return rc;
    }
    BCK(cudaEventRecord(h->e0, h->stream));
    BCK(cudaGraphLaunch(h->graph, h->stream));
    BCK(cudaEventRecord(h->e1, h->stream));
    BCK(cudaEventSynchronize(h->e1));
    h->solved = true;
    if (res) {
        std::vector<int32_t> st(h->count), it(h->count);
        BCK(cudaMemcpy(st.data(), h->st.status, sizeof(int32_t) * h->count, cudaMemcpyDeviceToHost));
        BCK(cudaMemcpy(it.data(), h->st.iters, sizeof(int32_t) * h->count, cudaMemcpyDeviceToHost));
        memset(res, 0, sizeof(*res));
        double fl = 0.0;
        for (int k = 0; k < h->count; ++k) {
            if (st[k] == kOptimal) res->solved++;
            else if (st[k] == kUnbounded) res->unbounded++;
            else if (st[k] == kIterLimit) res->iter_limit++;
            else res->failed++;
            res->iterations += it[k];
            const double mm = h->lps[k].m;
            // FP64 work per pivot: FTRAN + update (2 m^2 FMA) + top-k re-price (k m FMA) or full PRICE (m n FMA)
            const double price = h->opt.price_mode == 1 ? (double)h->opt.topk * mm : mm * h->lps[k].n;
            fl += it[k] * 2.0 * (2.0 * mm * mm + price);
        }
        float ms = 0.f;
        BCK(cudaEventElapsedTime(&ms, h->e0, h->e1));
        res->seconds = ms * 1e-3;
        res->fp64_flops = fl;
    }
    return LP_OK;
}

int lp_batch_get(const lp_batch* h, int32_t* status, int32_t* iterations, double* objective, double* x,
                 double* y) {
    if (!h) return LP_ERR_INVALID_ARG;
    if (!h->solved) return LP_ERR_STATE;
    if (status) BCK(cudaMemcpy(status, h->st.status, sizeof(int32_t) * h->count, cudaMemcpyDeviceToHost));
    if (iterations) BCK(cudaMemcpy(iterations, h->st.iters, sizeof(int32_t) * h->count, cudaMemcpyDeviceToHost));
    if (objective) BCK(cudaMemcpy(objective, h->st.obj, sizeof(double) * h->count, cudaMemcpyDeviceToHost));
    if (x) BCK(cudaMemcpy(x, h->st.x, sizeof(double) * h->sum_n, cudaMemcpyDeviceToHost));
    if (y) BCK(cudaMemcpy(y, h->st.y, sizeof(double) * h->sum_m, cudaMemcpyDeviceToHost));
    return LP_OK;
}

int lp_batch_get_trace(const lp_batch* h, int32_t k, int32_t* q, int32_t* r, int32_t cap, int32_t* count) {
    if (!h || k < 0 || k >= h->count || cap < 0) return LP_ERR_INVALID_ARG;
    if (!h->solved || h->opt.trace_cap <= 0) return LP_ERR_STATE;
    int32_t it = 0;
    BCK(cudaMemcpy(&it, h->st.iters + k, sizeof(int32_t), cudaMemcpyDeviceToHost));
    const int n = std::min(std::min(it, h->opt.trace_cap), cap);
    if (count) *count = n;
    if (n > 0 && q) BCK(cudaMemcpy(q, h->st.trace_q + (size_t)k * h->opt.trace_cap, sizeof(int32_t) * n, cudaMemcpyDeviceToHost));
    if (n > 0 && r) BCK(cudaMemcpy(r, h->st.trace_r + (size_t)k * h->opt.trace_cap, sizeof(int32_t) * n, cudaMemcpyDeviceToHost));
    return LP_OK;
}

int lp_batch_set_tuning(lp_batch* h, const int32_t* table) {
    if (!h || !table) return LP_ERR_INVALID_ARG;
    for (int bk = 0; bk < kBuckets; ++bk)
        if (!cfg_valid(h, bk, table[2 * bk], table[2 * bk + 1])) return LP_ERR_INVALID_ARG;
    for (int bk = 0; bk < kBuckets; ++bk) {
        h->cfg_threads[bk] = table[2 * bk];
        h->cfg_smem[bk] = table[2 * bk + 1];
    }
    if (h->graph) {
        cudaGraphExecDestroy(h->graph);
        h->graph = nullptr;
    }
    return LP_OK;
}

int lp_batch_tune(lp_batch* h, int32_t* table, int32_t trials) {
    if (!h || trials < 1) return LP_ERR_INVALID_ARG;
    if (h->graph) {
        cudaGraphExecDestroy(h->graph);
        h->graph = nullptr;
    }
    const int threads[3] = {128, 256, 512};
    for (int bk = 0; bk < kBuckets; ++bk) {
        if (h->bucket_begin[bk + 1] == h->bucket_begin[bk]) continue;
        float best = 1e30f;
        int bt = h->cfg_threads[bk], bs = h->cfg_smem[bk];
        for (int sm = 1; sm >= 0; --sm) {
            for (int t : threads) {
                if (!cfg_valid(h, bk, t, sm)) continue;
                h->cfg_threads[bk] = t;
                h->cfg_smem[bk] = sm;
                float tot = 0.f;
                BucketLaunch plan[kBuckets];
                int rc = plan_buckets(h, bk, bk + 1, plan);
                if (rc != LP_OK) return rc;
                for (int r = 0; r < trials; ++r) {
                    BCK(cudaEventRecord(h->e0, h->stream));
                    rc = launch_buckets(h, bk, bk + 1, plan, false);
                    if (rc != LP_OK) return rc;
                    BCK(cudaEventRecord(h->e1, h->stream));
                    BCK(cudaEventSynchronize(h->e1));
                    float ms = 0.f;
                    BCK(cudaEventElapsedTime(&ms, h->e0, h->e1));
                    tot += ms;
                }
                if (tot < best) { best = tot; bt = t; bs = sm; }
            }
        }
        h->cfg_threads[bk] = bt;
        h->cfg_smem[bk] = bs;
    }
    if (table)
        for (int bk = 0; bk < kBuckets; ++bk) { table[2 * bk] = h->cfg_threads[bk]; table[2 * bk + 1] = h->cfg_smem[bk]; }
    return LP_OK;
}

void lp_batch_destroy(lp_batch* h) {
    if (!h) return;
    if (h->stream) cudaStreamSynchronize(h->stream);
    bfree(h);
    delete h;
}

}  // extern "C"
