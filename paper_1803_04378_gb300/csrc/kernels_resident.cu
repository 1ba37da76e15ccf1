// kernels_resident.cu -- the persistent pivot kernel of the slack-structured
// engine with its working set in shared memory (k_iterate_r).
//
// The method, the slot layout and the arithmetic are those of k_iterate_s
// (kernels_struct.cu): PRICE over the k live rows, FTRAN and the rank-1 update
// over the k live columns of B^-1, slot moves, the same order of every sum --
// so the pivots, B^-1, bbar and y are bit-identical to it (-0 and 0 as one value).
// What differs is where the operands live and how the CTAs meet.
//
// Residence.  CTA b owns the columns j = b, b + G, ... of A and the rows
// i = b, b + G, ... of B^-1.  Their live parts stay in shared memory for the
// whole launch (kA: the FP32 copy of A that the screen reads, kB: the rows of
// B^-1), next to y, rho, the entering column, the slot maps and the CTA's
// slices of bbar, alpha, the basis and the tabu list; the rows of B^-1 are
// written through to memory, where the other CTAs read the pivot row and the
// reinversion reads the whole.  At 4096 x 8192, G = 152 and k = 344 that is
// 74 KB of A and 74 KB of B^-1 per CTA.
//
// Meeting.  The two grid barriers of a pivot carry the CTAs' records: each goes into
// every CTA's mailbox, its 16-byte chunks stamped with the sequence number of the
// meeting, and thread c polls its own CTA's mailbox for CTA c's.  Reading every
// CTA's record is the barrier, so a meeting costs one store and one load round
// trip instead of an atomic, a poll and the records' own loads.
//
// Order.  The ratio test's meeting publishes what the other CTAs read in the next step:
// the rows of B^-1, the moved slots of A_p, the tabu list.  The warp that sends its
// record has fenced first, after a block barrier behind those writes: a fence, then
// a store of the same thread, is a release for all that the CTA wrote before the
// barrier, and the polls acquire.  The fence runs beside FTRAN.  (A release in
// each of the record's stores costs 0.9 to 1.3 us a pivot, a fence in every polling
// warp 0 to 0.5, this 0 to 0.18.)  So do the repair's meeting and those without a record.
// The PRICE meeting publishes nothing.  After it the pivot row's owner overwrites the
// row, which every CTA has read: each sends its record on a condition over all of the
// row's values (the range of the new y), so a read that returned the later ones would
// be the cause of itself.
//
// PRICE decides on intervals.  The FP32 screen gives every column an interval
// that holds its reduced cost.  The record of a CTA is its largest lower end
// and the (at most four) columns whose upper end reaches it.  When only one
// column of all CTAs reaches the largest lower end it is Dantzig's choice, and
// its exact d_q is formed from the entering column that FTRAN stages anyway;
// several are re-priced in FP64 by every CTA alike.  Under the Bland safety net
// a record holds the smallest column that surely improves and the smaller ones
// that may.  Where the screen proves no improving column (the optimum, a tabu
// list that covers every improving one), steps aside or overflows, all own
// columns are priced in FP64 and the CTAs meet once more.
//
// The rank-1 update (warps kRPrice .., then the pricing warps that do not poll)
// runs under PRICE and its meeting, since only FTRAN needs it.
//
// What bounds it: latency.  A pivot is a chain of two meetings, two L2
// round trips (pivot row, entering column; 0.6 us each), seven block barriers and
// the reductions between them; of 17.2 us at 4096 x 8192 the FP64 pipe needs 2.6 us for
// FTRAN, and 2.5 us for the update that PRICE hides.  Against k_iterate_s, whose
// operands stay in L2 and whose 1024-thread CTAs meet through atomics: 30.1 -> 17.2 us
// per pivot at 4096 x 8192, 19.8 -> 9.0 at 701 x 1203, 20.6 -> 9.0 at 200 x 300,
// 24.3 -> 9.05 on a degenerate 256 x 512 under the safety net.
#include "lpgb_internal.cuh"
#include "struct_common.cuh"
#include "../../include/lpgb.h"

#include <algorithm>
#include <cfloat>
#include <cmath>

namespace lpgb {

namespace {

constexpr int kRThreads = 512;
constexpr int kRWarps = kRThreads / 32;
constexpr int kRPrice = 8;        // warps that screen and poll; the others apply the rank-1 update
constexpr int kRMail = kRWarps - 1;  // the warp that fences for the CTA and sends what publishes its data
constexpr int kRMaxCtas = 32 * (kRPrice - 1);  // a pricing warp that does not poll moves the slots of A
constexpr int kRChunks = 4;       // 16-byte chunks of a record: three payload words and the stamp
constexpr int kRWords = 3 * kRChunks;
constexpr unsigned kRMore = 1u << 31;  // PRICE record: more than one column listed
constexpr int kRList = 4;         // columns listed in a PRICE record
constexpr int kRWarpList = 16;    // columns kept per polling warp
constexpr int kRCand = 16;        // columns re-priced by every CTA
// Meetings of one step at most: the PRICE records, the FP64 pricing's where they decide
// nothing, the ratio test's records, and the two of a scanned tie set (a step that
// stops or repairs holds one).  A launch holds one more, at its start.  The next
// launch's numbers begin past all that this one can use: a number already stamped in
// a mailbox would be taken for an answer without waiting.
constexpr unsigned kRStepMeetings = 5;

// ---- the meeting of all CTAs ---------------------------------------------------------
__device__ __forceinline__ void st_relaxed_b128(ulonglong2* p, unsigned long long lo, unsigned long long hi) {
    asm volatile("{\n .reg .b128 t;\n mov.b128 t, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], t;\n}\n"
                 ::"l"(p), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ ulonglong2 ld_acquire_b128(const ulonglong2* p) {
    ulonglong2 v;
    asm volatile("{\n .reg .b128 t;\n ld.acquire.gpu.global.b128 t, [%2];\n mov.b128 {%0, %1}, t;\n}\n"
                 : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}

// One chunk of the CTA's record under `seq`, into CTA dest's mailbox.  Every CTA has a
// mailbox of its own, which no other polls, a sender's 16 bytes beside the next
// sender's: a warp polls 32 senders in four lines.  One record for all, 64 bytes apart
// and polled by every CTA, held up its writer (17.9 us a pivot against 17.0 then at
// 4096 x 8192 on 152 CTAs, 10.6 against 9.5 at 1024 x 2048); chunks of several CTAs in
// one line that all poll took 2.3 us a meeting.
__device__ __forceinline__ void meet_put(ulonglong2* buf, unsigned seq, int dest, int chunk, unsigned a, unsigned b,
                                         unsigned c) {
    st_relaxed_b128(buf + (((size_t)(seq & 1) * gridDim.x + dest) * kRChunks + chunk) * gridDim.x + blockIdx.x,
                    ((unsigned long long)b << 32) | a, ((unsigned long long)seq << 32) | c);
}

// Chunks C0 .. C1 - 1 of CTA c's record under `seq` into w (bounded wait; *fail
// on giving up).  A slot is written again two meetings later, which no CTA
// reaches before every CTA has read it.
template <int C0, int C1>
__device__ __forceinline__ void meet_get(const ulonglong2* buf, unsigned seq, int c, unsigned* w, volatile int* fail) {
    const ulonglong2* p = buf + ((size_t)(seq & 1) * gridDim.x + blockIdx.x) * kRChunks * gridDim.x + c;
    unsigned spins = 0;
    for (;;) {
        ulonglong2 v[C1 - C0];
        bool ok = true;
#pragma unroll
        for (int e = C0; e < C1; ++e) v[e - C0] = ld_acquire_b128(p + (size_t)e * gridDim.x);
#pragma unroll
        for (int e = C0; e < C1; ++e) {
            ok &= (unsigned)(v[e - C0].y >> 32) == seq;
            w[3 * e] = (unsigned)v[e - C0].x;
            w[3 * e + 1] = (unsigned)(v[e - C0].x >> 32);
            w[3 * e + 2] = (unsigned)v[e - C0].y;
        }
        if (ok) return;
        if (++spins > kBarrierSpins) {
            *fail = 1;
            return;
        }
    }
}

__device__ __forceinline__ long long words_ll(unsigned lo, unsigned hi) {
    return (long long)(((unsigned long long)hi << 32) | lo);
}
__device__ __forceinline__ unsigned ll_lo(long long v) { return (unsigned)v; }
__device__ __forceinline__ unsigned ll_hi(long long v) { return (unsigned)((unsigned long long)v >> 32); }

// ---- shared-memory layout ---------------------------------------------------------------
struct ResLayout {
    int kc;        // live slots held (a multiple of 64)
    int R, Cn;     // owned rows and columns per CTA, rounded up to 4
    size_t bytes;
};

__host__ __device__ inline ResLayout res_layout(int m, int n, int G, int kc, bool a, bool b) {
    ResLayout l;
    l.kc = kc;
    l.R = ((m + G - 1) / G + 3) & ~3;
    l.Cn = ((n + G - 1) / G + 3) & ~3;
    l.bytes = 8 * (size_t)(4 * kc + 3 * l.R + l.Cn) + (b ? 8 * (size_t)l.R * kc : 0) + (a ? 4 * (size_t)l.Cn * kc : 0) +
              4 * (size_t)(kc + 5 * l.Cn + l.R) + 4 * (size_t)((m + 7) & ~7);
    return l;
}

// d_j of a column given by its live rows (col, zero-padded or not: y is zero past
// the live slots) in the order of price_block: two row segments, each summed lane
// by lane and then across the warp.
template <typename Load>
__device__ __forceinline__ double exact_dot(Load col, const double2* y2, int kk, int lane) {
    const int nch = kk >> 6, mid = 32 * (nch / 2), end = 32 * nch;
    double a0 = 0.0, a1 = 0.0;
    for (int k = lane; k < mid; k += 32) {
        const double2 c = col(k), y = y2[k];
        a0 = fma(c.y, y.y, fma(c.x, y.x, a0));
    }
    for (int k = mid + lane; k < end; k += 32) {
        const double2 c = col(k), y = y2[k];
        a1 = fma(c.y, y.y, fma(c.x, y.x, a1));
    }
    const double p0 = pair_sum(a0), p1 = pair_sum(a1);
    return p0 + p1;
}

// s_c = sum y a_c and S_c = sum |y| |a_c| of four columns in FP32; lanes 8 c .. 8 c + 7
// get those of column c.  A term passes through at most 4 fused multiply-adds per
// 128 rows of its lane and five additions across the warp.
template <typename Load>
__device__ __forceinline__ void screen4(Load col, const float4* y4, int n4, int lane, float& s, float& a) {
    float v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = 0.f;
    for (int k = lane; k < n4; k += 32) {
        const float4 y = y4[k];
        const float4 w = make_float4(fabsf(y.x), fabsf(y.y), fabsf(y.z), fabsf(y.w));
        float4 u[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) u[c] = col(c, k);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            v[2 * c] = fmaf(u[c].x, y.x, v[2 * c]);
            v[2 * c + 1] = fmaf(fabsf(u[c].x), w.x, v[2 * c + 1]);
            v[2 * c] = fmaf(u[c].y, y.y, v[2 * c]);
            v[2 * c + 1] = fmaf(fabsf(u[c].y), w.y, v[2 * c + 1]);
            v[2 * c] = fmaf(u[c].z, y.z, v[2 * c]);
            v[2 * c + 1] = fmaf(fabsf(u[c].z), w.z, v[2 * c + 1]);
            v[2 * c] = fmaf(u[c].w, y.w, v[2 * c]);
            v[2 * c + 1] = fmaf(fabsf(u[c].w), w.w, v[2 * c + 1]);
        }
    }
    // transposed reduction: halves of the columns part at lanes 16 and 8 apart
    const bool h16 = lane & 16, h8 = lane & 8;
    float r[4], q[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float send = h16 ? v[i] : v[4 + i], keep = h16 ? v[4 + i] : v[i];
        r[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float send = h8 ? r[i] : r[2 + i], keep = h8 ? r[2 + i] : r[i];
        q[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        q[0] += __shfl_xor_sync(0xffffffffu, q[0], o);
        q[1] += __shfl_xor_sync(0xffffffffu, q[1], o);
    }
    s = q[0];
    a = q[1];
}

// The ratio test's tie threshold (row_record's arithmetic: max(1, |t|) by its bits).
__device__ __forceinline__ double tie_limit(double t, double tol) {
    const long long mag = __double_as_longlong(t) & 0x7fffffffffffffffLL;
    const double scale = __longlong_as_double(max(mag, __double_as_longlong(1.0)));
    return t + tol * scale;
}

// False only if the ratio of key k surely lies above the tie threshold of the
// smallest ratio (key kmin), without FP64 instructions: for tol <= 2^-39 and
// a smallest ratio t >= 2^-19 the threshold is within t (1 + 2^-20), so a tied
// ratio's upper 32 bits (20 of them mantissa) exceed t's by at most 3.
__device__ __forceinline__ bool tie_near(long long k, long long kmin, double tol) {
    const int h = (int)(k >> 32), hm = (int)(kmin >> 32);
    return h - hm <= 4 || hm < (1023 - 19) << 20 || __double_as_longlong(tol) > (long long)(1023 - 39) << 52;
}

// The CTA's ratio-test record (one warp; into w): chunk 0 the smallest ratio and the
// best row, chunk 1 its alpha and variable, marked kRMore when more than one row
// ties; then chunk 2 holds the best row's ratio and the size of the tie set.
// A lone smallest ratio with no other near it needs no threshold.
__device__ __forceinline__ void ratio_record(const Params& P, int owned, bool bland, const double* ral,
                                             const double* rb, const int* rvar, unsigned* w) {
    const int lane = threadIdx.x & 31;
    const int G = gridDim.x;
    const long long kpiv = dkey(P.tol_piv), kbig = dkey(DBL_MAX);
    if (owned <= 32) {
        const double al = lane < owned ? ral[lane] : 0.0;
        const int var = lane < owned ? rvar[lane] : INT_MAX;
        const long long kal = dkey(al);
        const bool ok = lane < owned && kal > kpiv;
        const double th = ok ? rb[lane] / al : DBL_MAX;
        const long long kth = dkey(th), kmin = warp_min_key(kth);
        const unsigned hold = __ballot_sync(0xffffffffu, kth == kmin);
        const bool near = kth != kmin && kth != kbig && tie_near(kth, kmin, P.tol_tie);
        int win = __ffs(hold) - 1, cnt = 1;
        if (kmin != kbig && (__popc(hold) > 1 || __any_sync(0xffffffffu, near))) {
            const bool tied = ok && kth <= dkey(tie_limit(kdouble(kmin), P.tol_tie));
            cnt = __popc(__ballot_sync(0xffffffffu, tied));
            long long kb;
            win = bland ? warp_argmin_index(var, tied) : warp_argmax_key(kal, var, tied, kb);
        }
        if (lane == win) {
            const bool none = kmin == kbig, more = cnt > 1;
            const long long a = __double_as_longlong(al), t = __double_as_longlong(th);
            w[0] = ll_lo(kmin); w[1] = ll_hi(kmin); w[2] = (unsigned)(none ? -1 : (int)blockIdx.x + G * lane);
            w[3] = ll_lo(a); w[4] = ll_hi(a); w[5] = none ? 0u : (unsigned)var | (more ? kRMore : 0u);
            w[6] = ll_lo(t); w[7] = ll_hi(t); w[8] = (unsigned)cnt;
        }
        return;
    }
    __shared__ RowRec o;
    row_record(P, owned, bland, ral, rb, rvar, &o);
    __syncwarp();
    if (lane < 3) {
        const bool more = o.cnt > 1 || dkey(o.th) != o.tmin;
        const long long v = lane == 0 ? o.tmin : __double_as_longlong(lane == 1 ? o.a : o.th);
        w[3 * lane] = ll_lo(v);
        w[3 * lane + 1] = ll_hi(v);
        w[3 * lane + 2] = lane == 0 ? (unsigned)o.row : lane == 1 ? (unsigned)o.var | (more ? kRMore : 0u) : (unsigned)o.cnt;
    }
}

template <bool kA, bool kB>
__global__ void __launch_bounds__(kRThreads, 1) k_iterate_r(DevState s, int iters, int kc, ulonglong2* xbuf,
                                                            unsigned seq0) {
    Ctrl* C = s.ctrl;
    const Params& P = s.p;
    const int m = P.m, n = P.n, ld = P.ld;
    const int G = gridDim.x, b = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool lead = b == 0;
    const int owned = (m - b + G - 1) / G, ownc = (n - b + G - 1) / G;  // <= 0 where b is past the end
    const int nwu = (G + 31) >> 5;  // polling warps
    const ResLayout lay = res_layout(m, n, G, kc, kA, kB);
    const int R = lay.R, Cn = lay.Cn;
    extern __shared__ __align__(16) double dyn[];
    double* ybuf = dyn;               // y in slot order, two copies by step
    double* rh = ybuf + 2 * kc;       // rho / alpha_r
    double* aq = rh + kc;             // the entering column's live rows
    double* bb = aq + kc;             // bbar, alpha, unit part of the entering column: own rows
    double* al = bb + R;
    double* au = al + R;
    double* cst = au + R;             // cost of own columns
    double* Bs = cst + Cn;            // own rows of B^-1
    float* A32 = reinterpret_cast<float*>(Bs + (kB ? (size_t)R * kc : 0));
    float* y32 = A32 + (kA ? (size_t)Cn * kc : 0);
    float* clo = y32 + kc;            // cost rounded down and up
    float* chi = clo + Cn;
    int* ctab = reinterpret_cast<int*>(chi + Cn);  // tabu expiry and basis membership of own columns
    int* cbas = ctab + Cn;
    int* khi = cbas + Cn;             // upper ends of the own columns' intervals
    int* rvar = khi + Cn;             // basic variable of own rows
    uint16_t* sr = reinterpret_cast<uint16_t*>(rvar + R);  // slot -> row, row -> slot
    uint16_t* rs = sr + ((m + 7) & ~7);
    __shared__ IterState S;
    __shared__ volatile int fail;
    __shared__ SlotMoves mv;
    __shared__ PricePatch ppat;
    __shared__ double rinv_sh, cq_sh, thr_sh, dpart[2], cd[kRCand];
    __shared__ int screen_sh;
    __shared__ unsigned pub[2 * kRList], rpub[9];
    __shared__ Cand cpub;
    __shared__ int rep_sh, rep_code, rep_end, rep_row;  // warm-start repair: running, outcome
    __shared__ double rep_val;
    __shared__ int bL, bcnt, bov, nrow, scan_sh;  // the CTA's PRICE record; rows taken by the update; scan
    __shared__ int wL[kRPrice], wov[kRPrice], wn[kRPrice];          // PRICE meeting, per polling warp
    __shared__ int wlj[kRPrice][kRWarpList], wlh[kRPrice][kRWarpList];
    __shared__ int cl[kRCand];
    __shared__ Cand wcand[kRWarps];
    __shared__ long long wmin[kRPrice];                             // ratio meeting, per polling warp
    __shared__ double wa[kRPrice], wth[kRPrice];
    __shared__ int wvar[kRPrice], wrow[kRPrice], wcnt[kRPrice], wmix[kRPrice];
    const long long kbig = dkey(DBL_MAX);
    unsigned seq = seq0;

    // ---- the launch's state into shared memory
    if (tid == 0) {
        fail = 0;
        S.status = C->status; S.it = C->it; S.q = C->q; S.r = C->r; S.tcount = C->tcount;
        S.abuf = C->abuf; S.pending = C->pending; S.flags = C->flags; S.degen_run = C->degen_run;
        S.bland = C->bland; S.dq = C->dq; S.theta = C->theta; S.alpha_r = C->alpha_r;
        S.leave = (S.r >= 0 && S.r < m) ? s.basis[S.r] : -1;
        S.nsb = C->nsb; S.n_degenerate = C->n_degenerate; S.n_tabu = C->n_tabu; S.n_bland = C->n_bland;
        S.n_asp = C->n_asp; S.n_price = C->n_price; S.n_update = C->n_update;
        S.z = C->z; S.bytes_price = C->bytes_price; S.bytes_update = C->bytes_update;
        S.k = C->k_live; S.par = C->map_par;
        screen_sh = P.screen && C->screen_off == 0;
        rep_sh = C->repair == 1;
        rep_code = 0;
    }
    const double rep_tol = C->repair_tol;
    const int rep_limit = C->repair_limit;
    __syncthreads();
    const int par = S.par;
    {
        const int k0 = S.k;
        for (int i = tid; i < m; i += kRThreads) {
            sr[i] = (uint16_t)__ldcg(s.slot_row + (size_t)par * m + i);
            rs[i] = (uint16_t)__ldcg(s.row_slot + (size_t)par * m + i);
        }
        for (int l = tid; l < ownc; l += kRThreads) {
            const int j = b + G * l;
            cst[l] = s.c[j]; clo[l] = s.c32lo[j]; chi[l] = s.c32hi[j];
            ctab[l] = __ldcg(s.tabu_until + j); cbas[l] = __ldcg(s.pos + j) >= 0;
        }
        for (int l = tid; l < owned; l += kRThreads) {
            const int i = b + G * l;
            bb[l] = __ldcg(s.bbar + i); al[l] = __ldcg(s.alpha + (size_t)S.abuf * ld + i);
            rvar[l] = __ldcg(s.basis + i);
        }
        for (int t = tid; t < kc; t += kRThreads) {
            ybuf[t] = t < k0 ? __ldcg(s.yp + (size_t)par * ld + t) : 0.0;
            rh[t] = 0.0;
            aq[t] = 0.0;
        }
        if (kA)
            for (int l = warp; l < ownc; l += kRWarps)
                for (int t = lane; t < kc; t += 32)
                    A32[(size_t)l * kc + t] = t < k0 ? __ldcg(s.A_p32 + (size_t)(b + G * l) * ld + t) : 0.f;
        if (kB)
            for (int l = warp; l < owned; l += kRWarps)
                for (int t = lane; t < kc; t += 32)
                    Bs[(size_t)l * kc + t] = t < k0 ? __ldcg(s.bp + (size_t)(b + G * l) * ld + t) : 0.0;
    }
    // a meeting without a record (off the chain: each sender fences)
    auto meet = [&] {
        __syncthreads();
        ++seq;
        if (tid < G) {
            __threadfence();
            meet_put(xbuf, seq, tid, 0, 0, 0, 0);
            unsigned w[3];
            meet_get<0, 1>(xbuf, seq, tid, w, &fail);
        }
        __syncthreads();
    };
    meet();  // every CTA has read the launch's state before the lead CTA changes any of it

    const bool screen_ok = screen_sh != 0;
    const int kup = fkey(__double2float_ru(P.tol_d)), kdn = fkey(__double2float_rd(P.tol_d));
    double* ycur = ybuf;
    double* ynxt = ybuf + kc;
    auto row_load = [&](int l, int i, int k) -> double2 {  // pair k of own row l (row i)
        return kB ? reinterpret_cast<const double2*>(Bs + (size_t)l * kc)[k]
                  : __ldcg(reinterpret_cast<const double2*>(s.bp + (size_t)i * ld) + k);
    };
    auto row_store = [&](int l, int i, int k, double2 v) {
        if (kB) reinterpret_cast<double2*>(Bs + (size_t)l * kc)[k] = v;
        __stcg(reinterpret_cast<double2*>(s.bp + (size_t)i * ld) + k, v);
    };
    // the pivot's moves of own columns of A_p, by threads t0, t0 + 1, .. of nt
    auto move_rows = [&](int t0, int nt) {
        if (t0 < 0 || (mv.join < 0 && mv.ent < 0)) return;
        int dst[3], src[3];
        const int nm = slot_row_moves(mv, dst, src);
        for (int l = t0; l < ownc && nm > 0; l += nt) {
            double* col = s.A_p + (size_t)(b + G * l) * ld;
            float* col32 = s.A_p32 + (size_t)(b + G * l) * ld;
            double val[3];
#pragma unroll
            for (int e = 0; e < 3; ++e)
                if (e < nm) val[e] = __ldcg(col + src[e]);
#pragma unroll
            for (int e = 0; e < 3; ++e)
                if (e < nm) { __stcg(col + dst[e], val[e]); __stcg(col32 + dst[e], (float)val[e]); }
        }
    };
    // the rank-1 update of the pending pivot on own rows but r: the calling warps
    // take rows from a common counter
    auto apply_rows = [&](int r) {
        const int kh = (mv.kn + 1) >> 1;
        const double2* rh2 = reinterpret_cast<const double2*>(rh);
        int nx = lane == 0 ? atomicAdd(&nrow, 1) : 0;
        for (;;) {
            const int l = __shfl_sync(0xffffffffu, nx, 0);
            if (l >= owned) break;
            if (lane == 0) nx = atomicAdd(&nrow, 1);
            const int i = b + G * l;
            if (i == r) continue;
            const double na = -al[l];
            double bte = 0.0;
            if (mv.src_te >= 0)
                bte = kB ? Bs[(size_t)l * kc + mv.src_te] : __ldcg(s.bp + (size_t)i * ld + mv.src_te);
            __syncwarp();
            if (na != 0.0) {
#pragma unroll 4
                for (int k = lane; k < kh; k += 32) {
                    const double2 o = row_load(l, i, k), p = rh2[k];
                    const int t0 = 2 * k, t1 = t0 + 1;
                    const double b0 = t0 == mv.J ? 0.0 : (t0 == mv.te && mv.src_te >= 0 ? bte : o.x);
                    const double b1 = t1 == mv.J ? 0.0 : (t1 == mv.te && mv.src_te >= 0 ? bte : o.y);
                    row_store(l, i, k, make_double2(fma(na, p.x, b0), fma(na, p.y, b1)));
                }
            } else if (lane == 0) {
                // alpha_i = 0: only the moved columns change
                if (mv.J >= 0) {
                    if (kB) Bs[(size_t)l * kc + mv.J] = 0.0;
                    __stcg(s.bp + (size_t)i * ld + mv.J, 0.0);
                }
                if (mv.src_te >= 0) {
                    if (kB) Bs[(size_t)l * kc + mv.te] = bte;
                    __stcg(s.bp + (size_t)i * ld + mv.te, bte);
                }
            }
        }
    };
    // row r of B^-1 becomes rho / alpha_r (its owner; every CTA has read the old row)
    auto apply_row_r = [&](int r) {
        if (r % G != b) return;
        const int kh = (mv.kn + 1) >> 1;
        for (int k = tid; k < kh; k += kRThreads) row_store(r / G, r, k, reinterpret_cast<const double2*>(rh)[k]);
    };
    // pair k of column j's live rows: A_p, but the live slot D whose row changes
    // with this pivot comes from A itself, since the column's owner may be moving it
    auto col_load = [&](int j, int k, int D) -> double2 {
        double2 v = __ldcg(reinterpret_cast<const double2*>(s.A_p + (size_t)j * ld) + k);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int t = 2 * k + e;
            double x = e ? v.y : v.x;
            if (t == D) x = __ldg(s.A_cm + (size_t)j * ld + sr[t]);
            if (t >= mv.kn) x = 0.0;
            if (e) v.y = x; else v.x = x;
        }
        return v;
    };

    // CHUZR's outcome into S (one thread): the leaving row, or the scan of a tie set
    // that several CTAs' different minima share (tmin: the key of the smallest ratio)
    auto take = [&](long long tmin, int row, int var, double theta, double alpha, int ties, bool scan) {
        S.pending = 0;
        scan_sh = 0;
        if (tmin == kbig) {
            S.status = kUnbounded;
        } else if (scan) {
            scan_sh = 1;
            thr_sh = kdouble(tmin);
        } else {
            S.r = row; S.leave = var; S.theta = theta; S.alpha_r = alpha; S.tcount = ties;
            if (ties > 1) S.flags |= kTfTieSet;
            S.abuf ^= 1;
        }
    };

    for (int step = 0; step < iters && !fail; ++step) {
        // ---- (A) apply the pivot chosen by the last ratio test
        const bool piv = S.status == kRunning && S.r >= 0 && S.r < m && S.q >= 0;
        if (min(S.k + 1, m) > kc) break;  // the live slots may outgrow the layout: the host launches a larger one
        const int r = S.r, q = S.q, leave = S.leave, kold = S.k;
        const double dq = S.dq, th = S.theta;
        const double* brow = s.bp + (size_t)(piv ? r : 0) * ld;
        const int join = piv && leave >= n ? leave - n : -1;
        // columns are dealt to threads from the upper half on: the lower warps have the slots
        const int ct = (tid + kRThreads / 2) & (kRThreads - 1);
        double pre = 0.0, blast = 0.0;
        float vj = 0.f;
        if (piv) {
            // issued before the moves are known: this thread's entry of the pivot
            // row, its last entry (the column that moves when a slack enters), and
            // the joining row of this thread's own column
            if (tid < kold) pre = __ldcg(brow + tid);
            if (q >= n && join < 0) blast = __ldcg(brow + kold - 1);
            if (join >= 0 && ct < ownc) vj = (float)__ldg(s.A_cm + (size_t)(b + G * ct) * ld + join);
        }
        if (tid == 0) {
            if (piv) {
                mv = slot_moves(n, leave, q, kold, [rs](int x) { return (int)rs[x]; },
                                [sr](int t) { return (int)sr[t]; });
                const bool push = P.tabu_tenure > 0 && (S.tcount > 1 || th <= P.tol_tie);
                ppat = pivot_patch(mv, q, leave, push, S.it + 1 + P.tabu_tenure);
            } else {
                mv.join = mv.ent = -1;
                mv.k0 = mv.k1 = mv.kn = kold;
                mv.tl = mv.u = mv.te = mv.w = mv.J = mv.src_te = -1;
                ppat = no_patch();
            }
        }
        if (tid == 32) rinv_sh = piv ? 1.0 / S.alpha_r : 0.0;  // beside the moves, not after them
        __syncthreads();
        const int kn = mv.kn, kk = (kn + 63) & ~63;
        // the scalar work goes to warps of its own, beside the slices below
        if (tid == kRThreads - 96 && piv) {
            for (int e = ppat.nsp - 1; e >= 0; --e)  // the slot maps after the moves (first match wins)
                sr[ppat.sp_slot[e]] = (uint16_t)ppat.sp_row[e];
            if (mv.join >= 0) {
                rs[mv.u] = (uint16_t)mv.tl;
                rs[mv.join] = (uint16_t)mv.J;
            }
            if (mv.ent >= 0) {
                rs[mv.w] = (uint16_t)mv.te;
                rs[mv.ent] = (uint16_t)(mv.k1 - 1);
            }
        }
        if (tid == kRThreads - 64) {
            bL = bov = INT_MIN;
            bcnt = nrow = 0;
            if (piv) {
                pivot_bookkeeping(s, S, lead);
                S.k = kn;
            }
        }
        int ybig = 0;
        {
            const double rinv = rinv_sh;
            for (int t = tid; t < kk; t += kRThreads) {
                double rn = 0.0, yv = 0.0;
                if (t < kn) {
                    yv = ycur[t];
                    if (piv) {
                        double rv = t == tid ? pre : (t < kold ? __ldcg(brow + t) : 0.0);
                        if (t == mv.J) { rv = 1.0; yv = 0.0; }
                        else if (t == mv.te && mv.src_te >= 0) { rv = blast; yv = ycur[mv.src_te]; }
                        rn = rv * rinv;  // one reciprocal per pivot: a division per slot would load the FP64 pipe
                        yv = __dadd_rn(yv, __dmul_rn(dq, rn));
                    }
                }
                rh[t] = rn;
                ynxt[t] = yv;
                y32[t] = (float)yv;
                // screen range: |y| <= 2^40 (exponent field, no FP64 instruction)
                ybig |= ((__double_as_longlong(yv) >> 52) & 0x7ff) > 1023 + 40;
            }
        }
        // the live slot whose row of A changes (-1: none)
        const int D = !piv ? -1 : mv.join >= 0 ? mv.J : (mv.ent >= 0 && mv.te != mv.k0 - 1 ? mv.te : -1);
        if (piv) {
            for (int l = kRThreads - 1 - tid; l < owned; l += kRThreads) {
                const int i = b + G * l;
                const double v = i == r ? th : __dsub_rn(bb[l], __dmul_rn(al[l], th));
                bb[l] = v;
                s.bbar[i] = v;
                if (i == r) rvar[l] = q;
            }
            for (int l = ct; l < ownc; l += kRThreads) {
                const int j = b + G * l;
                if (D >= 0) {
                    float v;
                    if (mv.join >= 0)
                        v = l == ct ? vj : (float)__ldg(s.A_cm + (size_t)j * ld + mv.join);
                    else
                        v = kA ? A32[(size_t)l * kc + mv.k0 - 1] : __ldcg(s.A_p32 + (size_t)j * ld + mv.k0 - 1);
                    if (kA) A32[(size_t)l * kc + D] = v;
                    else __stcg(s.A_p32 + (size_t)j * ld + D, v);
                }
                if (j == q) cbas[l] = 1;
                if (j == leave) {
                    cbas[l] = 0;
                    if (ppat.tabu_j == leave) ctab[l] = ppat.tabu_until;
                }
            }
        }
        const bool yrange = __syncthreads_or(ybig) == 0;
        { double* t = ycur; ycur = ynxt; ynxt = t; }
        const double2* y2 = reinterpret_cast<const double2*>(ycur);
        if (S.status != kRunning) {
            // a reinversion is due or the iteration limit is reached: apply the
            // update and stop (row r once every CTA has read it)
            if (piv) {
                move_rows(tid, kRThreads);
                apply_rows(r);
                meet();
                if (fail) break;
                apply_row_r(r);
                if (tid == 0) {
                    if (lead) { S.bytes_update += 16.0 * m * (double)kn; S.n_update++; }
                    S.pending = 0;
                }
            }
            break;
        }
        if (rep_sh) {
            // ---- a warm-start repair pivot (k_repair_pick's rule): the most negative
            // basic value leaves (ties: the smallest position) and the live slot with
            // the most negative entry of its row enters (ties: the smallest row).  The
            // entering column is a live column, so there is no FTRAN, and one meeting
            // does.
            if (piv) {
                move_rows(tid, kRThreads);
                apply_rows(r);
            }
            __syncthreads();
            ++seq;
            if (warp == kRMail) {
                __threadfence();  // the updated rows
                const long long klim = dkey(-rep_tol);
                long long kb = kbig;
                int pi = INT_MAX, var = 0;
                for (int l = lane; l < owned; l += 32) {
                    const long long key = dkey(bb[l]);
                    if (key < klim && key < kb) { kb = key; pi = b + G * l; var = rvar[l]; }
                }
                const long long wm = warp_min_key(kb);
                const int win = warp_argmin_index(pi, kb == wm && wm != kbig);
                const int pw = __shfl_sync(0xffffffffu, pi, max(win, 0)), vw = __shfl_sync(0xffffffffu, var, max(win, 0));
                for (int d = lane; d < G; d += 32) {
                    meet_put(xbuf, seq, d, 0, ll_lo(wm), ll_hi(wm), (unsigned)(win < 0 ? -1 : pw));
                    meet_put(xbuf, seq, d, 1, 0, 0, (unsigned)vw);
                }
            }
            if (warp < nwu) {
                unsigned w[kRWords];
                long long kb = kbig;
                int pi = INT_MAX, var = 0;
                if (tid < G) {
                    meet_get<0, 2>(xbuf, seq, tid, w, &fail);
                    kb = words_ll(w[0], w[1]);
                    pi = (int)w[2];
                    var = (int)w[5];
                }
                const long long wm = warp_min_key(kb);
                const int win = warp_argmin_index(pi, kb == wm && wm != kbig);
                if (lane == max(win, 0)) { wmin[warp] = wm; wrow[warp] = win < 0 ? -1 : pi; wvar[warp] = var; }
            }
            __syncthreads();
            if (fail) break;
            int gw = 0;
            for (int w = 1; w < nwu; ++w)
                if (wmin[w] < wmin[gw] || (wmin[w] == wmin[gw] && wmin[w] != kbig && wrow[w] < wrow[gw])) gw = w;
            const int p = wmin[gw] == kbig ? -1 : wrow[gw], pvar = wvar[gw];
            const double pval = kdouble(wmin[gw]);
            // row r once every CTA has read it
            if (piv) apply_row_r(r);
            if (p < 0 || S.it >= rep_limit) {
                __syncthreads();
                if (tid == 0) {
                    rep_code = p < 0 ? 2 : 4;
                    rep_end = S.it;
                    rep_sh = 0;
                    S.r = S.q = -1;
                    S.pending = 0;
                }
                __syncthreads();
                if (rep_code == 2) continue;  // feasible: the method goes on from here
                break;
            }
            long long ek = kbig;
            int er = INT_MAX;
            for (int t = tid; t < kn; t += kRThreads) {
                const long long key = dkey(__ldcg(s.bp + (size_t)p * ld + t));
                const int row = sr[t];
                if (key < 0 && (key < ek || (key == ek && row < er))) { ek = key; er = row; }
            }
            const long long wm = warp_min_key(ek);
            const int win = warp_argmin_index(er, ek == wm && wm != kbig);
            if (lane == max(win, 0)) { wcand[warp].d_all = wm; wcand[warp].j_all = win < 0 ? -1 : er; }
            __syncthreads();
            if (tid == 0) {
                long long km = kbig;
                int jr = -1;
                for (int w = 0; w < kRWarps; ++w)
                    if (wcand[w].j_all >= 0 &&
                        (jr < 0 || wcand[w].d_all < km || (wcand[w].d_all == km && wcand[w].j_all < jr))) {
                        km = wcand[w].d_all;
                        jr = wcand[w].j_all;
                    }
                rep_row = jr;
                rep_val = kdouble(km);
            }
            __syncthreads();
            if (rep_row < 0) {
                // no slack can repair the row
                if (tid == 0) {
                    rep_code = 3;
                    rep_end = S.it;
                    S.r = S.q = -1;
                    S.pending = 0;
                }
                break;
            }
            const int es = rs[rep_row];
            double* anxt = s.alpha + (size_t)(S.abuf ^ 1) * ld;
            for (int l = tid; l < owned; l += kRThreads) {
                const int i = b + G * l;
                const double v = kB ? Bs[(size_t)l * kc + es] : __ldcg(s.bp + (size_t)i * ld + es);
                al[l] = v;
                anxt[i] = v;
            }
            __syncthreads();
            if (tid == 0) {
                S.q = n + rep_row; S.r = p; S.leave = pvar;
                S.dq = -ycur[es];
                S.theta = pval / rep_val;
                S.alpha_r = rep_val;
                S.tcount = 1; S.flags = 0; S.pending = 0;
                S.abuf ^= 1;
            }
            __syncthreads();
            continue;
        }
        // ---- PRICE + CHUZC
        const bool bland = S.bland != 0;
        const int it = S.it;
        int qn = -1;         // the entering variable, or -1: the FP64 pricing decides
        bool dq_known = false;
        if (screen_ok && yrange) {
            ++seq;
            if (warp < kRPrice) {
                // slack candidates (own live slots t = b + G * lane), by the last pricing
                // warp: their tabu expiry is loaded before its columns
                const int nsl = warp == kRPrice - 1 && kn > b ? (kn - b + G - 1) / G : 0;
                int srow = -1, stab = 0;
                if (lane < nsl) {
                    srow = sr[b + G * lane];
                    stab = patched_tabu(s, ppat, n + srow);
                }
                const int n4 = kk >> 2;
                const int depth = 4 * ((n4 + 31) >> 5) + 5;
                const float umul = __fmul_ru((float)(depth + 3), 6.0200691e-8f);  // (d + 3) u 1.01, rounded up
                const float uabs = __fmul_ru((float)(kk + 8), 7.8886091e-31f);     // (k + 8) 2^-100: underflow
                const float4* y4 = reinterpret_cast<const float4*>(y32);
                // bL: the largest lower end, or (Bland) minus the smallest surely improving index
                for (int e0 = 4 * warp; e0 < ownc; e0 += 4 * kRPrice) {
                    float sv, av;
                    screen4(
                        [&](int c, int k) {
                            const int l = min(e0 + c, ownc - 1);
                            return kA ? reinterpret_cast<const float4*>(A32 + (size_t)l * kc)[k]
                                      : __ldcg(reinterpret_cast<const float4*>(s.A_p32 + (size_t)(b + G * l) * ld) + k);
                        },
                        y4, n4, lane, sv, av);
                    const int l = e0 + (lane >> 3);
                    if ((lane & 7) == 0 && l < ownc) {
                        const float E = __fmaf_ru(umul, av, uabs);
                        const bool in = !cbas[l] && (bland || ctab[l] <= it);
                        const int lo = fkey(__fsub_rd(clo[l], __fadd_ru(sv, E)));
                        khi[l] = in ? fkey(__fadd_ru(__fsub_ru(chi[l], sv), E)) : INT_MIN;
                        if (in && (!bland || lo > kup)) atomicMax(&bL, bland ? -(b + G * l) : lo);
                    }
                }
                auto slack = [&](int t, int& lo, int& hi, int& j) {
                    const int row = t == lane ? srow : (int)sr[b + G * t];
                    const int tb = t == lane ? stab : patched_tabu(s, ppat, n + row);
                    const double d = -ycur[b + G * t];
                    const bool in = bland || tb <= it;
                    j = n + row;
                    lo = in ? fkey(__double2float_rd(d)) : INT_MIN;
                    hi = in ? fkey(__double2float_ru(d)) : INT_MIN;
                };
                for (int t = lane; t < nsl; t += 32) {
                    int lo, hi, j;
                    slack(t, lo, hi, j);
                    if (hi != INT_MIN && (!bland || lo > kup)) atomicMax(&bL, bland ? -j : lo);
                }
                asm volatile("bar.sync 1, %0;\n" ::"n"(32 * kRPrice) : "memory");
                // the columns that can be the CTA's choice: those whose upper end reaches bL
                // (Bland: that may improve and precede the smallest surely improving one)
                const int L0 = bL;
                auto offer = [&](int hi, int j) {
                    if (hi == INT_MIN || !(bland ? hi > kdn && -j > L0 : hi >= L0)) return;
                    const int key = bland ? -j : hi;
                    const int e = atomicAdd(&bcnt, 1);
                    if (e < kRList) { pub[2 * e] = (unsigned)key; pub[2 * e + 1] = (unsigned)j; }
                    else atomicMax(&bov, key);
                };
                for (int l = tid; l < ownc; l += 32 * kRPrice) offer(khi[l], b + G * l);
                for (int t = lane; t < nsl; t += 32) {
                    int lo, hi, j;
                    slack(t, lo, hi, j);
                    offer(hi, j);
                }
                asm volatile("bar.sync 1, %0;\n" ::"n"(32 * kRPrice) : "memory");
                if (tid < G) {
                    // chunk 0 says all when at most one column is listed
                    const int cnt = min(bcnt, kRList);
                    meet_put(xbuf, seq, tid, 0, (unsigned)bL, cnt ? pub[0] : (unsigned)INT_MIN,
                             (cnt ? pub[1] : 0u) | (cnt > 1 ? kRMore : 0u));
                    if (cnt > 1) {
                        meet_put(xbuf, seq, tid, 1, (unsigned)cnt, pub[2], pub[3]);
                        meet_put(xbuf, seq, tid, 2, (unsigned)bov, pub[4], pub[5]);
                        meet_put(xbuf, seq, tid, 3, 0, pub[6], pub[7]);
                    }
                }
                if (warp < nwu) {
                    unsigned w[kRWords];
                    w[0] = w[1] = w[6] = (unsigned)INT_MIN;
                    w[2] = 0;
                    w[3] = 1;
                    if (tid < G) {
                        meet_get<0, 1>(xbuf, seq, tid, w, &fail);
                        if (w[2] & kRMore) meet_get<1, 4>(xbuf, seq, tid, w, &fail);
                    }
                    const int L = __reduce_max_sync(0xffffffffu, (int)w[0]);
                    const bool more = __any_sync(0xffffffffu, w[2] & kRMore);
                    int ov = INT_MIN, cnt = 0;
                    auto list = [&](bool listed, int key, int j) {
                        const bool in = listed && key != INT_MIN && (bland ? key > L : key >= L);
                        const unsigned bal = __ballot_sync(0xffffffffu, in);
                        if (in) {
                            const int x = cnt + __popc(bal & ((1u << lane) - 1u));
                            if (x < kRWarpList) { wlh[warp][x] = key; wlj[warp][x] = j; }
                        }
                        cnt += __popc(bal);
                    };
                    list(true, (int)w[1], (int)(w[2] & ~kRMore));
                    if (more) {
                        const bool mine = w[2] & kRMore;
                        list(mine, (int)w[4], (int)w[5]);
                        list(mine && w[3] > 2, (int)w[7], (int)w[8]);
                        list(mine && w[3] > 3, (int)w[10], (int)w[11]);
                        ov = __reduce_max_sync(0xffffffffu, mine ? (int)w[6] : INT_MIN);
                    }
                    if (cnt > kRWarpList) { cnt = kRWarpList; ov = INT_MAX; }
                    if (lane == 0) { wL[warp] = L; wov[warp] = ov; wn[warp] = cnt; }
                }
            }
            // the others, and the pricing warps that do not poll: the pivot's moves and update
            if (piv && warp >= nwu) {
                if (warp < kRPrice) move_rows(tid - 32 * nwu, 32 * (kRPrice - nwu));
                apply_rows(r);
            }
            __syncthreads();
            if (fail) break;
            // ---- CHUZC: every warp reads the polling warps' lists, one per lane
            int L, cnt, j1;
            bool over;
            if (nwu == 1) {
                L = wL[0];
                cnt = wn[0];
                j1 = wlj[0][0];
                over = bland ? wov[0] > L : wov[0] >= L && wov[0] != INT_MIN;
            } else {
                const int lL = lane < nwu ? wL[lane] : INT_MIN, lov = lane < nwu ? wov[lane] : INT_MIN;
                const int ln = lane < nwu ? wn[lane] : 0;
                const int lh = ln > 0 ? wlh[lane][0] : INT_MIN, lj = ln > 0 ? wlj[lane][0] : -1;
                L = __reduce_max_sync(0xffffffffu, lL);
                const unsigned first = __ballot_sync(0xffffffffu, ln > 0 && (bland ? lh > L : lh >= L));
                cnt = __popc(first);
                j1 = __shfl_sync(0xffffffffu, lj, first ? __ffs(first) - 1 : 0);
                if (__any_sync(0xffffffffu, ln > 1)) {
                    cnt = 0;
                    for (int w = 0; w < nwu; ++w)
                        for (int e = 0; e < wn[w]; ++e)
                            if (bland ? wlh[w][e] > L : wlh[w][e] >= L) { ++cnt; j1 = wlj[w][e]; }
                }
                over = __any_sync(0xffffffffu, bland ? lov > L : lov >= L && lov != INT_MIN);
            }
            // surely improving, and no list overflowed where it matters
            const bool sure = bland ? L != INT_MIN : L > kup;
            if (sure && !over && cnt + (bland ? 1 : 0) <= kRCand) {
                if (bland && cnt == 0) qn = -L;
                else if (!bland && cnt == 1) qn = j1;
                else {
                    // several candidates: each priced exactly by one warp, in every CTA alike
                    if (tid == 0) {
                        int x = 0;
                        for (int w = 0; w < nwu; ++w)
                            for (int e = 0; e < wn[w]; ++e)
                                if (bland ? wlh[w][e] > L : wlh[w][e] >= L) cl[x++] = wlj[w][e];
                        if (bland) cl[x++] = -L;
                    }
                    __syncthreads();
                    const int nc = cnt + (bland ? 1 : 0);
                    for (int e = warp; e < nc; e += kRWarps) {
                        const int j = cl[e];
                        double d;
                        if (j < n) d = s.c[j] - exact_dot([&](int k) { return col_load(j, k, D); }, y2, kk, lane);
                        else d = -ycur[rs[j - n]];
                        if (lane == 0) cd[e] = d;
                    }
                    __syncthreads();
                    long long best = LLONG_MIN;
                    double d = 0.0;
                    const long long ktol = dkey(P.tol_d);
                    for (int e = 0; e < nc; ++e) {
                        const long long key = dkey(cd[e]);
                        const int j = cl[e];
                        if (bland ? (key > ktol && (qn < 0 || j < qn)) : beats(key, j, best, qn)) {
                            best = key; qn = j; d = cd[e];
                        }
                    }
                    if (tid == 0) S.dq = d;
                    dq_known = true;
                }
                if (tid == 0 && bland) S.flags |= kTfBland;
            }
        } else {
            if (piv) {
                move_rows(tid, kRThreads);
                apply_rows(r);
            }
            __syncthreads();
        }
        if (qn < 0) {
            // ---- full FP64 PRICE of own columns and live slots, one more meeting
            Cand cand;
            cand_init(cand);
            const long long ktol = dkey(P.tol_d);
            for (int l = warp; l < ownc; l += kRWarps) {
                if (cbas[l]) continue;
                const double2* col = reinterpret_cast<const double2*>(s.A_p + (size_t)(b + G * l) * ld);
                const double d = cst[l] - exact_dot([&](int k) { return __ldcg(col + k); }, y2, kk, lane);
                if (lane == 0) cand_offer(cand, d, b + G * l, ctab[l] <= it, ktol, kNoRank);
            }
            for (int t = b + G * tid; t < kn; t += G * kRThreads) {
                const int j = n + sr[t];
                cand_offer(cand, -ycur[t], j, patched_tabu(s, ppat, j) <= it, ktol, kNoRank);
            }
            cand = cand_warp_reduce(cand);
            if (lane == 0) wcand[warp] = cand;
            __syncthreads();
            ++seq;
            if (warp == 0) {
                cand_init(cand);
                if (lane < kRWarps) cand = wcand[lane];
                cand = cand_warp_reduce(cand);
                if (lane == 0) cpub = cand;
            }
            __syncthreads();  // (and wcand is written again)
            if (warp < nwu) {
                unsigned w[kRWords];
                if (tid < G) {
                    __threadfence();
                    meet_put(xbuf, seq, tid, 0, ll_lo(cpub.d_all), ll_hi(cpub.d_all), (unsigned)cpub.j_all);
                    meet_put(xbuf, seq, tid, 1, ll_lo(cpub.d_nt), ll_hi(cpub.d_nt), (unsigned)cpub.j_nt);
                    meet_put(xbuf, seq, tid, 2, ll_lo(cpub.d_min), ll_hi(cpub.d_min), (unsigned)cpub.j_min);
                }
                cand_init(cand);
                if (tid < G) {
                    meet_get<0, 3>(xbuf, seq, tid, w, &fail);
                    cand.d_all = words_ll(w[0], w[1]); cand.d_nt = words_ll(w[3], w[4]); cand.d_min = words_ll(w[6], w[7]);
                    cand.j_all = (int)w[2]; cand.j_nt = (int)w[5]; cand.j_min = (int)w[8];
                }
                cand = cand_warp_reduce(cand);
                if (lane == 0) wcand[warp] = cand;
            }
            __syncthreads();
            if (fail) break;
            if (tid == 0) {
                Cand g = wcand[0];
                for (int w = 1; w < nwu; ++w) cand_merge(g, wcand[w]);
                const Chuzc d = chuzc_decide(g, bland, P.tol_d);
                if (d.optimal) {
                    S.status = kOptimal;
                    S.q = -1;
                } else {
                    S.q = d.q;
                    S.dq = d.dq;
                    S.flags |= d.flags;
                }
                if (lead) S.n_asp += d.asp;
            }
            __syncthreads();
            qn = S.q;
            dq_known = true;
        } else if (tid == 0) {
            S.q = qn;
        }
        if (lead && tid == kRThreads - 64) {
            S.bytes_price += 8.0 * kn * (double)(n - S.nsb);
            S.n_price++;
            S.bytes_update += (piv ? 16.0 : (qn >= 0 ? 8.0 : 0.0)) * m * (double)kn;
            S.n_update += piv || qn >= 0;
        }
        // ---- (B) the entering column's live rows and its entries on own basic slacks
        if (piv) apply_row_r(r);
        if (qn < 0 || qn >= n + m) {  // optimal
            if (tid == 0) S.pending = 0;
            break;
        }
        if (qn < n) {
            for (int k = tid; 2 * k < kk; k += kRThreads) reinterpret_cast<double2*>(aq)[k] = col_load(qn, k, D);
            for (int l = kRThreads - 1 - tid; l < owned; l += kRThreads) {
                const int v = rvar[l];
                au[l] = v >= n ? __ldg(s.A_cm + (size_t)qn * ld + (v - n)) : 0.0;
            }
            if (tid == kRThreads / 2) cq_sh = __ldg(s.c + qn);
        } else {
            const int unit = rs[qn - n];
            for (int t = tid; t < kk; t += kRThreads) aq[t] = t == unit ? 1.0 : 0.0;
            for (int l = tid; l < owned; l += kRThreads) au[l] = 0.0;
        }
        __syncthreads();
        // ---- FTRAN of own rows (two per warp at a time), and the exact d_q
        {
            double* anxt = s.alpha + (size_t)(S.abuf ^ 1) * ld;
            const double2* aq2 = reinterpret_cast<const double2*>(aq);
            const int kh = (kn + 1) >> 1;
            for (int l0 = warp; l0 < owned; l0 += 2 * kRWarps) {
                const int l1 = l0 + kRWarps;
                const bool two = l1 < owned;
                const int i0 = b + G * l0, i1 = b + G * l1;
                double a0 = 0.0, a1 = 0.0, c0 = 0.0, c1 = 0.0;
#pragma unroll 4
                for (int k = lane; k < kh; k += 32) {
                    const double2 w = aq2[k];
                    const double2 x = row_load(l0, i0, k);
                    const bool in = 2 * k + 1 < kn;
                    a0 = fma(x.x, w.x, a0);
                    if (in) a1 = fma(x.y, w.y, a1);
                    if (two) {
                        const double2 z = row_load(l1, i1, k);
                        c0 = fma(z.x, w.x, c0);
                        if (in) c1 = fma(z.y, w.y, c1);
                    }
                }
                const double s0 = warp_sum2_fixed(a0, a1);
                const double s1 = two ? warp_sum2_fixed(c0, c1) : 0.0;
                if (lane == 0) {
                    const double v = s0 + au[l0];
                    al[l0] = v;
                    anxt[i0] = v;
                    s.row_var[i0] = rvar[l0];
                    if (two) {
                        const double u = s1 + au[l1];
                        al[l1] = u;
                        anxt[i1] = u;
                        s.row_var[i1] = rvar[l1];
                    }
                }
            }
            // What the other CTAs read after the ratio meeting was written before this step's
            // last block barrier.  The record's warp, which has the fewest rows, fences
            // here, beside FTRAN: after the next block barrier it cost 0.6 us of every pivot.
            if (warp == kRMail) __threadfence();
            if (!dq_known && qn < n && warp >= kRWarps - 3 && warp < kRWarps - 1) {
                // the two row segments of price_block
                const int nch = kk >> 6, sg = warp - (kRWarps - 3);
                const int k1 = sg ? 32 * nch : 32 * (nch / 2);
                double a = 0.0;
                for (int k = (sg ? 32 * (nch / 2) : 0) + lane; k < k1; k += 32) {
                    const double2 c = aq2[k], y = y2[k];
                    a = fma(c.y, y.y, fma(c.x, y.x, a));
                }
                a = pair_sum(a);
                if (lane == 0) dpart[sg] = a;
            }
        }
        __syncthreads();
        // ---- the CTA's ratio-test record, by the warp that fenced
        ++seq;
        if (warp == kRMail) {
            ratio_record(P, owned, bland, al, bb, rvar, rpub);
            __syncwarp();
            for (int d = lane; d < G; d += 32) {
                meet_put(xbuf, seq, d, 0, rpub[0], rpub[1], rpub[2]);
                meet_put(xbuf, seq, d, 1, rpub[3], rpub[4], rpub[5]);
                if (rpub[5] & kRMore) meet_put(xbuf, seq, d, 2, rpub[6], rpub[7], rpub[8]);
            }
        } else if (tid == kRThreads - 64 && !dq_known) {
            S.dq = qn < n ? cq_sh - (dpart[0] + dpart[1]) : -ycur[rs[qn - n]];
        }
        if (warp < nwu) {
            unsigned w[kRWords];
            long long tmin = kbig;
            double ra = 0.0;
            int var = 0, row = -1;
            bool more = false;
            if (tid < G) {
                meet_get<0, 2>(xbuf, seq, tid, w, &fail);
                tmin = words_ll(w[0], w[1]);
                row = (int)w[2];
                ra = __longlong_as_double(words_ll(w[3], w[4]));
                var = (int)(w[5] & ~kRMore);
                more = w[5] & kRMore;
            }
            const long long wm = warp_min_key(tmin);
            const bool hold = tmin == wm && row >= 0;
            const unsigned bal = __ballot_sync(0xffffffffu, hold);
            int win = bal ? __ffs(bal) - 1 : 0, tot = 1;
            double rth = kdouble(wm);
            bool mix = false;
            // usually one record holds the smallest ratio, it is its CTA's only tied
            // row, and no other record lies near it: that row.  Else the records that
            // hold the smallest ratio (same threshold) merge, and others within the
            // threshold need the scan of all rows
            if (wm != kbig && (__popc(bal) > 1 || __any_sync(0xffffffffu, hold ? more : tie_near(tmin, wm, P.tol_tie)))) {
                rth = kdouble(tmin);
                int cnt = hold ? 1 : 0;
                if (more) {
                    meet_get<2, 3>(xbuf, seq, tid, w, &fail);
                    rth = __longlong_as_double(words_ll(w[6], w[7]));
                    cnt = (int)w[8];
                }
                const long long wt = dkey(tie_limit(kdouble(wm), P.tol_tie));
                mix = __any_sync(0xffffffffu, !hold && tmin <= wt);
                tot = __reduce_add_sync(0xffffffffu, hold ? cnt : 0);
                long long kb;
                win = bland ? warp_argmin_index(var, hold) : warp_argmax_key(dkey(ra), var, hold, kb);
            }
            if (lane == win) {
                if (nwu == 1) {
                    take(wm, row, var, rth, ra, tot, mix);
                } else {
                    wmin[warp] = wm; wa[warp] = ra; wth[warp] = rth;
                    wvar[warp] = var; wrow[warp] = row; wcnt[warp] = tot; wmix[warp] = mix;
                }
            }
        }
        __syncthreads();
        if (fail) break;
        if (nwu > 1) {
            // the polling warps' results, one per lane
            if (warp == 0) {
                const bool in = lane < nwu;
                const long long km = in ? wmin[lane] : kbig;
                const double a = in ? wa[lane] : 0.0, t = in ? wth[lane] : 0.0;
                const int var = in ? wvar[lane] : 0, row = in ? wrow[lane] : -1, wc = in ? wcnt[lane] : 0;
                const bool wx = in && wmix[lane] != 0;
                const long long gmin = warp_min_key(km);
                const bool hold = in && km == gmin;
                const unsigned bal = __ballot_sync(0xffffffffu, hold);
                int gw = __ffs(bal) - 1, tie = __shfl_sync(0xffffffffu, wc, gw);
                bool scan = false;
                long long gthr = 0;
                if (gmin != kbig && (__popc(bal) > 1 || __any_sync(0xffffffffu, hold ? wx : in && tie_near(km, gmin, P.tol_tie)))) {
                    gthr = dkey(tie_limit(kdouble(gmin), P.tol_tie));
                    scan = __any_sync(0xffffffffu, hold ? wx : in && km <= gthr);
                    long long kb;
                    gw = bland ? warp_argmin_index(var, hold) : warp_argmax_key(dkey(a), var, hold, kb);
                    tie = __reduce_add_sync(0xffffffffu, hold ? wc : 0);
                }
                if (lane == gw) take(gmin, row, var, t, a, tie, scan);
            }
            __syncthreads();
        }
        if (scan_sh) {
            // CTAs with other minima lie within the tie tolerance: scan the rows of all CTAs
            meet();
            if (fail) break;
            const double thr = tie_limit(thr_sh, P.tol_tie);
            const double* anxt = s.alpha + (size_t)(S.abuf ^ 1) * ld;
            RowCand best = {0.0, 0, -1, 0.0};
            int cnt = 0;
            for (int i = tid; i < m; i += kRThreads) {
                const double a = __ldcg(anxt + i), x = __ldcg(s.bbar + i);
                if (a > P.tol_piv && x <= thr * a) {
                    cnt++;
                    const RowCand c = {a, __ldcg(s.row_var + i), i, 0.0};
                    if (row_beats(c, best, bland)) best = c;
                }
            }
            best = block_row_best(best, cnt, bland);  // in thread 0
            if (tid == 0) {
                if (best.row < 0) {
                    S.status = kUnbounded;
                    if (lead) C->err = kErrBadIndex;
                } else {
                    S.theta = __ldcg(s.bbar + best.row) / best.a;
                    S.r = best.row; S.leave = best.var; S.alpha_r = best.a; S.tcount = cnt;
                    if (cnt > 1) S.flags |= kTfTieSet;
                    S.abuf ^= 1;
                }
            }
            meet();  // every CTA has scanned before any CTA's next step changes bbar
            if (fail) break;
        }
        if (S.status != kRunning) break;
    }
    __syncthreads();
    // ---- what other kernels read: the slot maps, the basic slacks' slots, y
    for (int l = tid; l < owned; l += kRThreads) {
        const int v = rvar[l];
        s.uslot[b + G * l] = v >= n ? (int)rs[v - n] : -1;
    }
    if (lead) {
        for (int i = tid; i < m; i += kRThreads) {
            s.slot_row[(size_t)par * m + i] = sr[i];
            s.row_slot[(size_t)par * m + i] = rs[i];
        }
        const int kn = S.k;
        if (kn <= kc)  // (else the launch did not fit and no step ran)
            for (int t = tid; t < ld; t += kRThreads) s.yp[(size_t)par * ld + t] = t < kn ? ycur[t] : 0.0;
        if (tid == 0) {
            iterate_flush(s, S);
            if (rep_code) {
                C->repair = rep_code;
                C->repair_end = rep_end;
            }
        }
    }
    report_timeout(fail, &C->err);
}

// Self-test of the bounded meeting: CTA 0's record for the last CTA is never sent, so that
// CTA alone must give up after the spin limit and report it.
__global__ void k_meeting_selftest(ulonglong2* xbuf, int32_t* err) {
    __shared__ volatile int fail;
    const int tid = threadIdx.x, G = gridDim.x;
    if (tid == 0) fail = 0;
    __syncthreads();
    if (tid < G) {
        if (blockIdx.x != 0 || tid != G - 1) meet_put(xbuf, 1, tid, 0, 0, 0, 0);
        unsigned w[3];
        meet_get<0, 1>(xbuf, 1, tid, w, &fail);
    }
    __syncthreads();
    report_timeout(fail, err);
}

using ResKernel = void (*)(DevState, int, int, ulonglong2*, unsigned);
ResKernel res_kernel(bool a, bool b) {
    return a ? (b ? k_iterate_r<true, true> : k_iterate_r<true, false>) : k_iterate_r<false, false>;
}

}  // namespace

cudaError_t launch_meeting_selftest(int blocks, void* meet, int32_t* err, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3((blocks + 31) / 32 * 32);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_meeting_selftest, static_cast<ulonglong2*>(meet), err);
}

// CTAs of a launch.  A CTA's share of the screen, the update and FTRAN falls with
// the number of CTAs, and the two meetings of a pivot grow with it (one warp polls
// up to 32 records, five warps 152 and a second reduction).
// Measured, us per pivot at 16 / 32 / 64 / 112 / 152 CTAs: 128 x 256 8.4 / 8.6 / 9.0 /
// 9.5 / 10.1, 256 x 512 9.3 / 8.3 / 8.5 / 9.0 / 9.8, 512 x 1024 11.2 / 9.6 / 8.8 / 9.1 / 9.7,
// 701 x 1203 - / 10.1 / 9.0 / 9.1 / 9.8, 1024 x 2048 - / 12.2 / 10.4 / 9.5 / 10.1, 2048 x 4096
// - / - / - / 12.6 / 11.8: the best number follows the cube root of m n, with one polling
// warp wherever that is near.
int resident_ctas(int sms, int m, int n) {
    int g = (int)std::lround(0.85 * std::cbrt((double)m * n));
    if (g < 56) g = std::min(std::max(g, 16), 32);
    return std::max(1, std::min(std::min(g, std::max(m, n)), std::min(kRMaxCtas, sms)));
}

unsigned resident_meetings(int iters) { return kRStepMeetings * (unsigned)iters + 1; }

size_t resident_meet_bytes(int ctas) { return sizeof(ulonglong2) * 2 * kRChunks * (size_t)ctas * ctas; }

cudaError_t resident_room(size_t* room) {
    size_t r[3] = {};
    cudaError_t e = raise_smem_limit<k_iterate_r<true, true>>(&r[0]);
    if (e == cudaSuccess) e = raise_smem_limit<k_iterate_r<true, false>>(&r[1]);
    if (e == cudaSuccess) e = raise_smem_limit<k_iterate_r<false, false>>(&r[2]);
    *room = std::min(r[0], std::min(r[1], r[2]));
    return e;
}

// The layouts in order: A and B^-1 in shared memory, A alone, neither.  Each is faster
// than k_iterate_s wherever it is the one that fits (us per pivot, k live rows):
//   both     4096 x 8192, k = 300   17.9 / 32.5;  5500 x 11000, k = 200    22 / 38
//   A alone  4096 x 8192, k = 500   22.1 / 36.3;  k = 700    28.5 / 41.8;
//            5500 x 11000, k = 500  30 / 49;      1800 x 2000, k = 1000  22.3 / 31.8
//   neither  4096 x 8192, k = 1000  37.7 / 50.4;  k = 2000   78.7 / 86.5;
//            5500 x 11000, k = 900  52 / 70;      k = 2500  141 / 150;  120 x 70000  16.5 / 29.6
bool resident_plan(int m, int n, int ld, int ctas, int k_live, int iters, size_t room, ResidentPlan* out) {
    // room for every pivot of the launch to add a live slot, and at least one
    const int want = std::min(ld, (k_live + iters + 1 + 63) & ~63);
    for (int v = 0; v < 3; ++v) {
        const bool a = v < 2, b = v < 1;
        const int least = std::min(ld, (k_live + 1 + 63) & ~63);
        for (int kc = want; kc >= least; kc -= 64) {
            const ResLayout l = res_layout(m, n, ctas, kc, a, b);
            if (l.bytes <= room) {
                out->ctas = ctas; out->kc = kc; out->a = a; out->b = b; out->smem = l.bytes;
                return true;
            }
        }
    }
    return false;
}

cudaError_t launch_iterate_r(const DevState& s, const ResidentPlan& p, int iters, void* meet, unsigned seq0,
                             cudaStream_t st) {
    ResKernel k = res_kernel(p.a, p.b);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.ctas);
    cfg.blockDim = dim3(kRThreads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, s, iters, p.kc, static_cast<ulonglong2*>(meet), seq0);
}

}  // namespace lpgb
