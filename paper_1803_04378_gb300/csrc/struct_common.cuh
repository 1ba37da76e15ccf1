// struct_common.cuh -- building blocks of the two persistent kernels on the
// slack-structured inverse (kernels_struct.cu, kernels_resident.cu): the slot
// moves of a pivot, the fixed-point warp sum of FTRAN, a CTA's ratio-test
// record and the integer image of a float.  Included by one translation unit
// per kernel; everything lives in an anonymous namespace.
#pragma once
#include "iter_common.cuh"

namespace lpgb {
namespace {

// The slot moves of one pivot (every CTA computes the same values).
struct SlotMoves {
    int join, ent;   // rows entering / leaving R (-1: none)
    int k0, k1, kn;  // live slots before, after the join, after the drop
    int tl;          // old slot of `join`
    int u;           // row displaced from slot k0 by the join
    int te;          // slot of `ent`, which receives row w
    int w;           // row moved into slot te
    int J;           // new slot of the joining row's column (-1: none)
    int src_te;      // old slot whose column moves to te (-1: none or the join)
};

// slot_of / row_at: the current row -> slot and slot -> row maps.
template <typename SlotOf, typename RowAt>
__device__ __forceinline__ SlotMoves slot_moves(int n, int leave, int q, int k, SlotOf slot_of, RowAt row_at) {
    SlotMoves v;
    v.join = leave >= n ? leave - n : -1;
    v.ent = q >= n ? q - n : -1;
    v.k0 = k;
    v.tl = v.join >= 0 ? slot_of(v.join) : -1;
    v.u = v.join >= 0 ? row_at(k) : -1;
    v.k1 = k + (v.join >= 0 ? 1 : 0);
    v.te = v.ent >= 0 ? slot_of(v.ent) : -1;
    v.w = v.ent >= 0 ? (v.join >= 0 ? v.join : row_at(k - 1)) : -1;
    v.kn = v.k1 - (v.ent >= 0 ? 1 : 0);
    v.J = v.join >= 0 ? (v.ent >= 0 ? v.te : v.k0) : -1;
    v.src_te = (v.ent >= 0 && v.join < 0) ? v.k0 - 1 : -1;
    return v;
}

// The rows of A_p that move with a pivot: slot dst[e] receives the row of slot
// src[e] (at most three; all sources are read before any is written).
__device__ __forceinline__ int slot_row_moves(const SlotMoves& v, int (&dst)[3], int (&src)[3]) {
    int nm = 0;
    if (v.ent >= 0 && v.join >= 0) {
        dst[0] = v.te; src[0] = v.tl;
        dst[1] = v.k0; src[1] = v.te;
        nm = 2;
        if (v.tl != v.k0) { dst[2] = v.tl; src[2] = v.k0; nm = 3; }
    } else if (v.ent >= 0) {
        if (v.te != v.k0 - 1) { dst[0] = v.te; src[0] = v.k0 - 1; dst[1] = v.k0 - 1; src[1] = v.te; nm = 2; }
    } else if (v.join >= 0 && v.tl != v.k0) {
        dst[0] = v.k0; src[0] = v.tl; dst[1] = v.tl; src[1] = v.k0; nm = 2;
    }
    return nm;
}

// new slot_row entry of slot t / new row_slot entry of row x
__device__ __forceinline__ int moved_slot_row(const SlotMoves& v, int t, int old) {
    if (v.ent >= 0 && t == v.te) return v.w;
    if (v.ent >= 0 && t == v.k1 - 1) return v.ent;
    if (v.join >= 0 && t == v.k0) return v.join;
    if (v.join >= 0 && t == v.tl) return v.u;
    return old;
}
__device__ __forceinline__ int moved_row_slot(const SlotMoves& v, int x, int old) {
    if (v.ent >= 0 && x == v.ent) return v.k1 - 1;
    if (v.ent >= 0 && x == v.w) return v.te;
    if (v.join >= 0 && x == v.join) return v.J;
    if (v.join >= 0 && x == v.u) return v.tl;
    return old;
}

// Source of slot t's rho and y after the moves: an old slot, or -2 for the
// joining row (rho = 1, y = 0: its old column is e_r and its y is zero).
__device__ __forceinline__ int vec_src(const SlotMoves& v, int t) {
    if (t == v.J) return -2;
    if (t == v.te && v.src_te >= 0) return v.src_te;
    return t;
}

// Warp sum of a + b over the 32 lanes (every lane gets it) in 64-bit fixed
// point.  The values are aligned to the warp's largest binary exponent E
// (one redux): a value is t 2^(E - 1079) with |t| < 2^57, rounded to nearest;
// the t are added exactly as integers, and the sum is rounded to
// binary64 once (ll_scaled).  Relative to 2^(E - 1022), which bounds every
// |value|, the error is below 2^-51 plus the final rounding -- no more than
// the FP64 butterfly's -- and the sum does not depend on the lane order.  It
// spends no FP64 instruction (each holds the FP64 pipe for ~64 cycles on this
// chip, and the butterfly needs six per row).  Subnormal, infinite and NaN
// inputs take the FP64 butterfly.
__device__ __forceinline__ double warp_sum2_fixed(double a, double b) {
    const unsigned long long ua = (unsigned long long)__double_as_longlong(a);
    const unsigned long long ub = (unsigned long long)__double_as_longlong(b);
    const int ea = (int)((ua >> 52) & 0x7ff), eb = (int)((ub >> 52) & 0x7ff);
    const bool odd = (ea == 0 && (ua << 1) != 0) || (eb == 0 && (ub << 1) != 0) || ea == 0x7ff || eb == 0x7ff;
    const unsigned emax = __reduce_max_sync(0xffffffffu, (unsigned)max(ea, eb));
    if (__any_sync(0xffffffffu, odd) || emax == 0) return warp_sum(a + b);
    auto fix = [emax](unsigned long long u, int e) -> long long {
        if (e == 0) return 0;  // +-0
        const long long mant = (long long)((u & 0xFFFFFFFFFFFFFull) | (1ull << 52));
        const int sh = e - (int)emax + 4;  // at most 4
        long long t = 0;
        if (sh >= 0) t = mant << sh;
        else if (sh > -60) t = (mant + (1ll << (-sh - 1))) >> (-sh);
        return (u >> 63) ? -t : t;
    };
    long long t = fix(ua, ea) + fix(ub, eb);
    // the exact sum by three independent reduxes (22, 22 and the signed upper bits);
    // a five-level butterfly of 64-bit shuffles has the same value 0.2 us later
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)t & 0x3fffffu);
    const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)(t >> 22) & 0x3fffffu);
    const int hi = __reduce_add_sync(0xffffffffu, (int)(t >> 44));
    t = (long long)lo + ((long long)mid << 22) + (long long)((unsigned long long)(long long)hi << 44);
    return t == 0 ? 0.0 : ll_scaled(t, (int)emax - 1079);
}

// order-preserving integer image of a float (no NaN; -0 and +0 share one key)
__device__ __forceinline__ int fkey(float x) {
    int b = __float_as_int(x);
    if ((b & 0x7fffffff) == 0) b = 0;
    return b >= 0 ? b : (b ^ 0x7fffffff);
}

__device__ PricePatch pivot_patch(const SlotMoves& v, int q, int leave, bool push, int tabu_until) {
    PricePatch p = no_patch();
    p.basic_j = q;
    p.free_j = leave;
    if (push) { p.tabu_j = leave; p.tabu_until = tabu_until; }
    // the slot -> row entries that differ from the current map, in the
    // precedence order of moved_slot_row
    if (v.ent >= 0) {
        p.sp_slot[p.nsp] = v.te; p.sp_row[p.nsp] = v.w; ++p.nsp;
        p.sp_slot[p.nsp] = v.k1 - 1; p.sp_row[p.nsp] = v.ent; ++p.nsp;
    }
    if (v.join >= 0) {
        p.sp_slot[p.nsp] = v.k0; p.sp_row[p.nsp] = v.join; ++p.nsp;
        p.sp_slot[p.nsp] = v.tl; p.sp_row[p.nsp] = v.u; ++p.nsp;
    }
    return p;
}

// The CTA's ratio-test record from its rows' (alpha', bbar, variable): its
// smallest ratio, and its best row and tie count under that ratio's tie
// threshold (one warp, one lane per row).  On this chip every FP64
// instruction holds a scheduler's FP64 pipe for 64 cycles whatever the number
// of active lanes, so the ratios of 32 rows are formed by one warp-wide
// division; the minimum, the tie band and the largest pivot are taken on
// integer keys, across the warp by redux (a dependent shuffle costs more).
__device__ void row_record(const Params& P, int owned, bool bland, const double* ral, const double* rb,
                           const int* rvar, RowRec* out) {
    const int lane = threadIdx.x & 31;
    const int G = gridDim.x;
    const long long kpiv = dkey(P.tol_piv), kbig = dkey(DBL_MAX);
    // pass 1: ratios and their minimum
    long long kmin_l = kbig;
    double th0 = DBL_MAX;  // the first 32 rows' ratios, kept for pass 2
    for (int l0 = 0; l0 < owned; l0 += 32) {
        const int l = l0 + lane;
        const double al = l < owned ? ral[l] : 0.0;
        const bool ok = l < owned && dkey(al) > kpiv;
        const double th = ok ? rb[l] / al : DBL_MAX;
        if (l0 == 0) th0 = th;
        kmin_l = min(kmin_l, dkey(th));
    }
    const long long kmin = warp_min_key(kmin_l);
    const double tmin = kdouble(kmin);
    // max(1, |tmin|) by its bits: FP64 compares would cost the pipe as much as the FMA
    const long long mag = __double_as_longlong(tmin) & 0x7fffffffffffffffLL;
    const double scale = __longlong_as_double(max(mag, __double_as_longlong(1.0)));
    const double thr = kmin == kbig ? DBL_MAX : tmin + P.tol_tie * scale;
    const long long kthr = dkey(thr);
    // pass 2: the tie band, its size and best row (largest pivot, then smallest
    // basic index; Bland: smallest basic index), lane by lane
    long long ka = LLONG_MIN;
    int bvar = INT_MAX, bl = -1, cnt = 0;
    double bth = 0.0;
    if (kmin != kbig) {
        for (int l0 = 0; l0 < owned; l0 += 32) {
            const int l = l0 + lane;
            const double al = l < owned ? ral[l] : 0.0;
            const long long kal = dkey(al);
            const bool ok = l < owned && kal > kpiv;
            const double th = l0 == 0 ? th0 : (ok ? rb[l] / al : DBL_MAX);
            if (ok && dkey(th) <= kthr) {
                cnt++;
                const int v = rvar[l];
                const bool better = bl < 0 || (bland ? v < bvar : (kal > ka || (kal == ka && v < bvar)));
                if (better) { ka = kal; bvar = v; bl = l; bth = th; }
            }
        }
    }
    const int tot = __reduce_add_sync(0xffffffffu, cnt);
    long long kbest;
    const int win = bland ? warp_argmin_index(bvar, bl >= 0)
                          : warp_argmax_key(ka, bvar, bl >= 0, kbest);
    if (win < 0 ? lane == 0 : lane == win) {
        RowRec rp;
        rp.tmin = kmin; rp.thr = kthr;
        rp.a = win >= 0 ? kdouble(ka) : 0.0;
        rp.th = win >= 0 ? bth : 0.0;
        rp.var = win >= 0 ? bvar : 0; rp.row = win >= 0 ? (int)blockIdx.x + G * bl : -1;
        rp.cnt = tot; rp.pad_ = 0;
        *out = rp;
    }
}

}  // namespace
}  // namespace lpgb
