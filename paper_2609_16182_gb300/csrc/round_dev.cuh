// round_dev.cuh -- the per-row and per-column work of one presolve round:
// S1 activities, S2 row classes, S3 implied bounds (fused, per row), S3'/S4
// bound finalisation and fixing (per column), S5 parallel rows (per row).
// Included by the round kernels (k_round.cu), which launch it over a whole
// arena, and by the fused batch kernel (k_batch.cu), which runs it for one
// LP per thread block: both evaluate every row and column the same way, so
// an LP gets the same bits from either.
#pragma once
#include <cooperative_groups.h>

#include "lpp_dev.cuh"

namespace lpp {

namespace {

namespace cg = cooperative_groups;

// warp-aggregated counter: one atomic per warp with something to add, no
// barrier (the warps of a block end on their own); the whole warp must call it
__device__ __forceinline__ void warp_add(int32_t v, int32_t *dst) {
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(dst, v);
}

// appends v to list[*cnt ...] with one atomic per group of converged threads
__device__ __forceinline__ void coalesced_append(int32_t v, int32_t *cnt, int32_t *list) {
    cg::coalesced_group g = cg::coalesced_threads();
    int32_t base = 0;
    if (g.thread_rank() == 0) base = atomicAdd(cnt, (int32_t)g.size());
    base = g.shfl(base, 0);
    list[base + (int32_t)g.thread_rank()] = v;
}

// column j received a candidate: list it once per round for S3'
// (not needed when S3' checks every column this round)
__device__ __forceinline__ void touch_col(const Ctx &C, int32_t j) {
    if (!C.list_touched) {
        // a first round lists nothing (S3' runs on every column); with dual
        // records the flag alone lets the bound-source pass skip the columns
        // without a candidate
        if (C.dual_rec && C.ctouch[j] == 0u) C.ctouch[j] = 1u;
        return;
    }
    if (C.ctouch[j] == 0u && atomicExch(&C.ctouch[j], 1u) == 0u) coalesced_append(j, C.tl_cnt, C.tl_list);
}

// exact sign tests of a double on its bit pattern (integer pipes):
// s < 0 <=> negative and not -0;  s > 0 <=> positive bits, not +0
__device__ __forceinline__ bool lt0(double s) {
    return dbits(s) < 0 && dbits(s) != (long long)0x8000000000000000ULL;
}
__device__ __forceinline__ bool gt0(double s) { return dbits(s) > 0; }

// ------------------------------------------------ S3 filter in single precision
// An entry's implied bound can be accepted only if the row's slack is below
// what the entry alone can span:  with x1 = dU + a bmin the sign tests of
// pass_upper / pass_lower read  slack < |a| (u - l) - |a| bound_tol max(1, |old|)
// in every case of sign and side (slack = U - smin or smax - L; an infinite
// old bound or own term makes the span infinite).  The filter compares a lower
// estimate of the slack with an upper estimate of |a| (u - l), taken from the
// high words of the doubles in single precision, so it drops only entries
// whose exact test fails: each estimate is off by at least 2^-21 of its
// terms, the roundings of the exact test by at most a few 2^-53 of the same
// terms.  It replaces, for nearly every entry, a queue trip with two FP64
// instructions and two gathers by a few single-precision ones.
// High words (sign bit cleared) to single precision: above / below |x|, by
// at least 2^-21 |x|; then the same for signed values.  Above is infinity from
// 2^128 (1 - 2^-20) on, where the sum below would run past infinity's bits.
__device__ __forceinline__ float f32_above(uint32_t hi) {
    if (hi < (897u << 20)) return __uint_as_float(0x01000000u);  // |x| < 2^-126: 2^-125
    if (hi >= (1151u << 20) - 2u) return __uint_as_float(0x7f800000u);
    return __uint_as_float((hi << 3) - 0xc0000000u + 16u);
}
__device__ __forceinline__ float f32_below(uint32_t hi) {
    if (hi < (898u << 20)) return 0.0f;
    if (hi >= (1151u << 20)) return __uint_as_float(0x7f7fffffu);
    return __uint_as_float((hi << 3) - 0xc0000000u - 16u);
}
__device__ __forceinline__ uint32_t hi_word(double x) { return (uint32_t)((unsigned long long)dbits(x) >> 32); }
__device__ __forceinline__ float f32_hi(double x) {
    const uint32_t h = hi_word(x), m = h & 0x7fffffffu;
    return (int32_t)h < 0 ? -f32_below(m) : f32_above(m);
}
__device__ __forceinline__ float f32_lo(double x) {
    const uint32_t h = hi_word(x), m = h & 0x7fffffffu;
    return (int32_t)h < 0 ? -f32_above(m) : f32_below(m);
}
__device__ __forceinline__ float f32_mag(double x) { return f32_above(hi_word(x) & 0x7fffffffu); }

// Implied upper bound x/a on column j (from a*x_j <= x with a > 0, or
// a*x_j >= x with a < 0).  Accepted iff (uold = +inf or x/a < thr) and
// |x/a| <= max_implied, thr = uold - bound_tol*max(1,|uold|) (one rounding).
// Both tests are decided exactly on the real quotient by the sign of one
// fused multiply-add; the cap is tested only for candidates that pass.
// A candidate that cannot lower the column's current minimum cur (x/a >= cur)
// would not change the result: it is dropped by the same test, made against
// min(cur, thr), and skips the divide.  pass_upper makes the sign test (e: cur,
// encoded); apply_cand the cap, the divide and the atomic.
__device__ __forceinline__ bool pass_upper(const Ctx &C, unsigned long long e, double x, double a, double uold) {
    // x/a must lie below both cur and thr: one test against min(cur, thr),
    // taken on the order-preserving encoding (integer pipes)
    if (is_fin(uold)) {
        const unsigned long long et = enc_dbl(fma(-C.bound_tol, max1abs(uold), uold));
        e = et < e ? et : e;
    }
    if (e == kEncPosInf) return true;
    const double s = fma(-dec_dbl(e), a, x);
    return is_neg(a) ? gt0(s) : lt0(s);
}
// Implied lower bound x/a: accepted iff (lold = -inf or x/a > thr) and
// |x/a| <= max_implied, thr = lold + bound_tol*max(1,|lold|); a candidate
// that cannot raise the current maximum is dropped with it.
__device__ __forceinline__ bool pass_lower(const Ctx &C, unsigned long long e, double x, double a, double lold) {
    if (is_fin(lold)) {
        const unsigned long long et = enc_dbl(fma(C.bound_tol, max1abs(lold), lold));
        e = et > e ? et : e;
    }
    if (e == kEncNegInf) return true;
    const double s = fma(-dec_dbl(e), a, x);
    return is_neg(a) ? lt0(s) : gt0(s);
}

// The bound x / a, with one zero: of two candidates -0 and +0 the second does not
// improve on the first and is dropped, so their order would decide the sign.
__device__ __forceinline__ double bound_value(double x, double a) {
    const double v = x / a;
    return (dbits(v) & 0x7fffffffffffffffLL) == 0 ? 0.0 : v;
}

// candidate kinds: implied bounds (capped) and singleton-row bounds (not)
enum : int32_t { CQ_UPPER = 0, CQ_LOWER = 1, CQ_SING_UPPER = 2, CQ_SING_LOWER = 3 };  // bit 0: a lower bound

// the value x/a enters column j's candidates; ec: the side's candidate as read
// before (one that x/a does not improve on stands, whatever came since)
__device__ __forceinline__ void apply_cand(const Ctx &C, int32_t j, double x, double a, int32_t kind,
                                           unsigned long long ec) {
    // |x / a| <= max_implied, exactly where single precision does not decide
    if (kind < CQ_SING_UPPER) {
        const float cap = __fmul_rd(f32_below(hi_word(C.max_implied)), f32_below(hi_word(a) & 0x7fffffffu));
        if (!(f32_mag(x) <= cap) && gt0(fma(-C.max_implied, fabs(a), fabs(x)))) return;
    }
    const double v = bound_value(x, a);
    if (!is_fin(v)) return;
    const unsigned long long e = enc_dbl(v);
    if (kind == CQ_UPPER || kind == CQ_SING_UPPER) {
        if (e < ec) atomicMin(&C.cand_u[j], e);
    } else if (e > ec) {
        atomicMax(&C.cand_l[j], e);
    }
    touch_col(C, j);
}

// above |a| (u - l)
__device__ __forceinline__ float entry_span(double a, double2 b) {
    const float w = __fsub_ru(f32_hi(b.y), f32_lo(b.x));
    return __fmul_ru(f32_mag(a), w > 0.0f ? w : 0.0f);
}
// below the slack hi - lo of a row side
__device__ __forceinline__ float slack_below(double hi, double lo) { return __fsub_rd(f32_lo(hi), f32_hi(lo)); }
// may the exact test pass (a NaN slack or span, 0 times infinity, passes)
__device__ __forceinline__ bool span_passes(float slack, float span) { return !(slack >= span); }

// one entry that passed the filter: the exact test of one of its sides.
// flags: the candidate kind, | 4 if the entry's own term is finite (residual
// = slack + a * bound, else the slack itself), | 8 for the lhs side
enum : int32_t { CQ_OWN = 4, CQ_LHS = 8 };
// First against the column's current candidate cur in single precision: x / a
// improves on it only if  s + |a| (l - cur) < 0  (an upper bound; s the
// positive slack, l the own term's bound, 0 if infinite) or  s + |a| (cur - u)
// < 0  (a lower bound).  Most entries of a column that many rows hold fail
// here, without an FP64 instruction.
__device__ __forceinline__ void test_and_apply(const Ctx &C, double a, double slack, int32_t j, int32_t flags) {
    const int32_t kind = flags & 3;
    const bool upper = (kind & 1) == 0;
    const unsigned long long ec = *((volatile unsigned long long *)(upper ? &C.cand_u[j] : &C.cand_l[j]));
    double x = slack;
    if (kind < CQ_SING_UPPER) {
        const double2 b = C.lu[j];
        const bool own = flags & CQ_OWN;
        const double bnd = own ? (upper ? b.x : b.y) : 0.0;
        if (ec != (upper ? kEncPosInf : kEncNegInf)) {
            const double cur = dec_dbl(ec);
            const float d = upper ? __fsub_rd(f32_lo(bnd), f32_hi(cur)) : __fsub_rd(f32_lo(cur), f32_hi(bnd));
            const uint32_t ma = hi_word(a) & 0x7fffffffu;
            const float s = (flags & CQ_LHS) ? -f32_hi(slack) : f32_lo(slack);
            if (__fadd_rd(s, __fmul_rd(d >= 0.0f ? f32_below(ma) : f32_above(ma), d)) >= 0.0f) return;
        }
        if (own) x = fma(a, bnd, slack);
        if (!(upper ? pass_upper(C, ec, x, a, b.y) : pass_lower(C, ec, x, a, b.x))) return;
    }
    apply_cand(C, j, x, a, kind, ec);
}

// flags of an entry side: the rhs side bounds x_j from above for a > 0, the
// lhs side for a < 0
__device__ __forceinline__ int32_t side_flags(bool neg, bool lhs, bool own_finite) {
    return ((neg != lhs) ? CQ_LOWER : CQ_UPPER) | (own_finite ? CQ_OWN : 0) | (lhs ? CQ_LHS : 0);
}

// one entry, its candidates applied at once (long rows: few of them tighten)
__device__ __forceinline__ void tighten_entry(const Ctx &C, int32_t j, double a, bool up_row, bool lo_row,
                                              double dU, double dL, float fU, float fL, int nmin, int nmax,
                                              int32_t &tested) {
    const double2 b = C.lu[j];
    const bool neg = is_neg(a);
    const bool fmn = is_fin(neg ? b.y : b.x), fmx = is_fin(neg ? b.x : b.y);
    const bool w1 = up_row && (fmn ? nmin == 0 : nmin == 1), w2 = lo_row && (fmx ? nmax == 0 : nmax == 1);
    tested += (w1 ? 1 : 0) + (w2 ? 1 : 0);
    const float span = entry_span(a, b);
    if (w1 && span_passes(fU, span)) test_and_apply(C, a, dU, j, side_flags(neg, false, fmn));
    if (w2 && span_passes(fL, span)) test_and_apply(C, a, dL, j, side_flags(neg, true, fmx));
}

// Per-warp queue of the entry sides that passed the filter (and of the
// singleton rows' bounds).  The exact test, the divide, the cap and the
// atomic then run 32 at a time, one per lane, instead of on the one or two
// lanes of a warp that have one in a step: on GB300 an FP64 instruction
// costs the pipe the same however many lanes are active.  Every lane of the
// warp must call cq_push / cq_flush.  1.5 KB per warp: shared memory is taken
// from the L1, whose lines hold the bound gathers in flight.
struct CandQueue {
    double *a, *slack;
    int32_t *j, *flags;
    int32_t n;  // items held, the same in every lane
};
constexpr int kQueueCap = 64;

// the first cnt <= 32 items, one per lane; the rest move up
__device__ __forceinline__ void cq_run(const Ctx &C, CandQueue &q, int32_t cnt) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    const bool have = lane < cnt;
    const double ia = have ? q.a[lane] : 0.0, is = have ? q.slack[lane] : 0.0;
    const int32_t ij = have ? q.j[lane] : 0, ifl = have ? q.flags[lane] : 0;
    const int32_t rest = q.n - cnt;
    double ra = 0.0, rs = 0.0;
    int32_t rj = 0, rf = 0;
    if (lane < rest) {
        ra = q.a[32 + lane];
        rs = q.slack[32 + lane];
        rj = q.j[32 + lane];
        rf = q.flags[32 + lane];
    }
    __syncwarp();
    if (lane < rest) {
        q.a[lane] = ra;
        q.slack[lane] = rs;
        q.j[lane] = rj;
        q.flags[lane] = rf;
    }
    __syncwarp();
    q.n = rest;
    if (have) test_and_apply(C, ia, is, ij, ifl);
}

__device__ __forceinline__ void cq_push(const Ctx &C, CandQueue &q, bool want, double a, double slack, int32_t j,
                                        int32_t flags) {
    const unsigned b = __ballot_sync(0xffffffffu, want);
    if (b == 0u) return;
    const int lane = threadIdx.x & 31;
    if (want) {
        const int32_t p = q.n + __popc(b & ((1u << lane) - 1u));
        q.a[p] = a;
        q.slack[p] = slack;
        q.j[p] = j;
        q.flags[p] = flags;
    }
    q.n += __popc(b);
    if (q.n < 32) return;
    cq_run(C, q, 32);
}

__device__ __forceinline__ void cq_flush(const Ctx &C, CandQueue &q) {
    if (q.n > 0) cq_run(C, q, q.n);
}

// S2: class of a row from its activities, first match wins: infeasible
// sides, infeasible activity, empty, redundant, singleton.  Returns false if
// the row proves the LP infeasible.
// Order-preserving integer key of a non-NaN double (-0 and +0 equal): the
// row tests compare keys on the integer pipes instead of the FP64 pipe.
__device__ __forceinline__ long long dkey(double x) {
    const long long b = dbits(x);
    if ((b & 0x7fffffffffffffffLL) == 0) return 0;
    return b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
}

// The FP64 sums U + delta(U), L - delta(L) (delta(x) = feas_tol max(1, |x|))
// are formed only where the comparison with U or L itself, or their
// single-precision estimates, does not decide: a row's classification then
// costs no FP64 instruction in nearly every case.
__device__ __forceinline__ bool classify(const Ctx &C, double Lv, double Uv, int32_t len, double smin, double smax,
                                         int nmin, int nmax, uint8_t &kind) {
    const double ft = C.feas_tol;
    const bool Lf = is_fin(Lv), Uf = is_fin(Uv);
    kind = RK_KEPT;
    const long long kL = dkey(Lv), kU = dkey(Uv), ksmin = dkey(smin), ksmax = dkey(smax);
    if (Lf && Uf && kL > kU) {
        const double mL = max1abs(Lv), mU = max1abs(Uv);  // >= 1: their bits order like their values
        if (dkey(Lv - Uv) > dkey(ft * (dbits(mL) > dbits(mU) ? mL : mU))) return false;
    }
    if (nmin == 0 && Uf && ksmin > kU && ksmin > dkey(Uv + ft * max1abs(Uv))) return false;
    if (nmax == 0 && Lf && ksmax < kL && ksmax < dkey(Lv - ft * max1abs(Lv))) return false;
    if (len == 0) {
        kind = RK_EMPTY;
        return true;
    }
    bool lo_ok = !Lf;
    if (Lf && nmin == 0) {
        lo_ok = ksmin >= kL;
        if (!lo_ok) {
            const float d = __fmul_ru(f32_mag(ft), f32_mag(max1abs(Lv)));
            if (!(f32_hi(smin) < __fsub_rd(f32_lo(Lv), d))) lo_ok = ksmin >= dkey(Lv - ft * max1abs(Lv));
        }
    }
    if (lo_ok) {
        bool hi_ok = !Uf;
        if (Uf && nmax == 0) {
            hi_ok = ksmax <= kU;
            if (!hi_ok) {
                const float d = __fmul_ru(f32_mag(ft), f32_mag(max1abs(Uv)));
                if (!(f32_lo(smax) > __fadd_ru(f32_hi(Uv), d))) hi_ok = ksmax <= dkey(Uv + ft * max1abs(Uv));
            }
        }
        if (hi_ok) {
            kind = RK_REDUNDANT;
            return true;
        }
    }
    if (len == 1) kind = RK_SINGLETON;
    return true;
}


// writes the row's S1/S2 results and records (a singleton row's bounds L/a,
// U/a are the caller's to apply)
__device__ __forceinline__ int32_t finish_row(const Ctx &C, int32_t i, int32_t beg, int32_t len, double Lv,
                                              double Uv, double smin, double smax, int nmin, int nmax,
                                              bool rehash, unsigned long long h, uint8_t &kind) {
    const bool ok = classify(C, Lv, Uv, len, smin, smax, nmin, nmax, kind);
    C.act[i] = make_double2(smin, smax);
    C.ninf[i] = make_int2(nmin, nmax);
    if (rehash) C.hrow[i] = h;  // else the key stands: the row's entries did not change
    const int32_t lp = lp_of_row(C, i);
    if (!ok) {
        atomicMin(&C.verdict[lp * V_SLOTS + V_S2_ROW], C.rmap[i]);
        kind = RK_KEPT;
        C.rkind[i] = RK_KEPT;
        return 0;
    }
    C.rkind[i] = kind;
    if (kind == RK_KEPT) return 0;
    const int32_t o = C.rmap[i];
    C.rec_rk[o] = kind;
    C.rec_rr[o] = lp_round(C, lp);
    mark_lp_changed(C, lp);
    if (kind == RK_SINGLETON) {
        C.rec_ra[o] = C.cmap[C.A.idx[beg]];
        C.rec_rv[o] = C.A.val[beg];
    } else {
        C.rec_ra[o] = -1;
        C.rec_rv[o] = 0.0;
    }
    return 1;
}

// Queues the entry sides of a lane in todo: bit c the rhs side of entry k0 + c
// stride, bit 16 + c its lhs side (the whole warp together).
__device__ __forceinline__ void push_sides(const Ctx &C, CandQueue &q, unsigned todo, int32_t k0, int32_t stride,
                                           double dU, double dL, unsigned imin, unsigned imax, bool sing) {
    const int T = (int)__reduce_max_sync(0xffffffffu, (unsigned)__popc(todo));
    for (int t = 0; t < T; t++) {
        const bool want = todo != 0u;
        const int bit = want ? __ffs(todo) - 1 : 0;
        todo &= todo - 1u;
        const bool lhs = bit >= 16;
        int32_t j = 0;
        double a = 0.0;
        if (want) {
            const int32_t k = k0 + (bit & 15) * stride;
            j = C.A.idx[k];
            a = C.A.val[k];
        }
        const bool own = !(((lhs ? imax : imin) >> (bit & 15)) & 1u);
        int32_t f = side_flags(is_neg(a), lhs, own);
        if (sing) f = (f & 1) | CQ_SING_UPPER;  // the row's side itself, untested
        cq_push(C, q, want, a, lhs ? dL : dU, j, f);
    }
}

// S3 over the entries k0, k0 + stride, .. below end of a lane (none if end <=
// k0), T steps for the whole warp, four entries in flight: the entry sides
// that pass the filter are queued.
__device__ __forceinline__ void tighten_steps(const Ctx &C, CandQueue &q, int32_t T, int32_t k0, int32_t stride,
                                              int32_t end, bool up_row, bool lo_row, double dU, double dL, float fU,
                                              float fL, int nmin, int nmax, int32_t &tested) {
    for (int32_t it = 0; it < T; it += 4, k0 += 4 * stride) {
        int32_t j[4];
        double a[4];
        double2 b[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int32_t k = k0 + u * stride;
            j[u] = k < end ? C.A.idx[k] : -1;
            a[u] = k < end ? C.A.val[k] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 4; u++) b[u] = j[u] >= 0 ? C.lu[j[u]] : make_double2(0.0, 0.0);
        unsigned todo = 0, imin = 0, imax = 0;
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const bool neg = is_neg(a[u]), in = j[u] >= 0;
            const bool fmn = is_fin(neg ? b[u].y : b[u].x), fmx = is_fin(neg ? b[u].x : b[u].y);
            const bool w1 = in && up_row && (fmn ? nmin == 0 : nmin == 1);
            const bool w2 = in && lo_row && (fmx ? nmax == 0 : nmax == 1);
            tested += (w1 ? 1 : 0) + (w2 ? 1 : 0);
            const float span = entry_span(a[u], b[u]);
            imin |= (unsigned)!fmn << u;
            imax |= (unsigned)!fmx << u;
            todo |= (unsigned)(w1 && span_passes(fU, span)) << u | (unsigned)(w2 && span_passes(fL, span)) << (16 + u);
        }
        push_sides(C, q, todo, k0, stride, dU, dL, imin, imax, false);
    }
}

// ------------------------------------------------------- S1 + S2 + S3 groups
// Dirty flags of a row (rdirty): kEval, its activities must be taken again (a
// bound in it, its entries or its sides changed), kRekey, its S5 key (its
// entries changed, or the columns were renumbered).  A row without kEval has
// the same activities and class (kept) and yields the same implied bounds,
// which were then already applied or rejected.
enum : uint8_t { kEval = 1, kRekey = 2 };

// xor butterfly over W lanes, W at run time: every lane ends with the same bits
template <typename T>
__device__ __forceinline__ T lanes_sum(T v, int W, unsigned mask) {
    for (int o = W / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
    return v;
}

// bits 4 c + e to c + 4 e, in both halves
__device__ __forceinline__ unsigned transpose_4x4(unsigned x) {
    unsigned t = (x ^ (x >> 3)) & 0x0a0a0a0au;
    x ^= t ^ (t << 3);
    t = (x ^ (x >> 6)) & 0x00cc00ccu;
    return x ^ t ^ (t << 6);
}

// S1-S3 of row i by W lanes.  LONG: a warp (W = 32) per row of any length, S3
// walks the row again.  Else W = 1, 2 or 4 with at most 16 entries per lane,
// whose spans stay in registers for S3, so that S3 reads only the entries that
// pass the filter again.
template <bool LONG>
__device__ __forceinline__ void prop_row(const Ctx &C, int32_t i, bool valid, int W, int32_t &removed,
                                         int32_t &evaluated, int32_t &tested, CandQueue &q) {
    if constexpr (LONG) W = 32;
    const int wl = threadIdx.x & 31, lane = wl & (W - 1);
    const unsigned mask = LONG ? 0xffffffffu : ((1u << W) - 1u) << (wl & ~(W - 1));
    const uint8_t flag = valid ? C.rdirty[i] : 0;
    const bool act = flag & kEval, rehash = flag & kRekey;
    if (valid && !act && lane == 0) C.rkind[i] = RK_KEPT;
    int32_t beg = 0, end = 0;
    if (flag) {
        beg = C.A.ptr[i];
        end = C.A.ptr[i + 1];
    }
    const bool neg0 = rehash && end > beg ? is_neg(C.A.val[beg]) : false;
    double smin = 0.0, smax = 0.0;
    int nmin = 0, nmax = 0;
    unsigned long long h = 0;
    float span[LONG ? 1 : 16];
    unsigned imin = 0, imax = 0;  // entries with an infinite term
    // The lane's entries in steps of four, the tail of a step predicated: the
    // four bound gathers of a step overlap, and a warp whose lanes hold rows of
    // different lengths runs no separate remainder loop (which would issue
    // its FP64 work a second time for the lanes still in it).  A lone lane's sums
    // take the entries in the same order as a plain loop.
    // A lane of several (W = 2, 4) takes, in step c, the entries of residue class
    // lane + c W modulo 4 W, a chain each, added as a butterfly over 4 W lanes
    // adds them: the bits, and so the error, of 8 and 16 lanes per row.  (One
    // chain of a lane's 16 entries had up to 18 roundings where this has 7 or 8,
    // and a mean error 3 to 20% larger.)
    const int32_t es = !LONG && W > 1 ? 4 * W : W, cs = !LONG && W > 1 ? W : 4 * W;
    auto step = [&](int32_t k0, int c4) {
        int32_t jq[4];
        double aq[4];
        double2 bq[4];
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int32_t k = k0 + e * es;
            jq[e] = k < end ? C.A.idx[k] : 0;
            aq[e] = k < end ? C.A.val[k] : 0.0;
        }
#pragma unroll
        for (int e = 0; e < 4; e++) bq[e] = act && k0 + e * es < end ? C.lu[jq[e]] : make_double2(0.0, 0.0);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            if (k0 + e * es >= end) break;
            const double a = aq[e];
            const double2 b = bq[e];
            const bool neg = is_neg(a);
            const double bmin = neg ? b.y : b.x, bmax = neg ? b.x : b.y;
            const bool fmn = is_fin(bmin), fmx = is_fin(bmax);
            if (fmn) smin = fma(a, bmin, smin);
            else nmin++;
            if (fmx) smax = fma(a, bmax, smax);
            else nmax++;
            if constexpr (!LONG) {
                imin |= (unsigned)!fmn << (c4 + e);
                imax |= (unsigned)!fmx << (c4 + e);
                span[c4 + e] = entry_span(a, b);
            }
            if (rehash) h += entry_hash(jq[e], neg != neg0);
        }
    };
    if constexpr (LONG) {
        for (int32_t k0 = beg + lane; k0 < end; k0 += 4 * W) step(k0, 0);
    } else {
        double t0 = 0.0, t1 = 0.0, u0 = 0.0, u1 = 0.0;
#pragma unroll
        for (int c = 0; c < 4; c++) {
            if (beg + lane + c * cs < end) step(beg + lane + c * cs, 4 * c);
            if (W > 1) {  // the same W in the whole warp
                if (c == 0) {
                    t0 = smin;
                    t1 = smax;
                } else if (c == 1) {
                    u0 = smin;
                    u1 = smax;
                } else if (c == 2) {
                    t0 += smin;
                    t1 += smax;
                }
                if (c < 3) smin = smax = 0.0;
            }
        }
        if (W > 1) {
            smin = t0 + (u0 + smin);
            smax = t1 + (u1 + smax);
        }
    }
    if (W > 1) {  // the same W in the whole warp
        smin = lanes_sum(smin, W, mask);
        smax = lanes_sum(smax, W, mask);
        nmin = lanes_sum(nmin, W, mask);
        nmax = lanes_sum(nmax, W, mask);
        if (__any_sync(0xffffffffu, rehash)) h = lanes_sum(h, W, mask);
    }
    const int32_t len = end - beg;
    h += len_hash(len);
    if (rehash && !act && lane == 0) C.hrow[i] = h;
    bool up_row = false, lo_row = false;
    double Lv = 0.0, Uv = 0.0;
    int32_t kind = RK_KEPT;
    bool sing = false;
    if (act) {
        if (lane == 0) evaluated += len;
        Lv = C.L[i];
        Uv = C.U[i];
        if (lane == 0) {
            uint8_t k = RK_KEPT;
            removed += finish_row(C, i, beg, len, Lv, Uv, smin, smax, nmin, nmax, rehash, h, k);
            kind = k;
        }
        if (W > 1) kind = __shfl_sync(mask, kind, wl & ~(W - 1));
        if (kind == RK_KEPT && len >= 2) {
            up_row = is_fin(Uv) && nmin <= 1;
            lo_row = is_fin(Lv) && nmax <= 1;
        }
        sing = kind == RK_SINGLETON && lane == 0;
    }
    // S3 over the row's entries, in steps the whole warp takes together
    const float fU = slack_below(Uv, smin), fL = slack_below(smax, Lv);
    if constexpr (!LONG) {
        // a x_j <= U - (min activity of the others): every entry when no term
        // is infinite, the one infinite term alone when there is one
        // Bit 4 c + e: the entry of step c; with several lanes it is the lane's
        // (c + 4 e)th, and a transposition of the 4 x 4 bits puts them in order.
        const int nq = lane < len ? (len - lane + W - 1) / W : 0;
        const unsigned all = W > 1 ? transpose_4x4((1u << nq) - 1u) : (1u << nq) - 1u;
        const unsigned q1 = up_row ? (nmin == 0 ? all : imin) : 0u, q2 = lo_row ? (nmax == 0 ? all : imax) : 0u;
        tested += __popc(q1) + __popc(q2);
        unsigned todo = 0;
        if (q1 | q2) {
#pragma unroll
            for (int c = 0; c < 4; c++) {
                if (nq <= (W > 1 ? c : 4 * c)) break;
#pragma unroll
                for (int e = 4 * c; e < 4 * c + 4; e++)
                    todo |= (unsigned)span_passes(fU, span[e]) << e | (unsigned)span_passes(fL, span[e]) << (16 + e);
            }
            todo &= q1 | (q2 << 16);
        }
        if (W > 1 && todo) {
            todo = transpose_4x4(todo);
            imin = transpose_4x4(imin);
            imax = transpose_4x4(imax);
        }
        // a singleton row L <= a x_j <= U becomes the bounds L/a and U/a, always
        // applied (no threshold)
        if (sing) todo = (is_fin(Uv) ? 1u : 0u) | (is_fin(Lv) ? 1u << 16 : 0u);
        if (__any_sync(0xffffffffu, todo != 0u))  // the slacks are formed only when an entry needs them
            push_sides(C, q, todo, beg + lane, W, sing ? Uv : Uv - smin, sing ? Lv : Lv - smax, imin, imax, sing);
    } else {
        const int32_t trips = (up_row || lo_row) && lane < len ? (len - lane + W - 1) / W : 0;
        const int32_t T = (int32_t)__reduce_max_sync(0xffffffffu, (unsigned)trips);
        tighten_steps(C, q, T, beg + lane, W, (up_row || lo_row) ? end : beg, up_row, lo_row, Uv - smin, Lv - smax, fU,
                      fL, nmin, nmax, tested);
    }
}

// Lanes per row in S1-S3: a lane holds up to 16 entries (rows up to 16, 32 and
// 64 entries: 1, 2, 4 lanes), longer rows take a warp.  Fewer lanes per row
// cost fewer butterfly steps, each two FP64 instructions: 8 lanes for 17 to
// 32 entries cost 3.5 FP64 warp instructions a row, 2 lanes with four chains
// each 2.5 (one chain each 2.1, but off by more: the relaxation of 500 k rows
// takes 5.55 ms for 5.42).
__host__ __device__ __forceinline__ int prop_lanes(int c) { return c <= 2 ? 1 : (c == 5 ? 32 : 1 << (c - 2)); }

// ------------------------------------------------- S3' finalise + S4 fixing
// S3' + S4 on column j: apply the accepted candidates, check and snap the
// bounds, fix the column if l == u.  Adds to the counts changed, fixed and
// chg_nnz (a thread may finalise several columns); a changed short column is
// listed for the dirty-row marking.
__device__ __forceinline__ void colfin_one(const Ctx &C, int32_t j, bool full, int32_t &changed, int32_t &fixed,
                                           int32_t &chg_nnz) {
    const unsigned long long el = C.cand_l[j], eu = C.cand_u[j];
    const bool has = el != kEncNegInf || eu != kEncPosInf;
    uint8_t kind = CK_KEPT;
    uint8_t chg = 0;
    const int32_t lp = lp_of_col(C, j);
    if (has || (full && lp_round(C, lp) == 1)) {
        if (has) {
            C.cand_l[j] = kEncNegInf;
            C.cand_u[j] = kEncPosInf;
        }
        const double2 b = C.lu[j];
        double nl = b.x, nu = b.y;
        if (has) {
            const double dl = dec_dbl(el), du = dec_dbl(eu);
            if (dl > nl) nl = dl;
            if (du < nu) nu = du;
        }
        bool bad = false;
        if (is_fin(nl) && is_fin(nu)) {
            const double d = C.feas_tol * fmax(1.0, fmax(fabs(nl), fabs(nu)));
            if (nl - nu > d) {
                bad = true;
            } else if (nl != nu && fabs(nl - nu) <= d) {
                const double mid = 0.5 * (nl + nu);
                nl = mid;
                nu = mid;
            }
        }
        if (bad) {
            atomicMin(&C.verdict[lp * V_SLOTS + V_S3_COL], C.cmap[j]);
        } else {
            if (C.dual_rec && has) {
                // a side a candidate moved takes that candidate's row (a side
                // moved only by the snap keeps its earlier source)
                const int2 src = C.bsrc[j];
                const double dl = dec_dbl(el), du = dec_dbl(eu);
                if (dl > b.x || du < b.y) {
                    int4 r = C.rec_bs[C.cmap[j]];
                    if (dl > b.x) {
                        r.x = src.x != INT32_MAX ? src.x : -2;  // -2: no row matched (never expected)
                        r.y = lp_round(C, lp);
                    }
                    if (du < b.y) {
                        r.z = src.y != INT32_MAX ? src.y : -2;
                        r.w = lp_round(C, lp);
                    }
                    C.rec_bs[C.cmap[j]] = r;
                }
                C.bsrc[j] = make_int2(INT32_MAX, INT32_MAX);
            }
            if (nl != b.x || nu != b.y) {
                C.lu[j] = make_double2(nl, nu);
                changed++;
                chg = 1;
                mark_lp_changed(C, lp);
            }
            if (nl == nu) {
                kind = CK_FIXED;
                fixed++;
                C.fixv[j] = nl;
                const int32_t o = C.cmap[j];
                C.rec_ck[o] = CK_FIXED;
                C.rec_cr[o] = lp_round(C, lp);
                C.rec_cv[o] = nl;
                mark_lp_changed(C, lp);
            }
        }
    }
    C.ckind[j] = kind;
    C.cchg[j] = C.in_place && kind != CK_KEPT ? (uint8_t)(chg | CS_LEAVES) : chg;
    C.ctouch[j] = 0u;
    if (chg && !C.in_place) {
        // the column's length decides list or chunks for the dirty-row marking
        // and counts towards the marking threshold
        const int32_t len = C.T.ptr[j + 1] - C.T.ptr[j];
        if (len < kLongMin) coalesced_append(j, C.cl_cnt, C.cl_list);
        chg_nnz += len;
    }
}

// ------------------------------------------------------------ S5 parallel rows
// Inserts row i into the hash table of capacity cap (a power of two) and
// elects the leader of its key: the first equality row, else the first row
// (Sec. 3.2), by atomicMin on (is_ineq, row).  Returns the slot, -1 if the
// table is full (an internal error: the capacity is at least twice the rows).
__device__ __forceinline__ int32_t s5_insert_row(const Ctx &C, int32_t i, uint32_t cap, uint32_t off = 0) {
    unsigned long long key = C.hrow[i];
    if (key == 0) key = 1;
    uint32_t sl = (uint32_t)(key ^ (key >> 32)) & (cap - 1u);
    for (uint32_t probe = 0; probe < cap; probe++) {
        const unsigned long long prev = atomicCAS(&C.tkey[off + sl], 0ULL, key);
        if (prev == 0ULL || prev == key) {
            const double Lv = C.L[i], Uv = C.U[i];
            const bool eq = is_fin(Lv) && Lv == Uv;
            const unsigned long long code = ((unsigned long long)(eq ? 0u : 1u) << 32) | (uint32_t)i;
            atomicMin(&C.tlead[off + sl], code);
            return (int32_t)(off + sl);
        }
        sl = (sl + 1u) & (cap - 1u);
    }
    atomicOr(&C.st->err, 1);
    return -1;
}

// merge a parallel follower i (row = lam * leader) into its leader li
__device__ __forceinline__ void s5_accept(const Ctx &C, int32_t i, int32_t li, double lam) {
    C.rkind[i] = RK_PARALLEL;
    const int32_t o = C.rmap[i];
    const int32_t lp = lp_of_row(C, i);
    C.rec_rk[o] = RK_PARALLEL;
    C.rec_rr[o] = lp_round(C, lp);
    C.rec_ra[o] = C.rmap[li];
    C.rec_rv[o] = lam;
    mark_lp_changed(C, lp);
    const double Lj = C.L[i], Uj = C.U[i];
    double lo, hi;
    if (!is_neg(lam)) {
        lo = is_fin(Lj) ? Lj / lam : ninf_();
        hi = is_fin(Uj) ? Uj / lam : pinf();
    } else {
        lo = is_fin(Uj) ? Uj / lam : ninf_();
        hi = is_fin(Lj) ? Lj / lam : pinf();
    }
    if (is_fin(lo)) atomic_max_dbl(&C.mL[li], lo);
    if (is_fin(hi)) atomic_min_dbl(&C.mU[li], hi);
    C.hasf[li] = 1;
}

template <int W>
__device__ __forceinline__ bool match_group(const Ctx &C, int32_t i, bool valid, int32_t &removed,
                                            int32_t &unmatched) {
    const unsigned mask = group_mask<W>();
    const int lane = threadIdx.x & (W - 1);
    bool act = valid && C.rwork[i] == 1;
    int32_t li = -1;
    if (act) {
        li = (int32_t)(uint32_t)(C.tlead[C.rslot[i]] & 0xffffffffULL);
        if (li == i) act = false;  // the leader itself
    }
    // every lane of a group sees the same `act`
    int32_t bi = 0, bl = 0, len = 0;
    bool ok = false;
    double lam = 0.0;
    if (act) {
        bi = C.A.ptr[i];
        bl = C.A.ptr[li];
        len = C.A.ptr[i + 1] - bi;
        ok = (C.A.ptr[li + 1] - bl) == len;
        lam = C.A.val[bi] / C.A.val[bl];
    }
    if (ok) {
        for (int32_t k = lane; k < len; k += W) {
            const double ai = C.A.val[bi + k], al = C.A.val[bl + k];
            const double la = lam * al;
            const bool same = C.A.idx[bi + k] == C.A.idx[bl + k] &&
                              fabs(ai - la) <= C.par_tol * fmax(fabs(ai), fabs(la));
            if (!same) ok = false;
        }
    }
    // all lanes of the group agree on `ok`
    const unsigned bal = __ballot_sync(mask, !ok);
    const unsigned mine = group_bits<W>(bal);
    ok = act && mine == 0u;
    if (valid && lane == 0) {
        if (ok) {
            s5_accept(C, i, li, lam);
            C.rwork[i] = 0;
            removed++;
        } else if (act) {
            C.rwork[i] = 2;
            unmatched++;
        } else {
            C.rwork[i] = 0;
        }
    }
    return valid && lane == 0 && act && !ok;
}

// table capacity of a later pass over n listed rows: the power of two >= 2 n, at most C.tcap
__device__ __forceinline__ uint32_t s5_tail_cap(const Ctx &C, int32_t n) {
    uint32_t cap = 1;
    while (cap < 2u * (uint32_t)n && cap < (uint32_t)C.tcap) cap <<= 1;
    return cap;
}

// Later-pass match of entry t of a list of n rows (t >= n: no row): row i
// against the leader of its slot; rows longer than 32 entries are checked
// by the whole warp in turn, so every lane of the warp must call it.
// removed / left: the row merged, or left unmatched for the next pass.
__device__ __forceinline__ void s5_tail_match_one(const Ctx &C, const int32_t *list, int32_t n, int32_t t,
                                                  int32_t &removed, bool &left, int32_t &i) {
    removed = 0;
    left = false;
    i = -1;
    const int lane = threadIdx.x & 31;
    bool act = false, ok = false;
    int32_t li = -1, bi = 0, bl = 0, len = 0;
    double lam = 0.0;
    if (t < n) {
        // the list, the slots and the leaders change from pass to pass, also
        // within one launch (grid-wide passes): read at L2, never from L1
        i = __ldcg(list + t);
        const int32_t sl = __ldcg(C.rslot + i);
        act = sl >= 0;
        if (act) {
            li = (int32_t)(uint32_t)(__ldcg(C.tlead + sl) & 0xffffffffULL);
            if (li == i) act = false;  // the leader itself
        }
        if (act) {
            bi = C.A.ptr[i];
            bl = C.A.ptr[li];
            len = C.A.ptr[i + 1] - bi;
            ok = (C.A.ptr[li + 1] - bl) == len;
            lam = C.A.val[bi] / C.A.val[bl];
        }
    }
    if (ok && len <= 32) {
        for (int32_t k = 0; k < len; k++) {
            const double ai = C.A.val[bi + k], la = lam * C.A.val[bl + k];
            if (!(C.A.idx[bi + k] == C.A.idx[bl + k] && fabs(ai - la) <= C.par_tol * fmax(fabs(ai), fabs(la)))) {
                ok = false;
                break;
            }
        }
    }
    unsigned todo = __ballot_sync(0xffffffffu, ok && len > 32);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1u;
        const int32_t sbi = __shfl_sync(0xffffffffu, bi, src), sbl = __shfl_sync(0xffffffffu, bl, src);
        const int32_t slen = __shfl_sync(0xffffffffu, len, src);
        const double slam = __shfl_sync(0xffffffffu, lam, src);
        bool sok = true;
        for (int32_t k = lane; k < slen; k += 32) {
            const double ai = C.A.val[sbi + k], la = slam * C.A.val[sbl + k];
            if (!(C.A.idx[sbi + k] == C.A.idx[sbl + k] && fabs(ai - la) <= C.par_tol * fmax(fabs(ai), fabs(la))))
                sok = false;
        }
        sok = __all_sync(0xffffffffu, sok) != 0;
        if (lane == src) ok = sok;
    }
    if (act && ok) {
        s5_accept(C, i, li, lam);
        removed = 1;
    } else if (act) {
        left = true;
    }
}

// leaders take the followers' sides: L = max(L, merged), U = min(U, merged);
// crossing by more than the tolerance is infeasible, nearly equal sides snap
// (row i has followers: hasf[i])
__device__ __forceinline__ void s5_leader_one(const Ctx &C, int32_t i) {
    C.hasf[i] = 0;
    const unsigned long long eL = C.mL[i], eU = C.mU[i];
    C.mL[i] = kEncNegInf;
    C.mU[i] = kEncPosInf;
    double nL = C.L[i], nU = C.U[i];
    const double mL = dec_dbl(eL), mU = dec_dbl(eU);
    if (mL > nL) nL = mL;
    if (mU < nU) nU = mU;
    if (is_fin(nL) && is_fin(nU)) {
        const double d = C.feas_tol * fmax(1.0, fmax(fabs(nL), fabs(nU)));
        if (nL - nU > d) {
            atomicMin(&C.verdict[lp_of_row(C, i) * V_SLOTS + V_S5_ROW], C.rmap[i]);
            return;
        }
        if (nL != nU && fabs(nL - nU) <= d) {
            const double mid = 0.5 * (nL + nU);
            nL = mid;
            nU = mid;
        }
    }
    if (nL != C.L[i] || nU != C.U[i]) C.rdnext[i] = 1;
    C.L[i] = nL;
    C.U[i] = nU;
}

}  // namespace

}  // namespace lpp
