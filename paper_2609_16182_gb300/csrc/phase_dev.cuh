// phase_dev.cuh -- the block-level work of one round: bodies that the round's
// kernels launch over a grid (k_round.cu, k_compact.cu) and that the kernel
// holding all rounds of one LP (k_solo.cu) runs between grid barriers.
#pragma once
#include <cstring>

#include "compact_dev.cuh"
#include "lpp_dev.cuh"
#include "round_dev.cuh"

namespace lpp {

namespace {

// Rows of 257 to 4096 entries (kMidMin on), S1-S3 by the whole block with the
// sums of prop_row<true>: 32 lane-strided chains, then the butterfly.  All
// eight warps load the entries and their bounds, 512 at a time, into shared
// memory (the candidate queues' space, emptied before); warp 0 then runs the
// chains of the minimum and warp 1 those of the maximum while the next
// entries are on their way.  A warp alone walked such a row four loads at a
// time: 49 to 67 us a round for one row of 4000 entries among 20 k short ones.
constexpr int32_t kMidMin = 257;
constexpr int32_t kMidTile = 2 * kBlock;
static_assert(kMidTile * 24 == (kBlock / 32) * kQueueCap * 24, "the tile fills the queues' space");
struct MidShared {
    double smin, smax;
    unsigned long long h;
    int nmin, nmax, kind;
};

__device__ __forceinline__ void prop_mid(const Ctx &C, int32_t i, MidShared &M, double *tile, int32_t &removed,
                                         int32_t &evaluated, int32_t &tested, CandQueue &q) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double *s_a = tile, *s_l = tile + kMidTile, *s_h = tile + 2 * kMidTile;
    const int32_t beg = C.A.ptr[i], end = C.A.ptr[i + 1];
    const bool rehash = C.rdirty[i] & kRekey;
    cq_flush(C, q);
    if (tid == 0) {
        M.h = 0;
        M.nmin = M.nmax = 0;
    }
    const bool neg0 = rehash ? is_neg(C.A.val[beg]) : false;
    double sum = 0.0;  // warp 0: the lane's chain of the minimum, warp 1: of the maximum
    int nmin = 0, nmax = 0;
    unsigned long long h = 0;
    int32_t j[2];
    double a[2];
    double2 b[2];
    auto load = [&](int32_t t0) {
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int32_t k = t0 + u * kBlock + tid;
            j[u] = k < end ? C.A.idx[k] : -1;
            a[u] = k < end ? C.A.val[k] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 2; u++) b[u] = j[u] >= 0 ? C.lu[j[u]] : make_double2(0.0, 0.0);
    };
    load(beg);
    for (int32_t t0 = beg; t0 < end; t0 += kMidTile) {
        __syncthreads();  // the queues are empty, the chains of the tile before are done
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const bool neg = is_neg(a[u]);
            double bmin = neg ? b[u].y : b[u].x, bmax = neg ? b[u].x : b[u].y;
            // an infinite (or absent) term adds 0: a * 0 leaves the chain as it is
            if (!is_fin(bmin)) {
                nmin++;
                bmin = 0.0;
            }
            if (!is_fin(bmax)) {
                nmax++;
                bmax = 0.0;
            }
            if (rehash && j[u] >= 0) h += entry_hash(j[u], neg != neg0);
            s_a[u * kBlock + tid] = a[u];
            s_l[u * kBlock + tid] = bmin;
            s_h[u * kBlock + tid] = bmax;
        }
        __syncthreads();
        const int32_t steps = (min(end - t0, kMidTile) + 31) / 32;
        if (t0 + kMidTile < end) load(t0 + kMidTile);
        if (warp < 2) {
            const double *bb = warp == 0 ? s_l : s_h;
#pragma unroll 4
            for (int32_t t = 0; t < steps; t++) sum = fma(s_a[32 * t + lane], bb[32 * t + lane], sum);
        }
    }
    nmin = __reduce_add_sync(0xffffffffu, nmin);
    nmax = __reduce_add_sync(0xffffffffu, nmax);
    if (rehash) h = group_sum<32>(h, 0xffffffffu);
    if (warp < 2) sum = group_sum<32>(sum, 0xffffffffu);
    if (lane == 0) {
        if (nmin) atomicAdd(&M.nmin, nmin);
        if (nmax) atomicAdd(&M.nmax, nmax);
        if (rehash) atomicAdd(&M.h, h);
        if (warp < 2) (warp == 0 ? M.smin : M.smax) = sum;
    }
    __syncthreads();
    const double Lv = C.L[i], Uv = C.U[i];
    if (tid == 0) {
        uint8_t kind = RK_KEPT;
        evaluated += end - beg;
        removed += finish_row(C, i, beg, end - beg, Lv, Uv, M.smin, M.smax, M.nmin, M.nmax, rehash,
                              M.h + len_hash(end - beg), kind);
        M.kind = kind;
    }
    __syncthreads();
    const double smin = M.smin, smax = M.smax;
    const int rmin = M.nmin, rmax = M.nmax;
    const bool kept = M.kind == RK_KEPT;
    const bool up_row = kept && is_fin(Uv) && rmin <= 1, lo_row = kept && is_fin(Lv) && rmax <= 1;
    if (up_row || lo_row)  // block-uniform
        tighten_steps(C, q, (end - beg + kBlock - 1) / kBlock, beg + tid, kBlock, end, up_row, lo_row, Uv - smin,
                      Lv - smax, slack_below(Uv, smin), slack_below(smax, Lv), rmin, rmax, tested);
    __syncthreads();  // M is reused by the block's next row
}

// Blocks of a pass over the rows by length class, the longest rows first
// (blk_start[k]: class 5 - k), so that their latency runs beside the short
// rows.  lanes(c): lanes per row of class c < 5; per5: rows of class 5 per
// block (a block takes its rows beyond 256 entries one after the other, about
// 6 us each, so as few as fill the chip).
struct RowGrid {
    GroupGrid g;
    int32_t per5;
};
template <class Lanes>
__host__ __device__ __forceinline__ RowGrid row_grid(const SegMat &M, Lanes lanes) {
    RowGrid r;
    const int32_t cnt5 = M.cls_start[6] - M.cls_start[5];
    r.per5 = cnt5 <= 8 * 152 ? 1 : (cnt5 <= 32 * 152 ? 2 : 4);
    int32_t acc = 0;
    for (int k = 0; k < 6; k++) {
        const int c = 5 - k;
        r.g.blk_start[k] = acc;
        const int32_t per = c == 5 ? r.per5 : kBlock / lanes(c);
        acc += (M.cls_start[c + 1] - M.cls_start[c] + per - 1) / per;
    }
    r.g.blk_start[6] = acc;
    return r;
}
__host__ __device__ __forceinline__ RowGrid prop_grid(const SegMat &M) {
    return row_grid(M, [](int c) { return prop_lanes(c); });
}
__host__ __device__ __forceinline__ RowGrid class_grid(const SegMat &M) {
    return row_grid(M, [](int c) { return 1 << c; });
}

// the row of this thread in block b of class_grid (1 << c lanes per row), and its class
__device__ __forceinline__ int32_t class_row(const SegMat &M, const RowGrid &R, int32_t b, int &c, bool &valid) {
    c = 5 - grid_class(R.g, b);
    const int W = 1 << c, at = threadIdx.x / W;
    const int32_t per = c == 5 ? R.per5 : kBlock / W;
    const int32_t pos = M.cls_start[c] + (b - R.g.blk_start[5 - c]) * per + at;
    valid = at < per && pos < M.cls_start[c + 1];
    return valid ? M.order[pos] : 0;
}

// S1-S3 of the rows of block b of prop_grid
struct PropShared {
    double q[3 * (kBlock / 32) * kQueueCap];  // the warps' queues: coefficients, slacks, columns, flags
    MidShared m;
    int32_t mid[kBlock / 32], nmid;
};
__device__ __forceinline__ void prop_block(const Ctx &C, const RowGrid &R, int32_t b, PropShared &S, int32_t &removed,
                                           int32_t &evaluated, int32_t &tested) {
    constexpr int kQ = (kBlock / 32) * kQueueCap;  // items of the warps' queues
    const int warp = threadIdx.x >> 5;
    int32_t *qi = reinterpret_cast<int32_t *>(S.q + 2 * kQ);
    CandQueue q{S.q + warp * kQueueCap, S.q + kQ + warp * kQueueCap, qi + warp * kQueueCap, qi + kQ + warp * kQueueCap, 0};
    const int c = 5 - grid_class(R.g, b);
    const int W = prop_lanes(c);
    const int32_t per = c == 5 ? R.per5 : kBlock / W, at = threadIdx.x / W;
    const int32_t pos = C.A.cls_start[c] + (b - R.g.blk_start[5 - c]) * per + at;
    bool valid = at < per && pos < C.A.cls_start[c + 1];
    const int32_t i = valid ? C.A.order[pos] : 0;
    if (c < 5) {
        prop_row<false>(C, i, valid, W, removed, evaluated, tested, q);
    } else {
        if (threadIdx.x == 0) S.nmid = 0;
        __syncthreads();
        if (valid && (C.rdirty[i] & kEval) && C.A.ptr[i + 1] - C.A.ptr[i] >= kMidMin) {
            if ((threadIdx.x & 31) == 0) S.mid[atomicAdd(&S.nmid, 1)] = i;
            valid = false;
        }
        prop_row<true>(C, i, valid, 32, removed, evaluated, tested, q);
        __syncthreads();
        const int32_t nmid = S.nmid;
        for (int32_t t = 0; t < nmid; t++) prop_mid(C, S.mid[t], S.m, S.q, removed, evaluated, tested, q);
    }
    cq_flush(C, q);
}

// fixed-order block reduction (warp butterflies, then warps in order)
template <typename T>
__device__ __forceinline__ T block_reduce_ordered(T v, T *s_w) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    T t = T(0);
    if (threadIdx.x == 0)
        for (int w = 0; w < kBlock / 32; w++) t += s_w[w];
    __syncthreads();
    return t;  // thread 0
}

// ------------------------------------------------------------ long rows
// chunk b of the long rows: its partial sums
__device__ __forceinline__ void prop_long_chunk(const Ctx &C, int32_t b) {
    __shared__ double s_d[kBlock / 32];
    __shared__ int s_i[kBlock / 32];
    __shared__ unsigned long long s_h[kBlock / 32];
    const Chunk ch = C.A.chunks[b];
    const uint8_t flag = C.rdirty[ch.seg];
    if (!flag) return;  // block-uniform
    const bool rehash = flag & kRekey;
    const bool neg0 = rehash ? is_neg(C.A.val[C.A.ptr[ch.seg]]) : false;
    double smin = 0.0, smax = 0.0;
    int nmin = 0, nmax = 0;
    unsigned long long h = 0;
#pragma unroll 4
    for (int32_t k = ch.begin + threadIdx.x; k < ch.end; k += kBlock) {
        const int32_t j = __ldcs(C.A.idx + k);  // streamed once: evict first, keep the bounds cached
        const double a = __ldcs(C.A.val + k);
        const double2 lu = C.lu[j];
        const bool neg = is_neg(a);
        const double bmin = neg ? lu.y : lu.x, bmax = neg ? lu.x : lu.y;
        if (is_fin(bmin)) smin = fma(a, bmin, smin);
        else nmin++;
        if (is_fin(bmax)) smax = fma(a, bmax, smax);
        else nmax++;
        if (rehash) h += entry_hash(j, neg != neg0);
    }
    smin = block_reduce_ordered(smin, s_d);
    smax = block_reduce_ordered(smax, s_d);
    nmin = block_reduce_ordered(nmin, s_i);
    nmax = block_reduce_ordered(nmax, s_i);
    if (rehash) h = block_reduce_ordered(h, s_h);
    if (threadIdx.x == 0) {
        C.ch_act[b] = make_double2(smin, smax);
        C.ch_ninf[b] = make_int2(nmin, nmax);
        C.ch_hash[b] = h;
    }
}

// one warp for long row t: the chunk partials, lane-strided then a butterfly
__device__ __forceinline__ void prop_long_row(const Ctx &C, int32_t t, int32_t &removed, int32_t &evaluated) {
    const int lane = threadIdx.x & 31;
    const int32_t nlong = C.A.cls_start[7] - C.A.cls_start[6];
    if (t < nlong) {  // the same t in the whole warp
        const int32_t i = C.A.order[C.A.cls_start[6] + t];
        const uint8_t flag = C.rdirty[i];
        if (!flag) {
            if (lane == 0) {
                C.rkind[i] = RK_KEPT;
                C.lneed[t] = 0;
            }
        } else {
            double smin = 0.0, smax = 0.0;
            int nmin = 0, nmax = 0;
            unsigned long long h = 0;
            for (int32_t q = C.A.lfirst[t] + lane; q < C.A.lfirst[t + 1]; q += 32) {
                const double2 a = C.ch_act[q];
                const int2 c = C.ch_ninf[q];
                smin += a.x;
                smax += a.y;
                nmin += c.x;
                nmax += c.y;
                h += C.ch_hash[q];
            }
            smin = group_sum<32>(smin, 0xffffffffu);
            smax = group_sum<32>(smax, 0xffffffffu);
            nmin = group_sum<32>(nmin, 0xffffffffu);
            nmax = group_sum<32>(nmax, 0xffffffffu);
            h = group_sum<32>(h, 0xffffffffu);
            if (lane == 0) {
                const int32_t beg = C.A.ptr[i], len = C.A.ptr[i + 1] - beg;
                h += len_hash(len);
                const double Lv = C.L[i], Uv = C.U[i];
                uint8_t kind;
                removed += finish_row(C, i, beg, len, Lv, Uv, smin, smax, nmin, nmax, flag & kRekey, h, kind);
                evaluated += len;
                C.lneed[t] = kind == RK_KEPT && ((is_fin(Uv) && nmin <= 1) || (is_fin(Lv) && nmax <= 1));
            }
        }
    }
}

// chunk b of the long rows: S3
__device__ __forceinline__ void prop_long_tighten(const Ctx &C, int32_t b, int32_t &tested) {
    const Chunk ch = C.A.chunks[b];
    if (!C.lneed[ch.lidx]) return;
    const int32_t i = ch.seg;
    const double Lv = C.L[i], Uv = C.U[i];
    const double2 act = C.act[i];
    const int2 ni = C.ninf[i];
    const bool up_row = is_fin(Uv) && ni.x <= 1, lo_row = is_fin(Lv) && ni.y <= 1;
    const double dU = Uv - act.x, dL = Lv - act.y;
    const float fU = slack_below(Uv, act.x), fL = slack_below(act.y, Lv);
#pragma unroll 4
    for (int32_t k = ch.begin + threadIdx.x; k < ch.end; k += kBlock)
        tighten_entry(C, C.A.idx[k], C.A.val[k], up_row, lo_row, dU, dL, fU, fL, ni.x, ni.y, tested);
}

// ------------------------------------------ S3 bound sources (dual records)
// The dual postsolve moves a reduced cost on a tightened bound to the row
// that implied it, so each accepted candidate needs its row.  Between S3 and
// S3', every row S1-S3 evaluated this round (a dirty flag) runs over its
// entries again, row by row as S3 does: an entry whose column received a
// candidate re-derives its implied bound (or the singleton row's bound) on
// the stored activities with the activity kernels' arithmetic, and a value
// equal to the accepted candidate (encoded values compared: bit for bit)
// offers its original row index to the column's side (atomicMin: the
// smallest row wins).
__device__ __forceinline__ void bsrc_offer(const Ctx &C, int32_t j, double x, double a, bool upper, bool capped,
                                           unsigned long long el, unsigned long long eu, int32_t o) {
    if (capped && gt0(fma(-C.max_implied, fabs(a), fabs(x)))) return;
    const double v = bound_value(x, a);
    if (!is_fin(v)) return;
    const unsigned long long e = enc_dbl(v);
    if (upper) {
        if (e == eu) atomicMin(&C.bsrc[j].y, o);
    } else if (e == el) {
        atomicMin(&C.bsrc[j].x, o);
    }
}

// entries [k0, k1) of row i, every step-th from k0
__device__ __forceinline__ void bsrc_row(const Ctx &C, int32_t i, int32_t k0, int32_t k1, int32_t step) {
    const uint8_t kind = C.rkind[i];
    const int32_t len = C.A.ptr[i + 1] - C.A.ptr[i];
    if (!(kind == RK_SINGLETON || (kind == RK_KEPT && len >= 2))) return;
    const double Lv = C.L[i], Uv = C.U[i];
    const int32_t o = C.rmap[i];
    const double2 act = C.act[i];
    const int2 ni = C.ninf[i];
    const bool up_row = is_fin(Uv) && ni.x <= 1, lo_row = is_fin(Lv) && ni.y <= 1;
    const double dU = Uv - act.x, dL = Lv - act.y;
    for (int32_t k = k0; k < k1; k += step) {
        const int32_t j = C.A.idx[k];
        if (C.ctouch[j] == 0u) continue;  // no candidate this round (one 4-byte gather)
        const unsigned long long el = C.cand_l[j], eu = C.cand_u[j];
        if (el == kEncNegInf && eu == kEncPosInf) continue;
        const double a = C.A.val[k];
        const bool neg = is_neg(a);
        if (kind == RK_SINGLETON) {  // L <= a x_j <= U: bounds L/a and U/a (a < 0 swaps them), no cap
            if (is_fin(Lv)) bsrc_offer(C, j, Lv, a, neg, false, el, eu, o);
            if (is_fin(Uv)) bsrc_offer(C, j, Uv, a, !neg, false, el, eu, o);
            continue;
        }
        const double2 b = C.lu[j];
        const double bmin = neg ? b.y : b.x, bmax = neg ? b.x : b.y;
        const bool fmn = is_fin(bmin), fmx = is_fin(bmax);
        if (up_row && (fmn ? ni.x == 0 : ni.x == 1))  // a x_j <= U - (min activity of the others)
            bsrc_offer(C, j, fmn ? fma(a, bmin, dU) : dU, a, !neg, true, el, eu, o);
        if (lo_row && (fmx ? ni.y == 0 : ni.y == 1))  // a x_j >= L - (max activity of the others)
            bsrc_offer(C, j, fmx ? fma(a, bmax, dL) : dL, a, neg, true, el, eu, o);
    }
}

// the rows of block b of class_grid; rows of more than 64 entries by the whole block
__device__ __forceinline__ void bsrc_block(const Ctx &C, const RowGrid &R, int32_t b) {
    int c;
    bool valid;
    const int32_t i = class_row(C.A, R, b, c, valid);
    if (c < 5) {
        const int W = 1 << c;
        if (valid && C.rdirty[i] != 0)
            bsrc_row(C, i, C.A.ptr[i] + (int32_t)(threadIdx.x & (W - 1)), C.A.ptr[i + 1], W);
        return;
    }
    for (int32_t q = 0; q < R.per5; q++) {
        const int32_t pos = C.A.cls_start[5] + (b - R.g.blk_start[0]) * R.per5 + q;
        if (pos >= C.A.cls_start[6]) break;
        const int32_t k = C.A.order[pos];
        if (C.rdirty[k] != 0) bsrc_row(C, k, C.A.ptr[k] + (int32_t)threadIdx.x, C.A.ptr[k + 1], kBlock);
    }
}

// ------------------------------------------------------------ S5, first pass
__device__ __forceinline__ bool match_class(const Ctx &C, int c, int32_t i, bool valid, int32_t &removed,
                                            int32_t &unmatched) {
    switch (c) {
        case 0: return match_group<1>(C, i, valid, removed, unmatched);
        case 1: return match_group<2>(C, i, valid, removed, unmatched);
        case 2: return match_group<4>(C, i, valid, removed, unmatched);
        case 3: return match_group<8>(C, i, valid, removed, unmatched);
        case 4: return match_group<16>(C, i, valid, removed, unmatched);
        default: return match_group<32>(C, i, valid, removed, unmatched);
    }
}

// long row t: one block (parallel long rows are rare)
__device__ __forceinline__ void match_long(const Ctx &C, int32_t t, int32_t *out, int32_t *out_cnt, int32_t &removed,
                                           int32_t &unmatched) {
    const int32_t i = C.A.order[C.A.cls_start[6] + t];
    bool act = C.rwork[i] == 1;
    int32_t li = -1;
    if (act) {
        li = (int32_t)(uint32_t)(C.tlead[C.rslot[i]] & 0xffffffffULL);
        if (li == i) act = false;
    }
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
        for (int32_t k = threadIdx.x; k < len; k += kBlock) {
            const double ai = C.A.val[bi + k], al = C.A.val[bl + k];
            const double la = lam * al;
            if (!(C.A.idx[bi + k] == C.A.idx[bl + k] && fabs(ai - la) <= C.par_tol * fmax(fabs(ai), fabs(la))))
                ok = false;
        }
    }
    ok = __syncthreads_and(ok) != 0;
    if (threadIdx.x == 0) {
        if (act && ok) {
            s5_accept(C, i, li, lam);
            C.rwork[i] = 0;
            removed++;
        } else if (act) {
            C.rwork[i] = 2;
            unmatched++;
            out[atomicAdd(out_cnt, 1)] = i;
        } else {
            C.rwork[i] = 0;
        }
    }
}

// A barrier over the blocks of a cooperative launch: *bar, zero at the launch,
// counts the arrivals of all barriers so far; gen is the number passed, the same
// in every thread.  One release-add per block and one acquire load that sees the
// last one: no counter to reset, no second word to publish (with those, a call
// on 20 k rows, 110 barriers of 176 blocks, took 3 to 8% longer).  One block: a
// block barrier.
// A wait that takes too long (with every block resident: longer than any work
// between two barriers) sets *err bit 4 and returns false, as do then all later
// waits.  Work that may take longer changes *progress (if given) as it goes, and
// the waits count anew.
constexpr int32_t kBarSpins = 1 << 22;
__device__ bool grid_barrier(unsigned *bar, int32_t *err, unsigned &gen, const int32_t *progress = nullptr) {
    __shared__ int s_ok;
    __syncthreads();
    if (gridDim.x == 1) return true;
    gen++;
    if (threadIdx.x == 0) {
        const unsigned want = gen * gridDim.x;
        int ok = 1;
        int32_t seen = 0;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        for (int32_t spins = 0;; spins++) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if ((int)(v - want) >= 0) break;
            if ((spins & 255) != 255) continue;
            if (progress) {
                const int32_t p = *(const volatile int32_t *)progress;
                if (p != seen) spins = 0;
                seen = p;
            }
            if (spins > kBarSpins || (*(volatile int32_t *)err & 4)) {
                atomicOr(err, 4);
                ok = 0;
                break;
            }
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// S5's later passes p0, p0 + 1, ... of a cooperative launch: rows of the list
// l0/l1 (by the pass's parity; n rows at first, cnt[p] those pass p leaves, zero
// before) into the table, each against its slot's leader, the unmatched to the
// next list.  Mutable data (lists, slots, leaders, counts) is read at L2.
// The table's halves take turns: while pass p matches in one, the other is
// emptied for pass p + 1, so a pass has two barriers, not three; a list too long
// for half the table (the first passes, if at all: lists shrink) empties the
// slots it used behind a barrier of its own.  From kTailAlone rows on block 0
// goes on alone (its barriers are block barriers); n and removed are its then,
// and it counts its passes in *progress (if given): there are up to as many as
// rows, of rows of any length.
// On 2 M rows the tail took 326 us with three barriers a pass of the
// former kind, now 244; on 500 k rows 184, now 110.
constexpr int32_t kTailAlone = 2 * kBlock;
__device__ __forceinline__ bool s5_later_passes(const Ctx &C, int32_t *l0, int32_t *l1, int32_t *cnt, int32_t p0,
                                                int32_t max_iter, int32_t &n, int32_t &removed, unsigned *bar,
                                                int32_t *err, unsigned &gen, int32_t *progress = nullptr) {
    const int32_t gt = blockIdx.x * kBlock + threadIdx.x;
    bool one = gridDim.x == 1;
    uint32_t prev_off = 0, prev_cap = 0, own = 0;
    for (int32_t p = p0; p < max_iter && n > 0; p++) {
        const uint32_t half = (uint32_t)C.tcap / 2, cap = s5_tail_cap(C, n);
        const bool turns = cap <= half;
        uint32_t off = turns ? (p & 1) * half : 0;
        if (!one && turns && n <= kTailAlone) {
            if (blockIdx.x != 0) return true;
            one = true;  // in this pass's half from here on: the other one is not empty
            own = off;
        }
        if (one) off = own;
        const int32_t ft = one ? (int32_t)threadIdx.x : gt, fs = one ? kBlock : (int32_t)gridDim.x * kBlock;
        const int32_t *lst = (p - 1) & 1 ? l1 : l0;
        int32_t *nxt = (p - 1) & 1 ? l0 : l1;
        for (int32_t t = ft; t < n; t += fs) {
            const int32_t i = __ldcg(lst + t);
            C.rslot[i] = s5_insert_row(C, i, cap, off);
        }
        if (one) __syncthreads();
        else if (!grid_barrier(bar, err, gen)) return false;
        if (!one)
            for (uint32_t k = (uint32_t)gt; k < prev_cap; k += (uint32_t)fs) {
                C.tkey[prev_off + k] = 0ULL;
                C.tlead[prev_off + k] = ~0ULL;
            }
        for (int32_t tb = ft & ~31; tb < n; tb += fs) {  // warp-uniform: every lane calls the match
            int32_t rm, i;
            bool left;
            s5_tail_match_one(C, lst, n, tb + (threadIdx.x & 31), rm, left, i);
            removed += rm;
            const unsigned want = __ballot_sync(0xffffffffu, left);
            int32_t at = 0;
            if ((threadIdx.x & 31) == 0 && want) at = atomicAdd(cnt + p, __popc(want));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (left) nxt[at + __popc(want & ((1u << (threadIdx.x & 31)) - 1u))] = i;
        }
        if (one) __syncthreads();
        else if (!grid_barrier(bar, err, gen)) return false;
        if (one || !turns) {
            for (int32_t t = ft; t < n; t += fs) {
                const int32_t sl = __ldcg(C.rslot + __ldcg(lst + t));
                if (sl >= 0) {
                    C.tkey[sl] = 0ULL;
                    C.tlead[sl] = ~0ULL;
                }
            }
            if (one) __syncthreads();
            else if (!grid_barrier(bar, err, gen)) return false;
        }
        prev_off = off;
        prev_cap = turns ? cap : 0;
        n = __ldcg(cnt + p);
        if (one && progress && threadIdx.x == 0) *(volatile int32_t *)progress = p;
    }
    return true;
}

// The flat scatter's tile t starts at entry t * kFlatTile; the segment (or
// chunk) [b, e) that holds that entry records itself.  Segments and chunks
// are at most kFlatTile long, so each holds at most one tile start.
__device__ __forceinline__ void mark_tile(int32_t *tile, int32_t b, int32_t e, int32_t seg) {
    const int64_t t = ((int64_t)b + kFlatTile - 1) / kFlatTile;
    if (t * kFlatTile < e) tile[t] = seg;
}

__device__ __forceinline__ int32_t block_sum_int(int32_t v) {
    __shared__ int32_t s_w[kBlock / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    int32_t t = 0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kBlock / 32; w++) t += s_w[w];
    __syncthreads();
    return t;
}

__device__ __forceinline__ double block_sum_dbl(double v) {
    __shared__ double s_w[kBlock / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kBlock / 32; w++) t += s_w[w];
    __syncthreads();
    return t;
}

// long segment t (one warp): chunk offsets (prefix in chunk order), the
// total, and the sum of the chunks' side shifts (lane-strided, then a butterfly)
__device__ __forceinline__ void long_prefix(const SegMat &M, int32_t t, const int32_t *ch_cnt, int32_t *ch_off,
                                            int32_t *len_out, const double *ch_shift, double *shift_out) {
    const int lane = threadIdx.x & 31;
    const int32_t nlong = M.cls_start[7] - M.cls_start[6];
    if (t >= nlong) return;  // the same t in the whole warp
    const int32_t q1 = M.lfirst[t + 1];
    int32_t carry = 0;
    double sh = 0.0;
    for (int32_t q0 = M.lfirst[t]; q0 < q1; q0 += 32) {
        const int32_t q = q0 + lane;
        const int32_t c = q < q1 ? ch_cnt[q] : 0;
        int32_t inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (q < q1) {
            ch_off[q] = carry + inc - c;
            if (ch_shift) sh += ch_shift[q];
        }
        carry += __shfl_sync(0xffffffffu, inc, 31);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sh += __shfl_xor_sync(0xffffffffu, sh, o);
    if (lane == 0) {
        const int32_t seg = M.order[M.cls_start[6] + t];
        len_out[seg] = carry;
        if (shift_out) shift_out[seg] = sh;
    }
}

// S6 and the keep flag with the columns in place: a column that left in an
// earlier round (cinv < 0) is skipped, a kept one with entries stays as it is
// (no S6 test applies to it, its contribution is zero), and one that leaves
// now gets cinv = -1.
__device__ __forceinline__ int32_t colkeep_in_place(const Ctx &C, const CompactCtx &K, int32_t j) {
    const uint8_t st = C.cchg[j];
    const bool used = (st & CS_USED) || !(C.round == 1 || (st & CS_SUSPECT));
    if (used && C.ckind[j] == CK_KEPT && !K.lp_dead[lp_of_col(C, j)]) return 0;
    if (C.cinv[j] < 0) return 0;
    K.c_len[j] = used;
    const int32_t fixed = colkeep_one(C, K, j);
    if (!K.c_keep[j]) K.cinv[j] = -1;
    return fixed;
}

// ------------------------------------- columns in place: the rows' one pass
// Over a kept row's entries with one byte gathered per entry (its column's
// state): entries left and the side shift (as csr_count_row, the same order),
// whether a column's bounds changed (the row is then evaluated next round),
// and for the columns that may have become empty (those of rows that left,
// suspect_row; in round 1 all) whether the row holds them, for S6.  It takes
// the place of an A^T of the input kept through the rounds: the transpose at
// ingest, the marking of the changed columns' rows through it, the counts per
// column and their decrements.  A column that many rows hold would be stored
// by nearly each of them (the SM's L1 keeps the byte as first read, and stores
// to one address serialise in L2: 146 us a round on 7 M entries with ten dense
// columns); a small table of the columns the block has stored filters those.
// COUNT false: a round that removed nothing, the marking alone.
constexpr int kSeen = 512;  // slots of the table, a power of two
template <bool COUNT>
__device__ __forceinline__ void inplace_entry(const Ctx &C, int32_t j, uint8_t st, int32_t *seen) {
    if (!COUNT || (st & (CS_LEAVES | CS_USED)) || !(C.round == 1 || (st & CS_SUSPECT))) return;
    if (seen) {
        volatile int32_t *slot = seen + (j & (kSeen - 1));
        if (*slot == j) return;  // a thread of the block stores it
        *slot = j;
    }
    C.cchg[j] = st | CS_USED;  // every writer stores the same byte
}

// the columns of row i, if it leaves this round, may be empty now (W lanes)
__device__ __forceinline__ void suspect_row(const Ctx &C, int32_t i, bool valid, int W) {
    if (!valid || C.rkind[i] == RK_KEPT) return;
    const int32_t e = C.A.ptr[i + 1];
    for (int32_t k = C.A.ptr[i] + (int32_t)(threadIdx.x & (W - 1)); k < e; k += W) {
        const int32_t j = C.A.idx[k];
        const uint8_t st = C.cchg[j];
        if (!(st & CS_SUSPECT)) C.cchg[j] = st | CS_SUSPECT;
    }
}
__device__ __forceinline__ void suspect_block(const Ctx &C, const RowGrid &R, int32_t b) {
    int c;
    bool valid;
    const int32_t i = class_row(C.A, R, b, c, valid);
    suspect_row(C, i, valid, 1 << c);
}
__device__ __forceinline__ void suspect_chunk(const Ctx &C, int32_t b) {
    const Chunk ch = C.A.chunks[b];
    if (C.rkind[ch.seg] == RK_KEPT) return;
    for (int32_t k = ch.begin + threadIdx.x; k < ch.end; k += kBlock) {
        const int32_t j = C.A.idx[k];
        const uint8_t st = C.cchg[j];
        if (!(st & CS_SUSPECT)) C.cchg[j] = st | CS_SUSPECT;
    }
}

template <int W, bool COUNT>
__device__ __forceinline__ void inplace_row(const Ctx &C, const CompactCtx &K, int32_t i, bool valid, int32_t *seen) {
    const unsigned mask = group_mask<W>();
    const int lane = threadIdx.x & (W - 1);
    const bool keep = valid && C.rkind[i] == RK_KEPT && !K.lp_dead[lp_of_row(C, i)];
    int32_t beg = 0, end = 0;
    if (valid) {
        beg = C.A.ptr[i];
        end = C.A.ptr[i + 1];
        if (COUNT && lane == 0) mark_tile(K.tile_a, beg, end, i);
    }
    int32_t cnt = 0, any = 0;
    double sh = 0.0;
    for (int32_t k0 = beg + lane; keep && k0 < end; k0 += 4 * W) {
        int32_t jq[4];
        uint8_t sq[4];
#pragma unroll
        for (int q = 0; q < 4; q++) jq[q] = k0 + q * W < end ? C.A.idx[k0 + q * W] : -1;
#pragma unroll
        for (int q = 0; q < 4; q++) sq[q] = jq[q] >= 0 ? C.cchg[jq[q]] : (uint8_t)0;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if (jq[q] < 0) break;
            any |= sq[q] & CS_CHANGED;
            if (!COUNT) continue;
            if (sq[q] & CS_LEAVES) sh = fma(C.A.val[k0 + q * W], C.fixv[jq[q]], sh);
            else cnt++;
            inplace_entry<COUNT>(C, jq[q], sq[q], seen);
        }
    }
    any = group_sum<W>(any, mask);
    if (COUNT) {
        cnt = group_sum<W>(cnt, mask);
        sh = group_sum<W>(sh, mask);
    }
    if (valid && lane == 0) {
        if (any) C.rdnext[i] = 1;
        if (COUNT) {
            K.r_keep[i] = keep;
            K.r_len[i] = cnt;
            K.shift[i] = sh;
        }
    }
}

// A row of 257 to 4096 entries by the whole block, 512 entries in flight.
// The shift's 32 lane-strided chains run in one warp, from shared memory, in
// the tiles that hold a leaving column's entry.
constexpr int32_t kMidRow = 257;
constexpr int kMidStep = 2 * kBlock;
template <bool COUNT>
__device__ __forceinline__ void inplace_mid(const Ctx &C, const CompactCtx &K, int32_t i, double *s_a, double *s_v,
                                            int32_t *s_sum, int32_t *seen) {
    const int tid = threadIdx.x, lane = tid & 31;
    const int32_t beg = C.A.ptr[i], end = C.A.ptr[i + 1];
    if (tid < 2) s_sum[tid] = 0;
    int32_t cnt = 0, any = 0;
    double sh = 0.0;
    for (int32_t t0 = beg; t0 < end; t0 += kMidStep) {
        int32_t jq[2];
        uint8_t sq[2];
#pragma unroll
        for (int q = 0; q < 2; q++) jq[q] = t0 + q * kBlock + tid < end ? C.A.idx[t0 + q * kBlock + tid] : -1;
#pragma unroll
        for (int q = 0; q < 2; q++) sq[q] = jq[q] >= 0 ? C.cchg[jq[q]] : (uint8_t)0;
        int32_t leaves = 0;
#pragma unroll
        for (int q = 0; q < 2; q++) {
            if (jq[q] < 0) continue;
            any |= sq[q] & CS_CHANGED;
            if (!COUNT) continue;
            leaves |= sq[q] & CS_LEAVES;
            cnt += !(sq[q] & CS_LEAVES);
            inplace_entry<COUNT>(C, jq[q], sq[q], seen);
        }
        if (COUNT && __syncthreads_or(leaves)) {
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const bool lv = jq[q] >= 0 && (sq[q] & CS_LEAVES);
                s_a[q * kBlock + tid] = lv ? C.A.val[t0 + q * kBlock + tid] : 0.0;
                s_v[q * kBlock + tid] = lv ? C.fixv[jq[q]] : 0.0;
            }
            __syncthreads();
            if (tid < 32)
                for (int32_t t = 0; t < kMidStep / 32; t++) sh = fma(s_a[32 * t + lane], s_v[32 * t + lane], sh);
            __syncthreads();
        }
    }
    __syncthreads();
    any = __reduce_or_sync(0xffffffffu, (unsigned)any);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) {
        if (any) s_sum[1] = 1;
        if (cnt) atomicAdd(&s_sum[0], cnt);
    }
    if (COUNT && tid < 32) sh = group_sum<32>(sh, 0xffffffffu);
    __syncthreads();
    if (tid == 0) {
        if (s_sum[1]) C.rdnext[i] = 1;
        if (COUNT) {
            mark_tile(K.tile_a, beg, end, i);
            K.r_keep[i] = 1;
            K.r_len[i] = s_sum[0];
            K.shift[i] = sh;
        }
    }
    __syncthreads();
}

// The same row by the keep flags (the columns compacted each round): entries
// left and the side shift.
__device__ __forceinline__ void count_mid(const Ctx &C, const CompactCtx &K, int32_t i, double *s_a, double *s_v,
                                          int32_t *s_sum) {
    const int tid = threadIdx.x, lane = tid & 31;
    const int32_t beg = C.A.ptr[i], end = C.A.ptr[i + 1];
    if (tid == 0) s_sum[0] = 0;
    int32_t cnt = 0;
    double sh = 0.0;
    for (int32_t t0 = beg; t0 < end; t0 += kMidStep) {
        int32_t jq[2];
        bool kq[2];
#pragma unroll
        for (int q = 0; q < 2; q++) jq[q] = t0 + q * kBlock + tid < end ? C.A.idx[t0 + q * kBlock + tid] : -1;
#pragma unroll
        for (int q = 0; q < 2; q++) kq[q] = jq[q] < 0 || K.c_keep[jq[q]];
        cnt += (jq[0] >= 0 && kq[0]) + (jq[1] >= 0 && kq[1]);
        if (__syncthreads_or(!kq[0] || !kq[1])) {
#pragma unroll
            for (int q = 0; q < 2; q++) {
                s_a[q * kBlock + tid] = kq[q] ? 0.0 : C.A.val[t0 + q * kBlock + tid];
                s_v[q * kBlock + tid] = kq[q] ? 0.0 : C.fixv[jq[q]];
            }
            __syncthreads();
            if (tid < 32)
                for (int32_t t = 0; t < kMidStep / 32; t++) sh = fma(s_a[32 * t + lane], s_v[32 * t + lane], sh);
            __syncthreads();
        }
    }
    __syncthreads();
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0 && cnt) atomicAdd(&s_sum[0], cnt);
    if (tid < 32) sh = group_sum<32>(sh, 0xffffffffu);
    __syncthreads();
    if (tid == 0) {
        mark_tile(K.tile_a, beg, end, i);
        K.r_keep[i] = 1;
        K.r_len[i] = s_sum[0];
        K.shift[i] = sh;
    }
    __syncthreads();
}

// the rows of block b of class_grid
struct InplaceShared {
    double a[kMidStep], v[kMidStep];
    int32_t mid[kBlock / 32], nmid, sum[2];
    int32_t seen[kSeen];
};
template <bool COUNT>
__device__ __forceinline__ void inplace_block(const Ctx &C, const CompactCtx &K, const RowGrid &R, int32_t b,
                                              InplaceShared &S) {
    int c;
    bool valid;
    const int32_t i = class_row(C.A, R, b, c, valid);
    int32_t *seen = S.seen;
    if (COUNT) {
        for (int t = threadIdx.x; t < kSeen; t += kBlock) seen[t] = -1;
        __syncthreads();
    }
    switch (c) {
        case 0: inplace_row<1, COUNT>(C, K, i, valid, seen); break;
        case 1: inplace_row<2, COUNT>(C, K, i, valid, seen); break;
        case 2: inplace_row<4, COUNT>(C, K, i, valid, seen); break;
        case 3: inplace_row<8, COUNT>(C, K, i, valid, seen); break;
        case 4: inplace_row<16, COUNT>(C, K, i, valid, seen); break;
        default: {
            if (threadIdx.x == 0) S.nmid = 0;
            __syncthreads();
            if (valid && C.A.ptr[i + 1] - C.A.ptr[i] >= kMidRow && C.rkind[i] == RK_KEPT && !K.lp_dead[lp_of_row(C, i)]) {
                if ((threadIdx.x & 31) == 0) S.mid[atomicAdd(&S.nmid, 1)] = i;
                valid = false;
            }
            inplace_row<32, COUNT>(C, K, i, valid, seen);
            __syncthreads();
            const int32_t nmid = S.nmid;
            for (int32_t t = 0; t < nmid; t++) inplace_mid<COUNT>(C, K, S.mid[t], S.a, S.v, S.sum, seen);
        }
    }
}

// chunk b of the long rows, columns in place
template <bool COUNT>
__device__ __forceinline__ void inplace_chunk(const Ctx &C, const CompactCtx &K, int32_t b) {
    const Chunk ch = C.A.chunks[b];
    const int32_t i = ch.seg;
    const bool keep = C.rkind[i] == RK_KEPT && !K.lp_dead[lp_of_row(C, i)];
    int32_t cnt = 0, any = 0;
    double sh = 0.0;
    if (keep) {  // eight entries per thread and step in flight; the shift in entry order
        for (int32_t k0 = ch.begin + threadIdx.x; k0 < ch.end; k0 += 8 * kBlock) {
            int32_t jq[8];
            uint8_t sq[8];
#pragma unroll
            for (int q = 0; q < 8; q++) jq[q] = k0 + q * kBlock < ch.end ? C.A.idx[k0 + q * kBlock] : -1;
#pragma unroll
            for (int q = 0; q < 8; q++) sq[q] = jq[q] >= 0 ? C.cchg[jq[q]] : (uint8_t)0;
#pragma unroll
            for (int q = 0; q < 8; q++) {
                if (jq[q] < 0) break;
                any |= sq[q] & CS_CHANGED;
                if (!COUNT) continue;
                if (sq[q] & CS_LEAVES) sh = fma(C.A.val[k0 + q * kBlock], C.fixv[jq[q]], sh);
                else cnt++;
                inplace_entry<COUNT>(C, jq[q], sq[q], nullptr);
            }
        }
    }
    if (__reduce_or_sync(0xffffffffu, (unsigned)any) && (threadIdx.x & 31) == 0) C.rdnext[i] = 1;
    if (!COUNT) return;
    cnt = block_sum_int(cnt);
    sh = block_sum_dbl(sh);
    if (threadIdx.x == 0) {
        K.chr_cnt[b] = cnt;
        K.chr_shift[b] = sh;
        mark_tile(K.tile_a, ch.begin, ch.end, i);
        if (ch.begin == C.A.ptr[i]) {  // the first chunk writes the flag
            K.r_keep[i] = keep;
            K.r_ch0[i] = b;
        }
    }
}

// ---------------------------------------------------------------- scatter
// Flat ordered compaction of all entries.  Segments of at most kFlatTile
// entries, and the chunks of kChunk entries of the long ones, are the units.
// Block t takes the entries [t T, t T + T) of the matrix, T = kFlatTile:
//   1. one thread per segment between the segments of the entries t T and
//      (t + 1) T (coalesced, independent loads) marks the first in-tile entry
//      of each of its units in the tile, with a keep bit and the unit's base;
//      a block max-scan of the marks gives every entry the first in-tile
//      entry of its unit, or -1 if its segment is dropped;
//   2. striped (coalesced): keep = unit kept and the other index kept (one
//      gather of its new index, -1 if dropped); one ballot per warp and
//      step, exclusive scan of the counts;
//   3. striped: a kept entry x of unit s goes to
//         off[s] + (kept entries of s before x),
//      where the second term is scan(x) - scan(first in-tile entry of s) plus,
//      for a unit that started in an earlier tile, len[s] minus its kept
//      entries in this tile (it ends in this tile: it has at most T entries).
struct FlatArgs {
    const int32_t *ptr, *idx;
    const double *val;
    int32_t nnz, cnt, ntiles;
    const int32_t *seg_keep, *seg_off, *seg_len;  // per segment: kept, new offset, kept entries
    const int32_t *seg_ch0;                       // per long segment: its first chunk
    const int32_t *ch_off, *ch_cnt;               // per chunk: kept entries of its segment before it, its own
    const int32_t *oth_new;                       // per index of the other dimension: new index, -1 if dropped
    const uint8_t *oth_state;                     // columns in place, instead: their states (they keep their index)
    const int32_t *tile_seg;                      // per tile: segment of its first entry
    int32_t *out_idx;
    double *out_val;
};

constexpr int kFlatPer = kFlatTile / kBlock;  // entries per thread
constexpr int kFlatWords = kFlatTile / 32;    // ballot words per tile

struct FlatShared {
    int16_t __align__(16) start[kFlatTile];
    int32_t raw[kFlatTile];
    unsigned bal[kFlatWords + 1];
    int32_t cb[kFlatWords + 1];
    int32_t wmax[kBlock / 32];
    int32_t re, fp;
};
__device__ __forceinline__ void flat_tile(const FlatArgs &F, int t, FlatShared &S) {
    int16_t *s_start = S.start;
    int32_t *s_raw = S.raw, *s_cb = S.cb, *s_wmax = S.wmax;
    unsigned *s_bal = S.bal;
    int32_t &s_re = S.re, &s_fp = S.fp;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t k0 = (int32_t)((int64_t)t * kFlatTile);
    const int32_t len = F.nnz - k0 < kFlatTile ? F.nnz - k0 : kFlatTile;

    // 1a. no marks; 1b. one thread per segment marks its units
    {
        int4 *w = reinterpret_cast<int4 *>(s_start);
        for (int q = tid; q < kFlatTile / 8; q += kBlock) w[q] = make_int4(-1, -1, -1, -1);
    }
    if (tid == 0) s_fp = 0;
    __syncthreads();
    const int32_t lo = F.tile_seg[t];
    const int32_t hi = t + 1 < F.ntiles ? F.tile_seg[t + 1] : F.cnt - 1;
    const int32_t k1 = k0 + len;
    for (int32_t r = lo + tid; r <= hi; r += kBlock) {
        const int32_t pb = F.ptr[r], pe = F.ptr[r + 1];
        if (pe <= pb || pb >= k1) continue;  // empty, or after the tile
        const bool emit = F.seg_keep[r] != 0;
        // units of r that meet the tile: the segment, or chunks q0..q1
        int32_t q0 = 0, q1 = 0;
        const bool lng = pe - pb >= kLongMin;
        if (lng) {
            q0 = ((pb > k0 ? pb : k0) - pb) / kChunk;
            q1 = ((pe < k1 ? pe : k1) - 1 - pb) / kChunk;
        }
        for (int32_t q = q0; q <= q1; q++) {
            const int32_t vb = pb + q * kChunk;
            const int32_t ve = lng ? min(vb + kChunk, pe) : pe;
            const int32_t xs = vb > k0 ? vb - k0 : 0;
            s_start[xs] = (int16_t)(2 * xs + (emit ? 1 : 0));
            if (emit) {
                int32_t raw, ln;
                if (lng) {
                    const int32_t ch = F.seg_ch0[r] + q;
                    raw = F.seg_off[r] + F.ch_off[ch];
                    ln = F.ch_cnt[ch];
                } else {
                    raw = F.seg_off[r];
                    ln = F.seg_len[r];
                }
                if (vb < k0) {  // the unit holding entry k0
                    raw += ln;
                    s_re = ve - k0;
                    s_fp = 1;
                }
                s_raw[xs] = raw;
            }
        }
    }
    __syncthreads();
    // 1c. inclusive max-scan of the marks (blocked, 16 per thread)
    {
        const int x0 = tid * kFlatPer;
        int4 *w = reinterpret_cast<int4 *>(s_start + x0);
        int4 a = w[0], b = w[1];
        int16_t v[kFlatPer];
        memcpy(v, &a, 16);
        memcpy(v + 8, &b, 16);
        int32_t run = -1;
#pragma unroll
        for (int e = 0; e < kFlatPer; e++) {
            run = v[e] > run ? v[e] : run;
        }
        int32_t inc = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o && y > inc) inc = y;
        }
        if (lane == 31) s_wmax[warp] = inc;
        int32_t prev = __shfl_up_sync(0xffffffffu, inc, 1);
        if (lane == 0) prev = -1;
        __syncthreads();
        for (int q = 0; q < warp; q++) prev = s_wmax[q] > prev ? s_wmax[q] : prev;
        run = prev;
#pragma unroll
        for (int e = 0; e < kFlatPer; e++) {
            run = v[e] > run ? v[e] : run;
            v[e] = (x0 + e < len && (run & 1)) ? (int16_t)(run >> 1) : (int16_t)-1;
        }
        memcpy(&a, v, 16);
        memcpy(&b, v + 8, 16);
        w[0] = a;
        w[1] = b;
    }
    __syncthreads();

    // 2. keep flags, striped
    int32_t jn[kFlatPer];
#pragma unroll
    for (int i = 0; i < kFlatPer; i++) {
        const int x = i * kBlock + tid;
        jn[i] = -1;
        if (x < len && s_start[x] >= 0) jn[i] = F.idx[k0 + x];
    }
#pragma unroll
    for (int i = 0; i < kFlatPer; i++) {
        if (jn[i] >= 0) {
            if (F.oth_state) jn[i] = F.oth_state[jn[i]] & CS_LEAVES ? -1 : jn[i];
            else jn[i] = F.oth_new[jn[i]];
        }
        const unsigned bal = __ballot_sync(0xffffffffu, jn[i] >= 0);
        if (lane == 0) s_bal[i * (kBlock / 32) + warp] = bal;
    }
    __syncthreads();
    if (warp == 0) {  // exclusive scan of the ballot counts
        constexpr int per = kFlatWords / 32;
        int32_t c[per], tot = 0;
#pragma unroll
        for (int q = 0; q < per; q++) {
            c[q] = __popc(s_bal[lane * per + q]);
            tot += c[q];
        }
        int32_t inc = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        int32_t acc = inc - tot;
#pragma unroll
        for (int q = 0; q < per; q++) {
            s_cb[lane * per + q] = acc;
            acc += c[q];
        }
        if (lane == 31) {
            s_cb[kFlatWords] = inc;
            s_bal[kFlatWords] = 0u;
        }
    }
    __syncthreads();

    // 3. positions and copies, striped
    auto scan_at = [&](int y) {  // kept entries of the tile before position y (0 <= y <= T)
        const int q = y >> 5;
        return s_cb[q] + __popc(s_bal[q] & ((1u << (y & 31)) - 1u));
    };
    const int32_t fix = s_fp ? scan_at(s_re) : 0;
#pragma unroll
    for (int i = 0; i < kFlatPer; i++) {
        if (jn[i] < 0) continue;
        const int x = i * kBlock + tid;
        const int xs = s_start[x];
        int32_t p = s_raw[xs] - scan_at(xs) + scan_at(x);
        if (xs == 0) p -= fix;
        F.out_idx[p] = jn[i];
        F.out_val[p] = F.val[k0 + x];
    }
}

// kept row i's vectors to its new index p (sides shifted by the columns that
// left); renumbered: the columns' indices changed
__device__ __forceinline__ void rowvec_one(const Ctx &C, const CompactCtx &K, int32_t i, int32_t p, int32_t off,
                                           bool renumbered) {
    const double sh = K.shift[i];
    const double Lv = C.L[i], Uv = C.U[i];
    K.L2[p] = is_fin(Lv) ? Lv - sh : Lv;
    K.U2[p] = is_fin(Uv) ? Uv - sh : Uv;
    K.rmap2[p] = C.rmap[i];
    if (C.lp_row) K.lp_row2[p] = C.lp_row[i];
    K.rp2[p] = off;
    // a row that lost entries (fixed columns) changed: evaluate it next round;
    // its S5 key is taken again then, and an unchanged row's when columns were
    // dropped (the key hashes column indices, which the compaction renumbers)
    const bool lost = K.r_len[i] != C.A.ptr[i + 1] - C.A.ptr[i];
    K.rdirty2[p] = (uint8_t)((C.rdnext[i] | lost ? kEval : 0) | (lost | renumbered ? kRekey : 0));
    K.act2[p] = C.act[i];
    K.ninf2[p] = C.ninf[i];
    K.hrow2[p] = C.hrow[i];
}

// ---------------------------------------------------------- objective constant
// The contributions of tile t's columns, summed in a fixed order, and consumed:
// reset to zero once read (a column whose flags are not recomputed in a later
// round then contributes nothing).
__device__ __forceinline__ void offset_tile(double *contrib, int32_t n, double *part, int32_t t) {
    const int64_t base = (int64_t)t * kScanTile;
    double s = 0.0;
    for (int q = threadIdx.x; q < kScanTile; q += kBlock) {
        const int64_t j = base + q;
        if (j < n) {
            const double v = contrib[j];
            s += v;
            if (v != 0.0) contrib[j] = 0.0;
        }
    }
    s = block_sum_dbl(s);
    if (threadIdx.x == 0) part[t] = s;
}
// one block: thread t adds tiles t, t+256, ... in order, then the fixed-order block sum
__device__ __forceinline__ void offset_final(const double *part, int32_t ntiles, double *offset) {
    double s = 0.0;
    for (int32_t t = threadIdx.x; t < ntiles; t += kBlock) s += part[t];
    s = block_sum_dbl(s);
    if (threadIdx.x == 0) offset[0] += s;
}

}  // namespace

}  // namespace lpp
