// k_solo.cu -- all rounds of one LP in one cooperative kernel.
//
// A round of the launched path is some twenty kernels and two host reads; on
// an LP of up to a few hundred thousand entries each of them is latency (5 to
// 10 us), whatever the LP's size.  Here every round runs on the device: the
// blocks stay resident and the steps of a round, the bodies the round's kernels
// launch (phase_dev.cuh), are separated by grid barriers.  The control
// decisions (which steps run, whether to compact, whether to stop) are taken
// by every block alike from counters read after a barrier, as the host takes
// them in Engine::step, so an LP gets the bits of the launched path.  The rounds
// of a small LP take about half the launched time (kSoloNnz).
//
// The columns stay in place (Ctx::in_place); row vectors and matrix alternate
// between two buffers as there.  Counters exist twice, by the round's parity:
// the next round's are cleared after the first barrier of a round, when no
// block reads the previous round's any more.
#include <algorithm>

#include "../../include/lpp.h"
#include "lpp_launch.h"
#include "phase_dev.cuh"

namespace lpp {

namespace {

union PhaseShared {
    PropShared prop;
    InplaceShared rows;
    FlatShared flat;
};

struct SoloShared {
    Ctx C;
    CompactCtx K;
    int32_t cls[kNumClass];
    int32_t base[kNumClass], fill[kNumClass];  // the block's places per class
    int32_t w[2 * (kBlock / 32)], tot[2], before[2];
    int32_t pbase, kept;
    int32_t n2;
};

// sums of two ints over the block, to every thread
__device__ __forceinline__ int2 block_sum2(int32_t a, int32_t b, int32_t *s_w) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    a = __reduce_add_sync(0xffffffffu, a);
    b = __reduce_add_sync(0xffffffffu, b);
    __syncthreads();
    if (lane == 0) {
        s_w[warp] = a;
        s_w[kBlock / 32 + warp] = b;
    }
    __syncthreads();
    int2 t = make_int2(0, 0);
#pragma unroll
    for (int w = 0; w < kBlock / 32; w++) {
        t.x += s_w[w];
        t.y += s_w[kBlock / 32 + w];
    }
    return t;
}

// exclusive scan of two ints over the block; returns the totals
__device__ __forceinline__ int2 block_scan2(int32_t a, int32_t b, int32_t &ea, int32_t &eb, int32_t *s_w) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t xa = a, xb = b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t ya = __shfl_up_sync(0xffffffffu, xa, o), yb = __shfl_up_sync(0xffffffffu, xb, o);
        if (lane >= o) {
            xa += ya;
            xb += yb;
        }
    }
    __syncthreads();
    if (lane == 31) {
        s_w[warp] = xa;
        s_w[kBlock / 32 + warp] = xb;
    }
    __syncthreads();
    int2 t = make_int2(0, 0), p = make_int2(0, 0);
#pragma unroll
    for (int w = 0; w < kBlock / 32; w++) {
        if (w == warp) p = t;
        t.x += s_w[w];
        t.y += s_w[kBlock / 32 + w];
    }
    ea = p.x + xa - a;
    eb = p.y + xb - b;
    return t;
}

__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// rows [lo, hi) of a contiguous split of m rows over the grid, whole tiles of kBlock rows
__device__ __forceinline__ void row_range(int32_t m, int32_t &lo, int32_t &hi) {
    const int32_t tiles = (m + kBlock - 1) / kBlock, per = (tiles + gridDim.x - 1) / gridDim.x;
    const int64_t a = (int64_t)blockIdx.x * per * kBlock;
    lo = (int32_t)min((int64_t)m, a);
    hi = (int32_t)min((int64_t)m, a + (int64_t)per * kBlock);
}

// The block's count of new rows per class is in S.cls: reserves its places
// per class (S.base) among all blocks' in cls.  Every thread calls it.
__device__ __forceinline__ void reserve_classes(SoloShared &S, int32_t *cls) {
    __syncthreads();
    if (threadIdx.x < kNumClass) {
        const int32_t v = S.cls[threadIdx.x];
        S.base[threadIdx.x] = v ? atomicAdd(cls + threadIdx.x, v) : 0;
        S.fill[threadIdx.x] = 0;
    }
    __syncthreads();
}

// the rows [pb, pb + cnt) of ptr into order, by class (after a grid barrier on cls)
__device__ __forceinline__ void fill_order(SoloShared &S, const int32_t *cls, const int32_t *ptr, int32_t pb,
                                           int32_t cnt, int32_t *order) {
    const int lane = threadIdx.x & 31;
    int32_t start = 0;
    for (int32_t t0 = 0; t0 < cnt; t0 += kBlock) {
        const int32_t t = t0 + threadIdx.x;
        const bool in = t < cnt;
        const int c = in ? seg_class(ptr[pb + t + 1] - ptr[pb + t]) : kNumClass;
        const unsigned peers = __match_any_sync(0xffffffffu, c);
        const int first = __ffs(peers) - 1;
        int32_t at = 0;
        if (in && lane == first) at = atomicAdd(&S.fill[c], __popc(peers));
        at = __shfl_sync(0xffffffffu, at, first);
        if (in) {
            start = 0;
            for (int k = 0; k < c; k++) start += cls[k];
            order[start + S.base[c] + at + __popc(peers & ((1u << lane) - 1u))] = pb + t;
        }
    }
}

// block 0: the chunks of the long rows (class 6, in schedule order)
__device__ __forceinline__ void build_chunks(SoloShared &S, const int32_t *cls, const int32_t *ptr,
                                             const int32_t *order, Chunk *chunks, int32_t *lfirst, int32_t *nchunk) {
    int32_t start = 0;
    for (int k = 0; k < 6; k++) start += cls[k];
    const int32_t nlong = cls[6];
    int32_t carry = 0;
    for (int32_t t0 = 0; t0 < nlong; t0 += kBlock) {
        const int32_t t = t0 + threadIdx.x;
        int32_t sg = 0, pb = 0, pe = 0, v = 0, q, dummy;
        if (t < nlong) {
            sg = order[start + t];
            pb = ptr[sg];
            pe = ptr[sg + 1];
            v = (pe - pb + kChunk - 1) / kChunk;
        }
        const int2 tot = block_scan2(v, 0, q, dummy, S.w);
        if (t < nlong) {
            q += carry;
            lfirst[t] = q;
            for (int32_t k = pb; k < pe; k += kChunk, q++) chunks[q] = Chunk{sg, k, min(pe, k + kChunk), t};
        }
        carry += tot.x;
    }
    if (threadIdx.x == 0) {
        lfirst[nlong] = carry;
        *nchunk = carry;
    }
}

template <class F>
__device__ __forceinline__ void each_block(int32_t total, F &&f) {
    for (int32_t b = blockIdx.x; b < total; b += gridDim.x) {
        f(b);
        __syncthreads();  // the body's shared memory is reused
    }
}

__global__ void __launch_bounds__(kBlock, 2) k_solo(const __grid_constant__ SoloArgs F) {
    __shared__ SoloShared S;
    __shared__ PhaseShared P;
    const int tid = threadIdx.x;
    const int32_t gt = blockIdx.x * kBlock + tid, gstep = gridDim.x * kBlock;
    SoloCtl *ctl = F.ctl;
    if (*F.err_in) return;  // the input checks failed (the same for every block)
    int32_t m = F.m, nnz = F.nnz, cur = 0, nchunk = 0, rounds = 0, act_buf = 0, act_m = F.m;
    const int32_t n = F.n;
    uint8_t *rd = F.rdirty[0], *rd2 = F.rdirty[1], *rdnext = F.rdnext;
    const int32_t *rp = F.in_rp, *ci = F.in_ci;
    const double *rv = F.in_rv;
    bool s5_clean = false;
    long long s5_left = 0;
    int32_t status = LPP_OK, where = LPP_WHERE_NONE, vindex = -1, vround = 0;
    // every block takes the same branches, so each passes the same barriers
    unsigned gen = 0;
#define GRID_SYNC()                                                            \
    do {                                                                       \
        if (!grid_barrier(ctl->bar, &ctl->err, gen, &ctl->progress)) goto out; \
    } while (0)

    // the input's rows by class
    {
        int32_t lo, hi;
        row_range(m, lo, hi);
        if (tid < kNumClass) S.cls[tid] = 0;
        __syncthreads();
        for (int32_t i = lo + tid; i < hi; i += kBlock) atomicAdd(&S.cls[seg_class(rp[i + 1] - rp[i])], 1);
        reserve_classes(S, ctl->c[1].cls);
        GRID_SYNC();
        fill_order(S, ctl->c[1].cls, rp, lo, hi - lo, F.order);
        GRID_SYNC();
        if (ctl->c[1].cls[6] > 0) {
            if (blockIdx.x == 0) build_chunks(S, ctl->c[1].cls, rp, F.order, F.chunks, F.lfirst, &ctl->c[1].nchunk);
            GRID_SYNC();
        }
        nchunk = ctl->c[1].nchunk;
        __syncthreads();
        if (tid < kNumClass) S.cls[tid] = ctl->c[1].cls[tid];
        __syncthreads();
    }

    for (int32_t r = 1; r <= F.max_rounds; r++) {
        SoloCnt &N = ctl->c[r & 1], &X = ctl->c[(r & 1) ^ 1];
        const unsigned long long t0 = now_ns();
        const bool first = r == 1;
        const int nx = cur ^ 1;
        int32_t tcap = 2;
        while (tcap < 2 * (int64_t)m && tcap < F.tcap_max) tcap <<= 1;
        if (tid == 0) {
            Ctx &C = S.C;
            C = F.base;
            C.A.ptr = rp;
            C.A.idx = ci;
            C.A.val = rv;
            C.A.order = F.order;
            C.A.chunks = F.chunks;
            C.A.lfirst = F.lfirst;
            C.A.cnt = m;
            C.A.nchunks = nchunk;
            C.A.cls_start[0] = 0;
            for (int k = 0; k < kNumClass; k++) C.A.cls_start[k + 1] = C.A.cls_start[k] + S.cls[k];
            C.m = m;
            C.n = n;
            C.round = r;
            C.L = F.L[cur];
            C.U = F.U[cur];
            C.rmap = F.rmap[cur];
            C.act = F.act[cur];
            C.ninf = F.ninf[cur];
            C.hrow = F.hrow[cur];
            C.rdirty = rd;
            C.rdnext = rdnext;
            C.st = &N.st;
            C.tl_cnt = &N.tl_cnt;
            C.cl_cnt = &N.cl_cnt;
            C.cl_nnz = &N.cl_nnz;
            C.lp_changed = reinterpret_cast<uint8_t *>(&N.changed);
            C.tcap = tcap;
            C.s5_out = F.s5l[0];
            C.s5_out_cnt = &N.n1;
            C.list_touched = first ? 0 : 1;
            CompactCtx &K = S.K;
            K = F.K;
            K.rp2 = F.rp[nx];
            K.ci2 = F.ci[nx];
            K.rv2 = F.rv[nx];
            K.L2 = F.L[nx];
            K.U2 = F.U[nx];
            K.rmap2 = F.rmap[nx];
            K.act2 = F.act[nx];
            K.ninf2 = F.ninf[nx];
            K.hrow2 = F.hrow[nx];
            K.rdirty2 = rd2;
        }
        __syncthreads();
        const Ctx &C = S.C;
        const CompactCtx &K = S.K;
        rounds = r;
        act_buf = cur;
        act_m = m;
        const int32_t nlong = S.cls[6];
        const bool run_s5 = first || !s5_clean;

        // flags and the S5 table, beside S1-S3 (which touch neither)
        for (int32_t i = gt; i < m; i += gstep) rdnext[i] = 0;
        if (!first)
            for (int32_t j = gt; j < n; j += gstep) {
                C.ckind[j] = CK_KEPT;
                C.cchg[j] = 0;
            }
        if (run_s5)
            for (int32_t k = gt; k < tcap; k += gstep) {
                C.tkey[k] = 0ULL;
                C.tlead[k] = ~0ULL;
            }
        // S1-S3
        int32_t removed = 0, u0 = 0, u1 = 0;
        if (nlong > 0) each_block(nchunk, [&](int32_t b) { prop_long_chunk(C, b); });
        {
            const RowGrid R = prop_grid(C.A);
            each_block(R.g.blk_start[6], [&](int32_t b) { prop_block(C, R, b, P.prop, removed, u0, u1); });
        }
        GRID_SYNC();
        if (blockIdx.x == 0 && tid < (int)(sizeof(SoloCnt) / 4)) reinterpret_cast<int32_t *>(&X)[tid] = 0;
        if (nlong > 0) {
            for (int32_t t = gt >> 5; t < nlong; t += gstep >> 5) prop_long_row(C, t, removed, u0);
            GRID_SYNC();
            each_block(nchunk, [&](int32_t b) { prop_long_tighten(C, b, u1); });
            GRID_SYNC();
        }
        warp_add(removed, &N.st.rows_removed);
        removed = 0;
        if (C.dual_rec) {
            const RowGrid R = class_grid(C.A);
            each_block(R.g.blk_start[6], [&](int32_t b) { bsrc_block(C, R, b); });
            if (nlong > 0)
                each_block(nchunk, [&](int32_t b) {
                    const Chunk ch = C.A.chunks[b];
                    if (C.rdirty[ch.seg]) bsrc_row(C, ch.seg, ch.begin + tid, ch.end, kBlock);
                });
            GRID_SYNC();
        }
        // S3' + S4 on the columns, S5's insertion on the rows (independent)
        {
            int32_t changed = 0, fixed = 0, z = 0;
            if (first) {
                for (int32_t j = gt; j < n; j += gstep) colfin_one(C, j, true, changed, fixed, z);
            } else {
                const int32_t cnt = N.tl_cnt;
                for (int32_t t = gt; t < cnt; t += gstep) colfin_one(C, C.tl_list[t], false, changed, fixed, z);
            }
            __syncwarp();
            warp_add(changed, &N.st.bounds_changed);
            warp_add(fixed, &N.st.cols_fixed);
            if (run_s5)
                for (int32_t i = gt; i < m; i += gstep) {
                    int32_t slot = -1;
                    if (C.rkind[i] == RK_KEPT && rp[i + 1] - rp[i] >= 2) slot = s5_insert_row(C, i, (uint32_t)tcap);
                    C.rslot[i] = slot;
                    C.rwork[i] = slot >= 0 ? 1 : 0;
                }
        }
        GRID_SYNC();
        if (run_s5) {
            // first pass: every row against its leader
            int32_t um = 0;
            const RowGrid R = class_grid(C.A);
            each_block(R.g.blk_start[6], [&](int32_t b) {
                int c;
                bool valid;
                const int32_t i = class_row(C.A, R, b, c, valid);
                const bool left = match_class(C, c, i, valid, removed, um);
                const unsigned want = __ballot_sync(0xffffffffu, left);
                int32_t at = 0;
                if ((tid & 31) == 0 && want) at = atomicAdd(&N.n1, __popc(want));
                at = __shfl_sync(0xffffffffu, at, 0);
                if (left) F.s5l[0][at + __popc(want & ((1u << (tid & 31)) - 1u))] = i;
            });
            each_block(nlong, [&](int32_t t) { match_long(C, t, F.s5l[0], &N.n1, removed, um); });
            __syncwarp();
            warp_add(removed, &N.merged);
            removed = 0;
            GRID_SYNC();
            const int32_t n1 = N.n1;
            int32_t left = n1;
            if (n1 > 0 && F.par_max_iter > 1) {
                // the table empty again, then the later passes
                for (int32_t i = gt; i < m; i += gstep) {
                    const int32_t sl = C.rslot[i];
                    if (sl >= 0) {
                        C.tkey[sl] = 0ULL;
                        C.tlead[sl] = ~0ULL;
                    }
                }
                GRID_SYNC();
                if (!s5_later_passes(C, F.s5l[0], F.s5l[1], F.s5_cnt, 1, F.par_max_iter, left, removed, ctl->bar,
                                     &ctl->err, gen, &ctl->progress))
                    goto out;
                __syncwarp();
                warp_add(removed, &N.merged);
                removed = 0;
                if (gt == 0) N.n2 = left;
                GRID_SYNC();
                left = N.n2;
                for (int32_t q = gt; q < F.par_max_iter; q += gstep) F.s5_cnt[q] = 0;  // for the next round's passes
            }
            s5_clean = left == 0;
            s5_left += left;
            if (N.merged > 0)
                for (int32_t i = gt; i < m; i += gstep)
                    if (C.hasf[i]) s5_leader_one(C, i);
        }
        if (N.st.rows_removed + N.merged > 0) {
            if (!first) {  // the columns that may have become empty
                const RowGrid R = class_grid(C.A);
                each_block(R.g.blk_start[6], [&](int32_t b) { suspect_block(C, R, b); });
                if (nlong > 0) each_block(nchunk, [&](int32_t b) { suspect_chunk(C, b); });
            }
            GRID_SYNC();
        }
        {
            // the round's decisions, the same in every block
            // (verdicts are read here and after S6's barrier, not at the round's
            // end: another block may by then be in the next round's S2)
            int v = 0;
            while (v < V_SLOTS && C.verdict[v] == kNone) v++;
            const bool dead = v < V_SLOTS;
            const int32_t rows_removed = N.st.rows_removed + N.merged;
            const bool structural = first || rows_removed > 0 || N.st.cols_fixed > 0 || dead;
            const int32_t nnz0 = nnz;
            if (dead) {
                // the LP leaves empty: no rows, no columns, no contribution of the columns still in it
                for (int32_t j = gt; j < n; j += gstep)
                    if (C.cinv[j] >= 0) {
                        K.contrib[j] = 0.0;
                        K.cinv[j] = -1;
                    }
                if (blockIdx.x == 0 && tid == 0) K.rp2[0] = 0;
                m = 0;
                nnz = 0;
                cur = nx;
            } else if (structural) {
                const RowGrid R = class_grid(C.A);
                each_block(R.g.blk_start[6], [&](int32_t b) { inplace_block<true>(C, K, R, b, P.rows); });
                if (nlong > 0) each_block(nchunk, [&](int32_t b) { inplace_chunk<true>(C, K, b); });
                GRID_SYNC();
                if (nlong > 0)
                    for (int32_t t = gt >> 5; t < nlong; t += gstep >> 5)
                        long_prefix(C.A, t, K.chr_cnt, K.chr_off, K.r_len, K.chr_shift, K.shift);
                int32_t fixed = 0;
                for (int32_t j = gt; j < n; j += gstep) fixed += colkeep_in_place(C, K, j);
                __syncwarp();
                warp_add(fixed, &N.st.cols_fixed);
                if (nlong > 0) GRID_SYNC();
                // new rows and offsets: the blocks' sums, then each block's own scan
                int32_t lo, hi;
                row_range(m, lo, hi);
                int32_t ka = 0, la = 0;
                for (int32_t i = lo + tid; i < hi; i += kBlock) {
                    ka += K.r_keep[i];
                    la += K.r_keep[i] ? K.r_len[i] : 0;
                }
                int2 bt = block_sum2(ka, la, S.w);
                if (tid == 0) {
                    F.btot[2 * blockIdx.x] = bt.x;
                    F.btot[2 * blockIdx.x + 1] = bt.y;
                }
                GRID_SYNC();
                while (v > 0 && C.verdict[v - 1] != kNone) v--;  // S6's slot is the last
                ka = la = 0;
                int32_t ta = 0, tb = 0;
                for (int32_t b = tid; b < (int32_t)gridDim.x; b += kBlock) {
                    const int32_t x = F.btot[2 * b], y = F.btot[2 * b + 1];
                    ta += x;
                    tb += y;
                    if (b < (int32_t)blockIdx.x) {
                        ka += x;
                        la += y;
                    }
                }
                const int2 all = block_sum2(ta, tb, S.w), pre = block_sum2(ka, la, S.w);
                __syncthreads();
                if (tid < kNumClass) S.cls[tid] = 0;
                __syncthreads();
                int32_t pos = pre.x, off = pre.y;
                for (int32_t t0 = lo; t0 < hi; t0 += kBlock) {
                    const int32_t i = t0 + tid;
                    const bool kp = i < hi && K.r_keep[i];
                    const int32_t ln = kp ? K.r_len[i] : 0;
                    int32_t ea, eb;
                    const int2 tt = block_scan2(kp ? 1 : 0, ln, ea, eb, S.w);
                    if (i < hi) K.r_off[i] = off + eb;
                    if (kp) {
                        rowvec_one(C, K, i, pos + ea, off + eb, false);
                        atomicAdd(&S.cls[seg_class(ln)], 1);
                    }
                    pos += tt.x;
                    off += tt.y;
                }
                if (blockIdx.x == 0 && tid == 0) K.rp2[all.x] = all.y;
                reserve_classes(S, X.cls);
                GRID_SYNC();
                // the kept entries, and the new rows by class
                {
                    const int32_t ntiles = (int32_t)(((int64_t)nnz + kFlatTile - 1) / kFlatTile);
                    const FlatArgs fa{rp, ci, rv, nnz, m, ntiles, K.r_keep, K.r_off, K.r_len, K.r_ch0,
                                      K.chr_off, K.chr_cnt, K.c_new, C.cchg, K.tile_a, K.ci2, K.rv2};
                    each_block(ntiles, [&](int32_t b) { flat_tile(fa, b, P.flat); });
                }
                fill_order(S, X.cls, K.rp2, pre.x, pos - pre.x, F.order);
                GRID_SYNC();
                if (X.cls[6] > 0) {
                    if (blockIdx.x == 0) build_chunks(S, X.cls, K.rp2, F.order, F.chunks, F.lfirst, &X.nchunk);
                    GRID_SYNC();
                }
                nchunk = X.nchunk;
                __syncthreads();
                if (tid < kNumClass) S.cls[tid] = X.cls[tid];
                m = all.x;
                nnz = all.y;
                cur = nx;
                rp = F.rp[nx];
                ci = F.ci[nx];
                rv = F.rv[nx];
                uint8_t *t = rd;
                rd = rd2;
                rd2 = t;
            } else {
                if (N.st.bounds_changed > 0) {
                    const RowGrid R = class_grid(C.A);
                    each_block(R.g.blk_start[6], [&](int32_t b) { inplace_block<false>(C, K, R, b, P.rows); });
                    if (nlong > 0) each_block(nchunk, [&](int32_t b) { inplace_chunk<false>(C, K, b); });
                }
                GRID_SYNC();
                uint8_t *t = rd;
                rd = rdnext;
                rdnext = t;
            }
            if (N.st.cols_fixed > 0) s5_clean = false;  // rows lost entries
            if (blockIdx.x == 0 && tid == 0) {
                int32_t *q = F.rstat + 6 * (int64_t)(r - 1);
                q[0] = nnz0;
                q[1] = rows_removed;
                q[2] = N.st.cols_fixed;
                q[3] = N.st.bounds_changed;
                q[4] = (int32_t)(now_ns() - t0);
                if (N.st.err) atomicOr(&ctl->err, N.st.err);
            }
            if (v < V_SLOTS) {
                status = v == V_S6_COL ? LPP_UNBOUNDED : LPP_INFEASIBLE;
                where = (v == V_S2_ROW || v == V_S5_ROW) ? LPP_WHERE_ROW : LPP_WHERE_COL;
                vindex = C.verdict[v];
                vround = r;
                break;
            }
        }
        if (!N.changed) break;
        __syncthreads();  // every thread has read S before the next round rewrites it
    }
out:
    if (blockIdx.x == 0 && tid == 0) {
        SoloOut &o = ctl->out;
        o.status = status;
        o.where = where;
        o.index = vindex;
        o.round = vround;
        o.rounds = rounds;
        o.m = m;
        o.nnz = nnz;
        o.cur = cur;
        o.act_buf = act_buf;
        o.act_m = act_m;
        o.s5_left = s5_left;
    }
#undef GRID_SYNC
}

// ------------------------------------------------------------- after the rounds
// The steps of Engine::finish_cols and finish_csc (offset, keep flags and their
// scan, vectors, renumbering; rows of the entries, radix passes, gather, column
// pointers: some twenty launches of 3 to 9 us) with four to eight grid barriers
// of 1 to 2 us between them.  Each block keeps a contiguous range of entries,
// so a pass needs one table of 256 counts per block, and each block adds up the
// tables before its own (no separate scan).  The keys are the column slots: the
// compaction keeps their order, so they sort before the new indices are known,
// and the columns' compaction shares the first pass's barriers.  The last pass
// writes row and value, not key and payload, so no gather follows.
// Launched, these steps made calls on 20 k rows 2 to 3% longer.
constexpr int kFinTile = 2048;               // entries a block sorts at a time
constexpr int kFinWarps = kBlock / 32;
constexpr int kFinChunk = kFinTile / kFinWarps;
constexpr int kFinSteps = kFinChunk / 32;

struct FinShared {
    int32_t wh[kFinWarps][256], dbase[256], goff[256], wsum[kFinWarps];
    uint32_t k[kFinTile];
    int32_t v[kFinTile];
};

// last i in [lo, hi] with ptr[i] <= k (ptr[lo] <= k): the row that holds entry k
__device__ __forceinline__ int32_t row_holding(const int32_t *ptr, int32_t lo, int32_t hi, int32_t k) {
    while (lo < hi) {
        const int32_t mid = lo + (hi - lo + 1) / 2;
        if (ptr[mid] <= k) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// counts of the digits of keys [e0, e1) into the block's row of hist
__device__ __forceinline__ void fin_hist(FinShared &S, const uint32_t *keys, int32_t e0, int32_t e1, int shift,
                                         int32_t *hist) {
    static_assert(kBlock == 256, "a thread per digit");
    __syncthreads();
    S.dbase[threadIdx.x] = 0;
    __syncthreads();
    for (int32_t k = e0 + threadIdx.x; k < e1; k += kBlock) atomicAdd(&S.dbase[(keys[k] >> shift) & 255u], 1);
    __syncthreads();
    hist[blockIdx.x * 256 + threadIdx.x] = S.dbase[threadIdx.x];
}

// one stable pass over [e0, e1): to key/payload, or (last) to key, row and value
__device__ __forceinline__ void fin_scatter(FinShared &S, const uint32_t *kin, const int32_t *vin, bool first,
                                            bool last, int32_t e0, int32_t e1, int shift, const int32_t *hist,
                                            uint32_t *kout, int32_t *vout, const int32_t *row_of, const double *val,
                                            int32_t *tidx, double *tval) {
    const int d0 = threadIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the digit's place: all entries of smaller digits, its entries in earlier blocks
    int32_t tot = 0, before = 0;
#pragma unroll 8
    for (int32_t b = 0; b < (int32_t)gridDim.x; b++) {
        const int32_t v = hist[b * 256 + d0];
        tot += v;
        before += b < (int32_t)blockIdx.x ? v : 0;
    }
    int32_t inc = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    __syncthreads();
    if (lane == 31) S.wsum[warp] = inc;
    __syncthreads();
    int32_t pre = inc - tot;
    for (int w = 0; w < warp; w++) pre += S.wsum[w];
    S.goff[d0] = pre + before;
    for (int32_t base = e0; base < e1; base += kFinTile) {
        __syncthreads();
        for (int w = 0; w < kFinWarps; w++) S.wh[w][d0] = 0;
        __syncthreads();
        int32_t rk[kFinSteps];
        uint32_t ky[kFinSteps];
#pragma unroll
        for (int i = 0; i < kFinSteps; i++) {
            const int32_t k = base + warp * kFinChunk + i * 32 + lane;
            ky[i] = k < e1 ? kin[k] : 0u;
        }
#pragma unroll
        for (int i = 0; i < kFinSteps; i++) {
            const int32_t k = base + warp * kFinChunk + i * 32 + lane;
            const int d = k < e1 ? (int)((ky[i] >> shift) & 255u) : 256;
            const unsigned peers = digit_peers(d);
            const int run = d < 256 ? S.wh[warp][d] : 0;
            rk[i] = run + __popc(peers & ((1u << lane) - 1u));
            __syncwarp();
            if (d < 256 && lane == __ffs(peers) - 1) S.wh[warp][d] = run + __popc(peers);
            __syncwarp();
        }
        __syncthreads();
        int32_t cnt = 0;  // warps in order, then the tile's digits in order
        for (int w = 0; w < kFinWarps; w++) {
            const int32_t c = S.wh[w][d0];
            S.wh[w][d0] = cnt;
            cnt += c;
        }
        int32_t ti = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += y;
        }
        if (lane == 31) S.wsum[warp] = ti;
        __syncthreads();
        int32_t db = ti - cnt;
        for (int w = 0; w < warp; w++) db += S.wsum[w];
        S.dbase[d0] = db;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kFinSteps; i++) {
            const int32_t k = base + warp * kFinChunk + i * 32 + lane;
            if (k < e1) {
                const int d = (int)((ky[i] >> shift) & 255u);
                const int32_t q = S.dbase[d] + S.wh[warp][d] + rk[i];
                S.k[q] = ky[i];
                S.v[q] = first ? k : vin[k];
            }
        }
        __syncthreads();
        const int32_t nt = min(e1 - base, kFinTile);
        for (int32_t q = threadIdx.x; q < nt; q += kBlock) {
            const uint32_t kk = S.k[q];
            const int d = (int)((kk >> shift) & 255u);
            const int32_t g = S.goff[d] + (q - S.dbase[d]);
            const int32_t e = S.v[q];
            kout[g] = kk;
            if (last) {
                tidx[g] = row_of[e];
                tval[g] = val[e];
            } else {
                vout[g] = e;
            }
        }
        __syncthreads();
        S.goff[d0] += cnt;
    }
}

__global__ void __launch_bounds__(kBlock) k_solo_finish(const __grid_constant__ SoloFinish F) {
    __shared__ FinShared S;
    __shared__ int32_t s_w[2 * kFinWarps], s_r[2];
    const int tid = threadIdx.x;
    const int32_t gt = blockIdx.x * kBlock + tid, gstep = gridDim.x * kBlock;
    SoloCtl *ctl = F.ctl;
    if (*F.err_in || ctl->err) return;  // before the first barrier, the same for every block
    const int32_t n = F.n, m = ctl->out.m, nnz = ctl->out.nnz, cur = ctl->out.cur, nx = cur ^ 1;
    const int32_t *rp = F.rp[cur];
    int32_t *ci = F.ci[cur], *row_of = reinterpret_cast<int32_t *>(F.tv[nx]);
    const double *rv = F.rv[cur];
    uint32_t *kbuf[2] = {reinterpret_cast<uint32_t *>(F.ci[nx]), reinterpret_cast<uint32_t *>(F.ti[nx])};
    int32_t *vbuf[2] = {reinterpret_cast<int32_t *>(F.rv[nx]), reinterpret_cast<int32_t *>(F.rv[nx]) + F.half};
    int32_t *tp = F.tp[cur], *tidx = F.ti[cur];
    double *tval = F.tv[cur];
    const int32_t ctiles = (int32_t)(((int64_t)n + kScanTile - 1) / kScanTile);
    // the block's entries: whole tiles
    const int32_t tiles = (nnz + kFinTile - 1) / kFinTile, per = (tiles + gridDim.x - 1) / gridDim.x;
    const int32_t e0 = (int32_t)min((int64_t)nnz, (int64_t)blockIdx.x * per * kFinTile);
    const int32_t e1 = (int32_t)min((int64_t)nnz, (int64_t)e0 + (int64_t)per * kFinTile);
    int32_t lo, hi;
    row_range(n, lo, hi);
    int passes = 1;
    while (passes < 4 && (int64_t)n > (int64_t)1 << (8 * passes)) passes++;
    unsigned gen = 0;
#define GRID_SYNC()                                             \
    do {                                                        \
        if (!grid_barrier(ctl->bar + 1, &ctl->err, gen)) return; \
    } while (0)
    each_block(ctiles, [&](int32_t b) { offset_tile(F.contrib, n, F.part, b); });
    {
        int32_t alive = 0;
        for (int32_t j = lo + tid; j < hi; j += kBlock) alive += F.cinv[j] >= 0;
        const int2 t = block_sum2(alive, 0, s_w);
        if (tid == 0) F.btot[blockIdx.x] = t.x;
    }
    if (e0 < e1) {  // the entries' rows: searched between those of the block's first and last
        if (tid < 2) s_r[tid] = row_holding(rp, 0, m - 1, tid ? e1 - 1 : e0);
        __syncthreads();
        for (int32_t k = e0 + tid; k < e1; k += kBlock) row_of[k] = row_holding(rp, s_r[0], s_r[1], k);
    }
    fin_hist(S, reinterpret_cast<const uint32_t *>(ci), e0, e1, 0, F.hist);
    GRID_SYNC();
    int32_t nleft = 0;
    {
        if (blockIdx.x == 0 && n > 0) offset_final(F.part, ctiles, F.offset);
        int32_t a = 0, b = 0;
        for (int32_t q = tid; q < (int32_t)gridDim.x; q += kBlock) {
            const int32_t v = F.btot[q];
            a += v;
            b += q < (int32_t)blockIdx.x ? v : 0;
        }
        const int2 t = block_sum2(a, b, s_w);
        nleft = t.x;
        int32_t p0 = t.y;
        for (int32_t j0 = lo; j0 < hi; j0 += kBlock) {
            const int32_t j = j0 + tid;
            const bool on = j < hi && F.cinv[j] >= 0;
            int32_t e, unused;
            const int2 tt = block_scan2(on ? 1 : 0, 0, e, unused, s_w);
            if (on) {  // cmap[j] is j: the slots are the input's columns
                const int32_t q = p0 + e;
                F.pos[j] = q;
                F.lu2[q] = F.lu[j];
                F.c2[q] = F.c[j];
                F.cmap2[q] = F.cmap[j];
                F.cinv[j] = q;
            }
            p0 += tt.x;
        }
    }
    const uint32_t *kin = reinterpret_cast<const uint32_t *>(ci);
    const int32_t *vin = nullptr;
    for (int p = 0; p < passes; p++) {
        if (p > 0) {
            fin_hist(S, kin, e0, e1, 8 * p, F.hist);
            GRID_SYNC();
        }
        fin_scatter(S, kin, vin, p == 0, p == passes - 1, e0, e1, 8 * p, F.hist, kbuf[p & 1], vbuf[p & 1], row_of, rv,
                    tidx, tval);
        kin = kbuf[p & 1];
        vin = vbuf[p & 1];
        GRID_SYNC();
    }
    // new column indices, and where each column begins among the sorted keys
    for (int32_t k = gt; k < nnz; k += gstep) {
        ci[k] = F.pos[ci[k]];
        const int32_t kp = F.pos[kin[k]], kq = k == 0 ? -1 : F.pos[kin[k - 1]];
        for (int32_t j = kq + 1; j <= kp; j++) tp[j] = k;
    }
    const int32_t last = nnz > 0 ? F.pos[kin[nnz - 1]] : -1;
    for (int32_t j = last + 1 + gt; j <= nleft; j += gstep) tp[j] = nnz;
    if (blockIdx.x == 0 && tid == 0) {
        ctl->out.n = nleft;
        ctl->out.offset = *F.offset;
    }
#undef GRID_SYNC
}

}  // namespace

// blocks of a cooperative launch of k_solo for an LP of these sizes, 0 if the
// current device cannot take it or that of k_solo_finish: a block per 512 entries, which spreads the longer rows
// (a block or a warp each) over the SMs.  With 2048, 1024, 512 and 256 entries per
// block a presolve takes, in us: 500 skewed rows 1401, 1036, 857, 801; 5,000 rows
// 1047, 905, 850, 858; 20,000 rows 1299, 1162, 1163, 1165; 100,000 rows the same.
// One slot in 32 stays free: two of these blocks hold all registers of an SM, and
// no other stream's kernels or copies ran until a grid that held every SM twice
// had ended.  A server's submissions then waited for the request being presolved,
// its queue stayed short, and 80 requests of 0.55 M entries were presolved one by
// one: 108 ms, batched 60.  An LP of 1.9 M entries alone takes 1.80 ms for 1.78.
// Presolves in flight at once (share) get a part of the slots each: a grid that
// fills the device waits for all of it, and they would run one after the other.
// 20,000 rows from eight threads took four times as long.
int solo_blocks(int32_t m, int32_t n, int64_t nnz, int share) {
    static CoopCache cache;
    int most = solo_finish_blocks(n, nnz) > 0 ? coop_blocks((const void *)k_solo, cache) : 0;
    if (most > 0) most = std::max(1, (most - most / 32) / share);
    const int64_t want = std::max<int64_t>({1, ((int64_t)m + kBlock - 1) / kBlock, ((int64_t)n + 2 * kBlock - 1) / (2 * kBlock),
                                            (nnz + 2 * kBlock - 1) / (2 * kBlock)});
    return (int)std::min<int64_t>(want, most);
}
// of k_solo_finish: a tile of entries or two of columns each, one per SM at
// most (more read more tables of counts)
int solo_finish_blocks(int32_t n, int64_t nnz, int share) {
    static CoopCache cache;
    int sms = 0;
    int most = std::min(coop_blocks((const void *)k_solo_finish, cache, &sms), sms);
    if (most > 0) most = std::max(1, most / share);
    const int64_t want = std::max<int64_t>({1, (nnz + kFinTile - 1) / kFinTile, ((int64_t)n + 2 * kBlock - 1) / (2 * kBlock)});
    return (int)std::min<int64_t>(want, most);
}

bool launch_solo(const SoloArgs &F, int blocks, cudaStream_t s) {
    SoloArgs Fv = F;
    void *args[] = {&Fv};
    if (cudaLaunchCooperativeKernel((const void *)k_solo, dim3(blocks), dim3(kBlock), args, 0, s) != cudaSuccess) return false;
    note_launch();
    return true;
}
bool launch_solo_finish(const SoloFinish &F, int blocks, cudaStream_t s) {
    SoloFinish Fv = F;
    void *args[] = {&Fv};
    if (cudaLaunchCooperativeKernel((const void *)k_solo_finish, dim3(blocks), dim3(kBlock), args, 0, s) != cudaSuccess)
        return false;
    note_launch();
    return true;
}

}  // namespace lpp
