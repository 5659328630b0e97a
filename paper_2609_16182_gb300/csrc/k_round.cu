// k_round.cu -- the kernels of one presolve round up to compaction:
//   S1 activities, S2 row classes, S3 implied bounds (fused, one pass over the
//   CSR), S3'/S4 bound finalisation and fixing, S5 parallel rows.
//
// Load balance (Sec. 3.1, "length-based load balancing"): rows are grouped
// by length class.  S1-S3 give a row of up to 16 entries one lane, up to 32 and
// 64 two and four (prop_lanes), up to 256 a warp and up to 4096 a block; the other
// steps give class c <= 5 a group of W = 2^c lanes of a warp (lane t walks entries
// t, t+W, ...; the group then reduces with an xor butterfly).  Class 6 (more than
// 4096 entries) splits the row into chunks of 4096 entries, one thread block
// each, whose partial results are combined in chunk order.  The order of every
// floating-point sum depends only on the row's own length.
//
// Bound tightening follows Sec. 3.1 in Jacobi form: activities and the
// acceptance tests read the bounds of the round start, accepted implied
// bounds are combined with atomicMin / atomicMax on an order-preserving
// integer encoding, which is exact and independent of the order of updates.
//
// FP64 is scarce on this GPU (about two DFMA per SM and clock), so every
// per-entry sign, finiteness and max(1,|x|) test runs on integer pipes, the
// activity sums are fused multiply-adds, and an implied bound is divided out
// only after an exact FMA sign test (x - thr*a) says it will be accepted.
#include <algorithm>

#include "lpp_launch.h"
#include "phase_dev.cuh"

namespace lpp {

namespace {

// The round's flags and counters to zero: the status counters, the per-LP
// changed flags, the column lists' sizes, the next dirty flags and (outside a
// first round, whose S3' writes every column's) the columns' kinds and states.
__global__ void __launch_bounds__(kBlock) k_round_start(Ctx C, int32_t cols) {
    const int64_t t = (int64_t)blockIdx.x * kBlock + threadIdx.x, step = (int64_t)gridDim.x * kBlock;
    if (t < 8) reinterpret_cast<int32_t *>(C.st)[t] = 0;
    if (t < 3) C.tl_cnt[t] = 0;
    for (int64_t k = t; k < C.nlp; k += step) C.lp_changed[k] = 0;
    // flag arrays start 256-byte aligned
    auto zero = [&](uint8_t *p, int64_t cnt) {
        for (int64_t k = t; k < cnt / 16; k += step) reinterpret_cast<uint4 *>(p)[k] = make_uint4(0, 0, 0, 0);
        if (t < (cnt & 15)) p[cnt / 16 * 16 + t] = 0;
    };
    zero(C.rdnext, C.m);
    if (cols) {
        zero(C.ckind, C.n);
        zero(C.cchg, C.n);
    }
}

// an empty S5 table of cap slots; passes (if not 0): the pass sizes' array, zeroed
__global__ void __launch_bounds__(kBlock) k_s5_init(unsigned long long *tkey, unsigned long long *tlead, int32_t cap,
                                                    int32_t *cnt, int32_t passes) {
    const int64_t t = (int64_t)blockIdx.x * kBlock + threadIdx.x, step = (int64_t)gridDim.x * kBlock;
    for (int64_t k = t; k < cap / 2; k += step) {  // capacities are powers of two >= 2
        reinterpret_cast<ulonglong2 *>(tkey)[k] = make_ulonglong2(0ULL, 0ULL);
        reinterpret_cast<ulonglong2 *>(tlead)[k] = make_ulonglong2(~0ULL, ~0ULL);
    }
    for (int64_t k = t; k < passes; k += step) cnt[k] = 0;
}

__global__ void __launch_bounds__(kBlock, 4) k_prop_groups(Ctx C, RowGrid R) {
    __shared__ PropShared S;
    int32_t removed = 0, evaluated = 0, tested = 0;
    prop_block(C, R, blockIdx.x, S, removed, evaluated, tested);
    warp_add(removed, &C.st->rows_removed);
    if (C.count_work) {  // statistics of a timed run only
        warp_add(evaluated, &C.st->nnz_eval);
        warp_add(tested, &C.st->sides_tested);
    }
}

// ------------------------------------------------------------ long rows
__global__ void __launch_bounds__(kBlock) k_prop_long_partial(Ctx C) { prop_long_chunk(C, blockIdx.x); }

__global__ void __launch_bounds__(kBlock) k_prop_long_combine(Ctx C) {
    int32_t removed = 0, evaluated = 0;
    prop_long_row(C, (int32_t)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), removed, evaluated);
    warp_add(removed, &C.st->rows_removed);
    if (C.count_work) warp_add(evaluated, &C.st->nnz_eval);
}

__global__ void __launch_bounds__(kBlock) k_prop_long_tighten(Ctx C) {
    int32_t tested = 0;
    prop_long_tighten(C, blockIdx.x, tested);
    if (C.count_work) warp_add(tested, &C.st->sides_tested);
}

__global__ void __launch_bounds__(kBlock) k_bsrc_groups(Ctx C, RowGrid R) { bsrc_block(C, R, blockIdx.x); }

// the chunks of the long rows, a block per chunk
__global__ void __launch_bounds__(kBlock) k_bsrc_chunks(Ctx C) {
    const Chunk ch = C.A.chunks[blockIdx.x];
    if (C.rdirty[ch.seg] == 0) return;
    bsrc_row(C, ch.seg, ch.begin + threadIdx.x, ch.end, kBlock);
}

// ---------------------------------------- dependent equality rows (Sec. 5)
// the rows the host found dependent leave with their records (the row kinds
// of every other row were reset to kept before)
__global__ void __launch_bounds__(kBlock) k_mark_dependent(Ctx C, const int32_t *list, int32_t cnt) {
    const int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= cnt) return;
    const int32_t i = list[t];
    C.rkind[i] = RK_DEPENDENT;
    const int32_t o = C.rmap[i];
    C.rec_rk[o] = RK_DEPENDENT;
    C.rec_rr[o] = C.round;
    C.rec_ra[o] = -1;
    C.rec_rv[o] = 0.0;
}

// ------------------------------------------------- S3' finalise + S4 fixing
// every column (some LP in its first round)
// (grid-stride over a grid of at most 8 blocks per SM: the block sums run
// once per block, not once per 256 columns)
__global__ void __launch_bounds__(kBlock) k_colfin(Ctx C) {
    int32_t changed = 0, fixed = 0, chg_nnz = 0;
    for (int32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < C.n; j += gridDim.x * blockDim.x)
        colfin_one(C, j, true, changed, fixed, chg_nnz);
    block_add(changed, &C.st->bounds_changed);
    block_add(fixed, &C.st->cols_fixed);
    block_add(chg_nnz, C.cl_nnz);
}

// the columns that received a candidate (the others keep their bounds; their
// kind and change flag were reset at the start of the round)
__global__ void __launch_bounds__(kBlock) k_colfin_list(Ctx C) {
    const int32_t cnt = *C.tl_cnt;
    int32_t changed = 0, fixed = 0, chg_nnz = 0;
    for (int32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += gridDim.x * blockDim.x)
        colfin_one(C, C.tl_list[t], false, changed, fixed, chg_nnz);
    block_add(changed, &C.st->bounds_changed);
    block_add(fixed, &C.st->cols_fixed);
    block_add(chg_nnz, C.cl_nnz);
}

// ------------------------------------------------------------ S5 parallel rows
// first pass: rows kept by S2 with >= 2 entries take part
// (grid-stride, one block sum per block)
__global__ void __launch_bounds__(kBlock) k_s5_insert(Ctx C) {
    int32_t part = 0;
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < C.m; i += gridDim.x * blockDim.x) {
        int32_t slot = -1;
        if (C.rkind[i] == RK_KEPT && C.A.ptr[i + 1] - C.A.ptr[i] >= 2) slot = s5_insert_row(C, i, (uint32_t)C.tcap);
        C.rslot[i] = slot;
        C.rwork[i] = slot >= 0 ? 1 : 0;
        part += slot >= 0;
    }
    block_add(part, &C.st->participants);
}

__global__ void __launch_bounds__(kBlock) k_s5_match_groups(Ctx C, RowGrid R) {
    int32_t removed = 0, unmatched = 0;
    int c;
    bool valid;
    const int32_t i = class_row(C.A, R, blockIdx.x, c, valid);
    const bool left = match_class(C, c, i, valid, removed, unmatched);
    block_add(removed, &C.st->rows_removed);
    block_add(unmatched, &C.st->unmatched);
    block_append(left, i, C.s5_out_cnt, C.s5_out);
}

__global__ void __launch_bounds__(kBlock) k_s5_match_long(Ctx C) {
    int32_t removed = 0, unmatched = 0;
    match_long(C, blockIdx.x, C.s5_out, C.s5_out_cnt, removed, unmatched);
    warp_add(removed, &C.st->rows_removed);
    warp_add(unmatched, &C.st->unmatched);
}

// Later passes run on the list of rows the previous pass left unmatched
// (count *cnt, at most the launch's grid): insert, match against the new
// leader (one warp per row; unmatched rows go to the next list), then clear
// the slots used so that the table is empty for the next pass.  The table
// capacity of a pass is the power of two >= 2 * count, at most C.tcap.
__global__ void __launch_bounds__(kBlock) k_s5_tail_insert(Ctx C, const int32_t *list, const int32_t *cnt) {
    const int32_t n = *cnt;
    const int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int32_t i = list[t];
    C.rslot[i] = s5_insert_row(C, i, s5_tail_cap(C, n));
}

// one thread per listed row; rows longer than 32 entries are checked by the
// whole warp in turn
__global__ void __launch_bounds__(kBlock) k_s5_tail_match(Ctx C, const int32_t *list, const int32_t *cnt,
                                                         int32_t *out, int32_t *out_cnt) {
    const int32_t n = *cnt;
    const int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    int32_t removed, i;
    bool left;
    s5_tail_match_one(C, list, n, t, removed, left, i);
    block_add(removed, &C.st->rows_removed);
    block_append(left, i, out_cnt, out);
}

__global__ void __launch_bounds__(kBlock) k_s5_tail_clear(Ctx C, const int32_t *list, const int32_t *cnt) {
    const int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= *cnt) return;
    const int32_t sl = C.rslot[list[t]];
    if (sl >= 0) {
        C.tkey[sl] = 0ULL;
        C.tlead[sl] = ~0ULL;
    }
}

// All remaining later passes in one block, for a short list: the passes
// above (insert, match, clear) separated by block barriers instead of
// launches, with no host read between them.  Starts at pass p0 from list
// lists[(p0 - 1) & 1] of cnt[p0] rows, runs passes p0 .. max_iter - 1 (fewer
// once no row is left) and writes the rows left after the last one to
// cnt[max_iter].  The next list of a pass is written in the order the rows
// are left (unspecified, as in the launched form; the leaders of a pass do
// not depend on it).
constexpr int kTailBlock = 1024;
__global__ void __launch_bounds__(kTailBlock) k_s5_tail_block(Ctx C, int32_t *l0, int32_t *l1, int32_t *cnt,
                                                              int32_t p0, int32_t max_iter) {
    __shared__ int32_t s_n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int32_t n = cnt[p0], from = (p0 - 1) & 1, rem = 0;
    for (int32_t p = p0; p < max_iter && n > 0; p++) {
        const int32_t *lst = from ? l1 : l0;
        int32_t *nxt = from ? l0 : l1;
        const uint32_t cap = s5_tail_cap(C, n);
        for (int32_t t = tid; t < n; t += kTailBlock) C.rslot[lst[t]] = s5_insert_row(C, lst[t], cap);
        if (tid == 0) s_n = 0;
        __syncthreads();
        for (int32_t tb = warp * 32; tb < n; tb += kTailBlock) {  // warp-uniform: every lane calls the match
            int32_t rm, i;
            bool left;
            s5_tail_match_one(C, lst, n, tb + lane, rm, left, i);
            rem += rm;
            if (left) nxt[atomicAdd(&s_n, 1)] = i;
        }
        __syncthreads();
        for (int32_t t = tid; t < n; t += kTailBlock) {
            const int32_t sl = C.rslot[lst[t]];
            if (sl >= 0) {
                C.tkey[sl] = 0ULL;
                C.tlead[sl] = ~0ULL;
            }
        }
        __syncthreads();
        n = s_n;
        from ^= 1;
        __syncthreads();  // every thread has read s_n before the next pass resets it
    }
    block_add(rem, &C.st->rows_removed);
    if (tid == 0) cnt[max_iter] = n;
}

// All remaining later passes of a long list in one cooperative launch (every
// block resident; s5_later_passes).  Same starting point and result slot as
// k_s5_tail_block.
__global__ void __launch_bounds__(kBlock) k_s5_tail_grid(Ctx C, int32_t *l0, int32_t *l1, int32_t *cnt, int32_t p0,
                                                        int32_t max_iter, unsigned *bar) {
    int32_t n = __ldcg(cnt + p0), rem = 0;
    unsigned gen = 0;
    const bool ok = s5_later_passes(C, l0, l1, cnt + 1, p0, max_iter, n, rem, bar, &C.st->err, gen);
    block_add(rem, &C.st->rows_removed);
    if (blockIdx.x == 0 && threadIdx.x == 0 && ok) cnt[max_iter] = n;
}

__global__ void __launch_bounds__(kBlock) k_s5_leader(Ctx C) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= C.m || !C.hasf[i]) return;
    s5_leader_one(C, i);
}

// rows of the changed short columns need their activities next round: one
// thread per listed column; columns longer than 32 entries are walked by the
// whole warp in turn.  When the changed columns hold at least an eighth of the
// nonzeros, every row is marked instead (re-evaluating a row whose inputs did
// not change finds nothing new).
__global__ void __launch_bounds__(kBlock) k_mark_list(Ctx C, int64_t nnz) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if (8 * (int64_t)*C.cl_nnz >= nnz) {
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < C.m; i += stride) C.rdnext[i] = 1;
        return;
    }
    const int32_t cnt = *C.cl_cnt;
    const int lane = threadIdx.x & 31;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < cnt; base += stride) {
        const int64_t t = base + lane;
        int32_t b = 0, e = 0;
        if (t < cnt) {
            const int32_t j = C.cl_list[t];
            b = C.T.ptr[j];
            e = C.T.ptr[j + 1];
        }
        if (e - b <= 32)
            for (int32_t k = b; k < e; k++) C.rdnext[C.T.idx[k]] = 1;
        unsigned todo = __ballot_sync(0xffffffffu, e - b > 32);
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1u;
            const int32_t sb = __shfl_sync(0xffffffffu, b, src), se = __shfl_sync(0xffffffffu, e, src);
            for (int32_t k = sb + lane; k < se; k += 32) C.rdnext[C.T.idx[k]] = 1;
        }
    }
}

__global__ void __launch_bounds__(kBlock) k_mark_long(Ctx C, int64_t nnz) {
    const Chunk ch = C.T.chunks[blockIdx.x];
    if (!C.cchg[ch.seg] || 8 * (int64_t)*C.cl_nnz >= nnz) return;
    for (int32_t k = ch.begin + threadIdx.x; k < ch.end; k += kBlock) C.rdnext[C.T.idx[k]] = 1;
}

inline unsigned blocks_for(int64_t cnt, int threads) {
    return (unsigned)((cnt + threads - 1) / threads > 0 ? (cnt + threads - 1) / threads : 1);
}

}  // namespace

void launch_round_start(const Ctx &C, bool cols, cudaStream_t s) {
    const int64_t most = std::max<int64_t>({(int64_t)C.m / 16, (int64_t)C.n / 16, (int64_t)C.nlp, 64});
    (k_round_start<<<std::min<unsigned>(blocks_for(most, kBlock), 4u * 152u), kBlock, 0, s>>>(C, cols ? 1 : 0),
     note_launch());
}

void launch_s5_init(const Ctx &C, int32_t cap, int32_t *cnt, int32_t passes, cudaStream_t s) {
    (k_s5_init<<<std::min<unsigned>(blocks_for(std::max(cap / 2, passes), kBlock), 8u * 152u), kBlock, 0, s>>>(
         C.tkey, C.tlead, cap, cnt, passes),
     note_launch());
}

void launch_prop_short(const Ctx &C, cudaStream_t s) {
    const RowGrid R = prop_grid(C.A);
    if (R.g.blk_start[6] > 0) (k_prop_groups<<<R.g.blk_start[6], kBlock, 0, s>>>(C, R), note_launch());
}

bool prop_has_long(const Ctx &C) { return C.A.cls_start[7] > C.A.cls_start[6] && C.A.nchunks > 0; }

void launch_prop_long(const Ctx &C, cudaStream_t s) {
    const int32_t nlong = C.A.cls_start[7] - C.A.cls_start[6];
    if (nlong <= 0 || C.A.nchunks <= 0) return;
    (k_prop_long_partial<<<C.A.nchunks, kBlock, 0, s>>>(C), note_launch());
    (k_prop_long_combine<<<blocks_for((int64_t)nlong * 32, kBlock), kBlock, 0, s>>>(C), note_launch());
    (k_prop_long_tighten<<<C.A.nchunks, kBlock, 0, s>>>(C), note_launch());
}

void launch_bound_src(const Ctx &C, cudaStream_t s) {
    if (C.m <= 0 || C.n <= 0) return;
    const RowGrid R = class_grid(C.A);
    if (R.g.blk_start[6] > 0) (k_bsrc_groups<<<R.g.blk_start[6], kBlock, 0, s>>>(C, R), note_launch());
    if (C.A.cls_start[7] > C.A.cls_start[6] && C.A.nchunks > 0)
        (k_bsrc_chunks<<<C.A.nchunks, kBlock, 0, s>>>(C), note_launch());
}

void launch_mark_dependent(const Ctx &C, const int32_t *list, int32_t cnt, cudaStream_t s) {
    if (cnt > 0) (k_mark_dependent<<<blocks_for(cnt, kBlock), kBlock, 0, s>>>(C, list, cnt), note_launch());
}

void launch_colfin(const Ctx &C, bool full, cudaStream_t s) {
    if (C.n <= 0) return;
    if (full) (k_colfin<<<std::min<unsigned>(blocks_for(C.n, kBlock), 8u * 152u), kBlock, 0, s>>>(C), note_launch());
    else (k_colfin_list<<<std::min<unsigned>(blocks_for(C.n, kBlock), 8u * 152u), kBlock, 0, s>>>(C), note_launch());
}

void launch_mark_dirty(const Ctx &C, int64_t nnz, cudaStream_t s) {
    if (C.n <= 0) return;
    (k_mark_list<<<std::min<unsigned>(blocks_for(std::max(C.n, C.m), kBlock), 8u * 152u), kBlock, 0, s>>>(C, nnz),
     note_launch());
    if (C.T.cls_start[7] > C.T.cls_start[6] && C.T.nchunks > 0) (k_mark_long<<<C.T.nchunks, kBlock, 0, s>>>(C, nnz), note_launch());
}

void launch_s5_pass(const Ctx &C, cudaStream_t s) {
    if (C.m == 0) return;
    (k_s5_insert<<<std::min<unsigned>(blocks_for(C.m, kBlock), 8u * 152u), kBlock, 0, s>>>(C), note_launch());
    const RowGrid R = class_grid(C.A);
    if (R.g.blk_start[6] > 0) (k_s5_match_groups<<<R.g.blk_start[6], kBlock, 0, s>>>(C, R), note_launch());
    const int32_t nlong = C.A.cls_start[7] - C.A.cls_start[6];
    if (nlong > 0) (k_s5_match_long<<<nlong, kBlock, 0, s>>>(C), note_launch());
}

void launch_s5_tail(const Ctx &C, const int32_t *list, const int32_t *cnt, int32_t *out, int32_t *out_cnt,
                    int32_t max_rows, cudaStream_t s) {
    if (max_rows <= 0) return;
    (k_s5_tail_insert<<<blocks_for(max_rows, kBlock), kBlock, 0, s>>>(C, list, cnt), note_launch());
    (k_s5_tail_match<<<blocks_for(max_rows, kBlock), kBlock, 0, s>>>(C, list, cnt, out, out_cnt), note_launch());
    (k_s5_tail_clear<<<blocks_for(max_rows, kBlock), kBlock, 0, s>>>(C, list, cnt), note_launch());
}

void launch_s5_tail_block(const Ctx &C, int32_t *l0, int32_t *l1, int32_t *cnt, int32_t p0, int32_t max_iter,
                          cudaStream_t s) {
    (k_s5_tail_block<<<1, kTailBlock, 0, s>>>(C, l0, l1, cnt, p0, max_iter), note_launch());
}

// cooperative launch of k_s5_tail_grid, at most one block per SM and
// resident block slot, no more than the first list needs; false if the
// device cannot take a cooperative launch (the caller then launches passes)
bool launch_s5_tail_grid(const Ctx &C, int32_t *l0, int32_t *l1, int32_t *cnt, int32_t p0, int32_t max_iter,
                         int32_t rows, unsigned *bar, cudaStream_t s) {
    static CoopCache cache;
    const int most = coop_blocks((const void *)k_s5_tail_grid, cache);
    if (most <= 0) return false;
    const int64_t want = std::max<int64_t>(1, ((int64_t)rows + kBlock - 1) / kBlock);
    const unsigned grid = (unsigned)std::min<int64_t>(want, most);
    Ctx Cv = C;
    void *args[] = {&Cv, &l0, &l1, &cnt, &p0, &max_iter, &bar};
    if (cudaLaunchCooperativeKernel((const void *)k_s5_tail_grid, dim3(grid), dim3(kBlock), args, 0, s) != cudaSuccess)
        return false;
    note_launch();
    return true;
}

void launch_s5_leader(const Ctx &C, cudaStream_t s) {
    if (C.m > 0) (k_s5_leader<<<blocks_for(C.m, kBlock), kBlock, 0, s>>>(C), note_launch());
}

}  // namespace lpp
