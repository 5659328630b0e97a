// k_compact.cu -- S6 (empty columns) and S7 (compaction) of a round.
//
// After S5 every row is kept or removed and every column kept or fixed.  The
// compaction keeps the relative order of rows, columns and entries.  With the
// columns in place (Ctx::in_place, the default steps):
//   1. the columns of rows that left are noted (they may be empty now);
//   2. per kept row (CSR), one pass: entries left, the shift sum_j a_ij v_j over
//      its fixed columns, whether a bound in it changed, and which noted columns
//      it still holds; then S6: a column no row holds is fixed at the bound its
//      cost prefers (dual rule);
//   3. two exclusive scans: new row index, new row offset;
//   4. row vectors are gathered into the next buffers, the kept sides shifted
//      (L -= shift, U -= shift), and the entries scattered into the next CSR, column
//      indices as they are; columns and A^T are compacted once, after the rounds.
// With a step that reads columns' entries, A^T is compacted each round too:
// entries left per column (S6 from those, with locks for dual fixing), then rows
// by the columns' keep flags, four scans, column vectors, both scatters, renumbered.
// Long segments use the chunk lists of the schedule: a chunk counts its kept
// entries, the chunks of a segment are prefix-summed in order, and each chunk
// then writes its entries from its own offset.
#include <algorithm>

#include "lpp_launch.h"
#include "phase_dev.cuh"

namespace lpp {

namespace {

__global__ void k_lp_dead(Ctx C, CompactCtx K) {
    const int32_t lp = blockIdx.x * blockDim.x + threadIdx.x;
    if (lp >= C.nlp) return;
    bool d = K.lp_retired ? K.lp_retired[lp] != 0 : false;
    for (int v = 0; v < V_SLOTS; v++) d |= C.verdict[lp * V_SLOTS + v] != kNone;
    K.lp_dead[lp] = d;
}

// warp-group count of the entries of one segment that satisfy `keep`
template <int W, class Keep>
__device__ __forceinline__ int32_t group_count(const int32_t *idx, int32_t beg, int32_t end, Keep keep) {
    const int lane = threadIdx.x & (W - 1);
    int32_t c = 0;
    for (int32_t k = beg + lane; k < end; k += W) c += keep(idx[k]) ? 1 : 0;
    return group_sum<W>(c, group_mask<W>());
}

// ---------------------------------------------------------------- CSC count
template <int W>
__device__ __forceinline__ void csc_count_group(const Ctx &C, const CompactCtx &K, int32_t j, bool valid) {
    int32_t beg = 0, end = 0;
    if (valid) {
        beg = C.T.ptr[j];
        end = C.T.ptr[j + 1];
    }
    const uint8_t *rk = C.rkind;
    const int32_t cnt = group_count<W>(C.T.idx, beg, end, [rk](int32_t r) { return rk[r] == RK_KEPT; });
    if (valid && (threadIdx.x & (W - 1)) == 0) {
        K.c_len[j] = cnt;
        mark_tile(K.tile_t, beg, end, j);
    }
}

__global__ void __launch_bounds__(kBlock) k_csc_count_groups(Ctx C, CompactCtx K, GroupGrid g) {
    const int c = grid_class(g, blockIdx.x);
    const int W = 1 << c;
    const int32_t pos = C.T.cls_start[c] + (blockIdx.x - g.blk_start[c]) * (kBlock / W) + threadIdx.x / W;
    const bool valid = pos < C.T.cls_start[c + 1];
    const int32_t j = valid ? C.T.order[pos] : 0;
    switch (c) {
        case 0: csc_count_group<1>(C, K, j, valid); break;
        case 1: csc_count_group<2>(C, K, j, valid); break;
        case 2: csc_count_group<4>(C, K, j, valid); break;
        case 3: csc_count_group<8>(C, K, j, valid); break;
        case 4: csc_count_group<16>(C, K, j, valid); break;
        default: csc_count_group<32>(C, K, j, valid); break;
    }
}

__global__ void __launch_bounds__(kBlock) k_csc_count_long(Ctx C, CompactCtx K) {
    const Chunk ch = C.T.chunks[blockIdx.x];
    int32_t c = 0;
    for (int32_t k = ch.begin + threadIdx.x; k < ch.end; k += kBlock) c += C.rkind[C.T.idx[k]] == RK_KEPT;
    c = block_sum_int(c);
    if (threadIdx.x == 0) {
        K.cht_cnt[blockIdx.x] = c;
        mark_tile(K.tile_t, ch.begin, ch.end, ch.seg);
        if (ch.begin == C.T.ptr[ch.seg]) K.c_ch0[ch.seg] = blockIdx.x;
    }
}

__global__ void k_long_prefix(const SegMat M, const int32_t *ch_cnt, int32_t *ch_off, int32_t *len_out,
                              const double *ch_shift, double *shift_out) {
    long_prefix(M, (int32_t)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), ch_cnt, ch_off, len_out, ch_shift,
                shift_out);
}

template <int W>
__device__ __forceinline__ void lock_group(const Ctx &C, const CompactCtx &K, int32_t j, bool valid) {
    const unsigned mask = group_mask<W>();
    const int lane = threadIdx.x & (W - 1);
    int32_t beg = 0, end = 0, lk = 0;
    if (valid) {
        beg = C.T.ptr[j];
        end = C.T.ptr[j + 1];
    }
    for (int32_t k = beg + lane; k < end; k += W) lk |= entry_locks(C, C.T.idx[k], C.T.val[k]);
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) lk |= __shfl_xor_sync(mask, lk, o, W);
    if (valid && lane == 0) K.c_lock[j] = lk;
}

__global__ void __launch_bounds__(kBlock) k_locks_groups(Ctx C, CompactCtx K, RowGrid R) {
    int c;
    bool valid;
    const int32_t j = class_row(C.T, R, blockIdx.x, c, valid);
    if (c == 5) {  // columns of 65 to 4096 entries: the whole block (c_lock is zero before)
        for (int32_t q = 0; q < R.per5; q++) {
            const int32_t pos = C.T.cls_start[5] + (int32_t)(blockIdx.x - R.g.blk_start[0]) * R.per5 + q;
            if (pos >= C.T.cls_start[6]) break;
            const int32_t k = C.T.order[pos], e = C.T.ptr[k + 1];
            int32_t lk = 0;
#pragma unroll 4
            for (int32_t t = C.T.ptr[k] + (int32_t)threadIdx.x; t < e; t += kBlock) lk |= entry_locks(C, C.T.idx[t], C.T.val[t]);
            lk = __reduce_or_sync(0xffffffffu, (unsigned)lk);
            if ((threadIdx.x & 31) == 0 && lk) atomicOr(&K.c_lock[k], lk);
        }
        return;
    }
    switch (c) {
        case 0: lock_group<1>(C, K, j, valid); break;
        case 1: lock_group<2>(C, K, j, valid); break;
        case 2: lock_group<4>(C, K, j, valid); break;
        case 3: lock_group<8>(C, K, j, valid); break;
        default: lock_group<16>(C, K, j, valid); break;
    }
}

// long columns: one block per chunk, OR-ed into the column (zero before)
__global__ void __launch_bounds__(kBlock) k_locks_long(Ctx C, CompactCtx K) {
    const Chunk ch = C.T.chunks[blockIdx.x];
    int32_t lk = 0;
    for (int32_t k = ch.begin + threadIdx.x; k < ch.end; k += kBlock) lk |= entry_locks(C, C.T.idx[k], C.T.val[k]);
    lk = __reduce_or_sync(0xffffffffu, (unsigned)lk);
    if ((threadIdx.x & 31) == 0 && lk) atomicOr(&K.c_lock[ch.seg], lk);
}

// ------------------------------------------------------- S6 + column keep
// (grid-stride over a grid of at most 8 blocks per SM: one block sum per block)
__global__ void __launch_bounds__(kBlock) k_colkeep(Ctx C, CompactCtx K) {
    int32_t fixed = 0;
    for (int32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < C.n; j += gridDim.x * blockDim.x) {
        fixed += C.in_place ? colkeep_in_place(C, K, j) : colkeep_one(C, K, j);
    }
    block_add(fixed, &C.st->cols_fixed);
}

__global__ void __launch_bounds__(kBlock) k_suspect_rows(Ctx C, RowGrid R) { suspect_block(C, R, blockIdx.x); }
__global__ void __launch_bounds__(kBlock) k_suspect_long(Ctx C) { suspect_chunk(C, blockIdx.x); }

template <bool COUNT>
__global__ void __launch_bounds__(kBlock) k_inplace_rows(Ctx C, CompactCtx K, RowGrid R) {
    __shared__ InplaceShared S;
    inplace_block<COUNT>(C, K, R, blockIdx.x, S);
}
template <bool COUNT>
__global__ void __launch_bounds__(kBlock) k_inplace_long(Ctx C, CompactCtx K) {
    inplace_chunk<COUNT>(C, K, blockIdx.x);
}

// --------------------------------------------------------------- CSR count
template <int W>
__device__ __forceinline__ void csr_count_group(const Ctx &C, const CompactCtx &K, int32_t i, bool valid) {
    if (valid && (threadIdx.x & (W - 1)) == 0) mark_tile(K.tile_a, C.A.ptr[i], C.A.ptr[i + 1], i);
    csr_count_row<W>(C, K, i, valid, valid && C.rkind[i] == RK_KEPT && !K.lp_dead[lp_of_row(C, i)]);
}

__global__ void __launch_bounds__(kBlock) k_csr_count_groups(Ctx C, CompactCtx K, RowGrid R) {
    __shared__ double s_a[kMidStep], s_v[kMidStep];
    __shared__ int32_t s_mid[kBlock / 32], s_nmid, s_sum[1];
    int c;
    bool valid;
    const int32_t i = class_row(C.A, R, blockIdx.x, c, valid);
    switch (c) {
        case 0: csr_count_group<1>(C, K, i, valid); break;
        case 1: csr_count_group<2>(C, K, i, valid); break;
        case 2: csr_count_group<4>(C, K, i, valid); break;
        case 3: csr_count_group<8>(C, K, i, valid); break;
        case 4: csr_count_group<16>(C, K, i, valid); break;
        default: {
            if (threadIdx.x == 0) s_nmid = 0;
            __syncthreads();
            if (valid && C.A.ptr[i + 1] - C.A.ptr[i] >= kMidRow && C.rkind[i] == RK_KEPT && !K.lp_dead[lp_of_row(C, i)]) {
                if ((threadIdx.x & 31) == 0) s_mid[atomicAdd(&s_nmid, 1)] = i;
                valid = false;
            }
            csr_count_group<32>(C, K, i, valid);
            __syncthreads();
            const int32_t nmid = s_nmid;
            for (int32_t t = 0; t < nmid; t++) count_mid(C, K, s_mid[t], s_a, s_v, s_sum);
        }
    }
}

__global__ void __launch_bounds__(kBlock) k_csr_count_long(Ctx C, CompactCtx K) {
    const Chunk ch = C.A.chunks[blockIdx.x];
    const int32_t i = ch.seg;
    const bool keep = C.rkind[i] == RK_KEPT && !K.lp_dead[lp_of_row(C, i)];
    int32_t cnt = 0;
    double sh = 0.0;
    if (keep) {  // eight entries per thread and step in flight; the shift in entry order
        for (int32_t k0 = ch.begin + threadIdx.x; k0 < ch.end; k0 += 8 * kBlock) {
            int32_t jq[8], kq[8];
#pragma unroll
            for (int q = 0; q < 8; q++) jq[q] = k0 + q * kBlock < ch.end ? C.A.idx[k0 + q * kBlock] : 0;
#pragma unroll
            for (int q = 0; q < 8; q++) kq[q] = k0 + q * kBlock < ch.end ? K.c_keep[jq[q]] : 1;
#pragma unroll
            for (int q = 0; q < 8; q++) {
                if (k0 + q * kBlock >= ch.end) break;
                if (kq[q]) cnt++;
                else sh = fma(C.A.val[k0 + q * kBlock], C.fixv[jq[q]], sh);
            }
        }
    }
    cnt = block_sum_int(cnt);
    sh = block_sum_dbl(sh);
    if (threadIdx.x == 0) {
        K.chr_cnt[blockIdx.x] = cnt;
        K.chr_shift[blockIdx.x] = sh;
        mark_tile(K.tile_a, ch.begin, ch.end, i);
        if (ch.begin == C.A.ptr[i]) {  // the first chunk writes the flag
            K.r_keep[i] = keep;
            K.r_ch0[i] = blockIdx.x;
        }
    }
}

// ------------------------------------- the columns' one compaction (in place until then)
// keep flag of each column slot: still in the LP
__global__ void k_cols_alive(const int32_t *cinv, int32_t n, int32_t *keep) {
    const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < n) keep[j] = cinv[j] >= 0;
}
// the kept columns' vectors to their compacted positions; cinv then maps
// an input column to its final index
__global__ void k_cols_final(const Ctx C, const CompactCtx K, int32_t n, int32_t *cinv) {
    const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    if (!K.c_keep[j]) return;  // cinv already -1
    const int32_t p = K.c_pos[j];
    K.lu2[p] = C.lu[j];
    K.c2[p] = C.c[j];
    K.cmap2[p] = C.cmap[j];
    if (C.lp_col) K.lp_col2[p] = C.lp_col[j];
    cinv[C.cmap[j]] = p;
}
// the CSR's column indices renumbered in place
__global__ void k_idx_renumber(int32_t *idx, int64_t nnz, const int32_t *pos) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < nnz) idx[k] = pos[idx[k]];
}

// ---------------------------------------------------------- vector gathers
__device__ __forceinline__ void rowvec_at(const Ctx &C, const CompactCtx &K, int32_t i) {
    if (i >= C.m) return;
    if (i == C.m - 1) {
        K.rp2[K.r_pos[C.m]] = K.r_off[C.m];
        C.st->m_new = K.r_pos[C.m];
        C.st->nnz_new = K.r_off[C.m];
        if (C.in_place) {  // the column slots stay, no A^T is compacted
            C.st->n_new = C.n;
            C.st->nnz_new_t = K.r_off[C.m];
        }
    }
    const int32_t p = K.r_pos[i];
    if (!C.in_place) K.r_new[i] = K.r_keep[i] ? p : -1;
    if (K.r_keep[i]) rowvec_one(C, K, i, p, K.r_off[i], !C.in_place && K.c_pos[C.n] != C.n);
}

__device__ __forceinline__ void colvec_at(const Ctx &C, const CompactCtx &K, int32_t j) {
    if (j >= C.n) return;
    if (j == C.n - 1) {
        K.cp2[K.c_pos[C.n]] = K.c_off[C.n];
        C.st->n_new = K.c_pos[C.n];
        C.st->nnz_new_t = K.c_off[C.n];
    }
    const int32_t p = K.c_pos[j];
    K.c_new[j] = K.c_keep[j] ? p : -1;
    if (!K.c_keep[j]) return;
    K.lu2[p] = C.lu[j];
    K.c2[p] = C.c[j];
    K.cmap2[p] = C.cmap[j];
    if (C.lp_col) K.lp_col2[p] = C.lp_col[j];
    K.cp2[p] = K.c_off[j];
}

__global__ void __launch_bounds__(kBlock) k_rowvec(Ctx C, CompactCtx K) {
    rowvec_at(C, K, blockIdx.x * kBlock + threadIdx.x);
}
// rows, then columns from block rb on (the columns compacted each round)
__global__ void __launch_bounds__(kBlock) k_vecs(Ctx C, CompactCtx K, int32_t rb) {
    const int32_t b = blockIdx.x;
    if (b < rb) rowvec_at(C, K, b * kBlock + threadIdx.x);
    else colvec_at(C, K, (b - rb) * kBlock + threadIdx.x);
}

// without rows or columns: ptr[0] = 0 and the sizes
__global__ void k_empty(Ctx C, CompactCtx K) {
    if (C.m == 0) {
        K.rp2[0] = 0;
        C.st->m_new = 0;
        C.st->nnz_new = 0;
        if (C.in_place) {
            C.st->n_new = C.n;
            C.st->nnz_new_t = 0;
        }
    }
    if (C.n == 0 && !C.in_place) {
        K.cp2[0] = 0;
        C.st->n_new = 0;
        C.st->nnz_new_t = 0;
    }
}

__global__ void __launch_bounds__(kBlock) k_scatter_flat(FlatArgs F) {
    __shared__ FlatShared S;
    flat_tile(F, blockIdx.x, S);
}

__global__ void __launch_bounds__(kBlock) k_scatter_both(FlatArgs A, FlatArgs T) {
    __shared__ FlatShared S;
    const bool second = (int32_t)blockIdx.x >= A.ntiles;
    flat_tile(second ? T : A, blockIdx.x - (second ? A.ntiles : 0), S);
}

// ---------------------------------------------------------- objective constant
// one LP: tiles of kScanTile columns summed in a fixed order, then the tiles
__global__ void __launch_bounds__(kBlock) k_offset_tiles(double *contrib, int32_t n, double *part) {
    offset_tile(contrib, n, part, blockIdx.x);
}
__global__ void __launch_bounds__(kBlock) k_offset_final(const double *part, int32_t ntiles, double *offset) {
    offset_final(part, ntiles, offset);
}
// many LPs: column range of each LP, then one warp per LP
__global__ void k_lp_ranges(const int32_t *lp_col, int32_t n, int32_t *first, int32_t *last) {
    const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const int32_t lp = lp_col[j];
    if (j == 0 || lp_col[j - 1] != lp) first[lp] = j;
    if (j == n - 1 || lp_col[j + 1] != lp) last[lp] = j + 1;
}
__global__ void k_offset_lps(double *contrib, const int32_t *first, const int32_t *last, int32_t nlp,
                             double *offset) {
    const int32_t lp = (int32_t)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (lp >= nlp) return;
    double s = 0.0;
    for (int32_t j = first[lp] + lane; j < last[lp]; j += 32) {  // consumed as in k_offset_tiles
        const double v = contrib[j];
        s += v;
        if (v != 0.0) contrib[j] = 0.0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) offset[lp] += s;
}

inline unsigned blocks_for(int64_t cnt, int threads) {
    return (unsigned)std::max<int64_t>(1, (cnt + threads - 1) / threads);
}

}  // namespace

void launch_inplace_rows(const Ctx &C, const CompactCtx &K, bool count, cudaStream_t s, const SideStream *side) {
    const RowGrid R = class_grid(C.A);
    const int32_t acc = R.g.blk_start[6];
    // the long rows' chunks (and their prefix) on the side stream: disjoint
    // rows, each tile start lies in one row, a column's state byte gets the
    // same value from every writer
    const int32_t along = C.A.cls_start[7] - C.A.cls_start[6];
    const bool long_rows = along > 0 && C.A.nchunks > 0;
    const bool fork = long_rows && side && side->s;
    cudaStream_t sl = s;
    if (fork) {
        cudaEventRecord(side->fork, s);
        cudaStreamWaitEvent(side->s, side->fork, 0);
        sl = side->s;
    }
    if (long_rows) {
        if (count) {
            (k_inplace_long<true><<<C.A.nchunks, kBlock, 0, sl>>>(C, K), note_launch());
            (k_long_prefix<<<blocks_for((int64_t)along * 32, 128), 128, 0, sl>>>(C.A, K.chr_cnt, K.chr_off, K.r_len,
                                                                                  K.chr_shift, K.shift), note_launch());
        } else {
            (k_inplace_long<false><<<C.A.nchunks, kBlock, 0, sl>>>(C, K), note_launch());
        }
    }
    if (acc > 0) {
        if (count) (k_inplace_rows<true><<<acc, kBlock, 0, s>>>(C, K, R), note_launch());
        else (k_inplace_rows<false><<<acc, kBlock, 0, s>>>(C, K, R), note_launch());
    }
    if (fork) {
        cudaEventRecord(side->join, side->s);
        cudaStreamWaitEvent(s, side->join, 0);
    }
}

void launch_lp_dead(const Ctx &C, const CompactCtx &K, cudaStream_t s) {
    (k_lp_dead<<<blocks_for(C.nlp, 256), 256, 0, s>>>(C, K), note_launch());
}

static void launch_colkeep(const Ctx &C, const CompactCtx &K, cudaStream_t s) {
    if (C.n > 0) (k_colkeep<<<std::min<unsigned>(blocks_for(C.n, kBlock), 8u * 152u), kBlock, 0, s>>>(C, K), note_launch());
}

void launch_compact_counts(const Ctx &C, const CompactCtx &K, cudaStream_t s, const SideStream *side) {
    launch_lp_dead(C, K, s);
    if (C.in_place) {  // the rows' one pass marks the columns in use, then S6
        if (C.round > 1) {
            const RowGrid R = class_grid(C.A);
            if (R.g.blk_start[6] > 0) (k_suspect_rows<<<R.g.blk_start[6], kBlock, 0, s>>>(C, R), note_launch());
            if (C.A.cls_start[7] > C.A.cls_start[6] && C.A.nchunks > 0)
                (k_suspect_long<<<C.A.nchunks, kBlock, 0, s>>>(C), note_launch());
        }
        launch_inplace_rows(C, K, true, s, side);
        launch_colkeep(C, K, s);
        return;
    }
    // 1. column counts over kept rows, then S6 and the column keep flags
    const RowGrid ga = class_grid(C.A);
    const int32_t along = C.A.cls_start[7] - C.A.cls_start[6];
    const GroupGrid gt = group_grid(C.T);
    if (gt.blk_start[6] > 0) (k_csc_count_groups<<<gt.blk_start[6], kBlock, 0, s>>>(C, K, gt), note_launch());
    const int32_t tlong = C.T.cls_start[7] - C.T.cls_start[6];
    if (tlong > 0 && C.T.nchunks > 0) {
        (k_csc_count_long<<<C.T.nchunks, kBlock, 0, s>>>(C, K), note_launch());
        (k_long_prefix<<<blocks_for((int64_t)tlong * 32, 128), 128, 0, s>>>(C.T, K.cht_cnt, K.cht_off, K.c_len, nullptr,
                                                                             nullptr), note_launch());
    }
    if (C.dualfix && C.n > 0) {
        cudaMemsetAsync(K.c_lock, 0, sizeof(int32_t) * (size_t)C.n, s);
        const RowGrid rt = class_grid(C.T);
        if (rt.g.blk_start[6] > 0) (k_locks_groups<<<rt.g.blk_start[6], kBlock, 0, s>>>(C, K, rt), note_launch());
        if (tlong > 0 && C.T.nchunks > 0) (k_locks_long<<<C.T.nchunks, kBlock, 0, s>>>(C, K), note_launch());
    }
    launch_colkeep(C, K, s);
    // 2. row counts over kept columns and the side shifts; the long rows'
    // chunks (and their prefix) on the side stream when one is given: the
    // two touch disjoint rows, and each tile start lies in one row
    const bool long_rows = along > 0 && C.A.nchunks > 0;
    const bool fork = long_rows && side && side->s;
    cudaStream_t sl = s;
    if (fork) {
        cudaEventRecord(side->fork, s);
        cudaStreamWaitEvent(side->s, side->fork, 0);
        sl = side->s;
    }
    if (long_rows) {
        (k_csr_count_long<<<C.A.nchunks, kBlock, 0, sl>>>(C, K), note_launch());
        (k_long_prefix<<<blocks_for((int64_t)along * 32, 128), 128, 0, sl>>>(C.A, K.chr_cnt, K.chr_off, K.r_len,
                                                                              K.chr_shift, K.shift), note_launch());
    }
    if (ga.g.blk_start[6] > 0) (k_csr_count_groups<<<ga.g.blk_start[6], kBlock, 0, s>>>(C, K, ga), note_launch());
    if (fork) {
        cudaEventRecord(side->join, side->s);
        cudaStreamWaitEvent(s, side->join, 0);
    }
}

void launch_compact_scatter(const Ctx &C, const CompactCtx &K, int32_t nnz, cudaStream_t s) {
    // k_rowvec and k_colvec write the pointers (entry 0 with the first kept
    // segment or the total) and the new sizes; an empty dimension is left to k_empty
    if (C.m == 0 || C.n == 0) (k_empty<<<1, 1, 0, s>>>(C, K), note_launch());
    const int32_t rb = C.m > 0 ? (int32_t)blocks_for(C.m, kBlock) : 0;
    if (C.in_place) {
        if (rb > 0) (k_rowvec<<<rb, kBlock, 0, s>>>(C, K), note_launch());
    } else if (C.m > 0 || C.n > 0) {
        (k_vecs<<<rb + (C.n > 0 ? (int32_t)blocks_for(C.n, kBlock) : 0), kBlock, 0, s>>>(C, K, rb), note_launch());
    }
    const int32_t ntiles = (int32_t)(((int64_t)nnz + kFlatTile - 1) / kFlatTile);
    if (ntiles > 0) {
        FlatArgs fa{C.A.ptr, C.A.idx, C.A.val, nnz, C.m, ntiles, K.r_keep, K.r_off, K.r_len, K.r_ch0,
                    K.chr_off, K.chr_cnt, K.c_new, C.in_place ? C.cchg : nullptr, K.tile_a, K.ci2, K.rv2};
        if (C.in_place) {
            (k_scatter_flat<<<ntiles, kBlock, 0, s>>>(fa), note_launch());
        } else {
            FlatArgs ft{C.T.ptr, C.T.idx, C.T.val, nnz, C.n, ntiles, K.c_keep, K.c_off, K.c_len, K.c_ch0,
                        K.cht_off, K.cht_cnt, K.r_new, nullptr, K.tile_t, K.ri2, K.cv2};
            (k_scatter_both<<<2 * ntiles, kBlock, 0, s>>>(fa, ft), note_launch());
        }
    }
}

void launch_cols_alive(const int32_t *cinv, int32_t n, int32_t *keep, cudaStream_t s) {
    if (n > 0) (k_cols_alive<<<blocks_for(n, kBlock), kBlock, 0, s>>>(cinv, n, keep), note_launch());
}
void launch_cols_final(const Ctx &C, const CompactCtx &K, int32_t n, int32_t *cinv, int32_t *idx, int64_t nnz,
                       cudaStream_t s) {
    if (n > 0) (k_cols_final<<<blocks_for(n, kBlock), kBlock, 0, s>>>(C, K, n, cinv), note_launch());
    if (nnz > 0) (k_idx_renumber<<<blocks_for(nnz, kBlock), kBlock, 0, s>>>(idx, nnz, K.c_pos), note_launch());
}

void launch_offset(const Ctx &C, const CompactCtx &K, cudaStream_t s) {
    if (C.n == 0) return;
    if (C.nlp == 1) {
        const int32_t ntiles = (int32_t)((C.n + kScanTile - 1) / kScanTile);
        (k_offset_tiles<<<ntiles, kBlock, 0, s>>>(K.contrib, C.n, K.offset_part), note_launch());
        (k_offset_final<<<1, kBlock, 0, s>>>(K.offset_part, ntiles, K.offset), note_launch());
    } else {
        cudaMemsetAsync(K.lp_first, 0, sizeof(int32_t) * (size_t)C.nlp, s);
        cudaMemsetAsync(K.lp_last, 0, sizeof(int32_t) * (size_t)C.nlp, s);
        (k_lp_ranges<<<blocks_for(C.n, 256), 256, 0, s>>>(C.lp_col, C.n, K.lp_first, K.lp_last), note_launch());
        (k_offset_lps<<<blocks_for((int64_t)C.nlp * 32, 256), 256, 0, s>>>(K.contrib, K.lp_first, K.lp_last, C.nlp,
                                                                           K.offset), note_launch());
    }
}

}  // namespace lpp
