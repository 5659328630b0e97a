// lpp_noalloc.cu -- row activities of a device-resident LP without any
// device allocation (lpp_row_activity_noalloc in lpp.h).
//
// Some callers cannot allocate device memory at the moment they need row
// activities: a GPU LP solver that reserved its whole memory budget up front
// and treats any further allocation as a failure, or a pipeline whose device
// memory is planned once and must not change while it runs.  For them this
// entry point computes the same quantities as the activity step of
// lpp_presolve using only the arrays the caller passes plus one fixed
// scratch array compiled into the library.
//
// A warp takes 32 consecutive rows, with as many lanes per row as its length
// asks for.  Rows of more than 32 entries belong to fixed 4096-entry windows of
// the entry array, a block each, so that the work is split by entries wherever
// such rows stand together: the block of the window in which a row starts takes
// it, and rows of more than 4096 are split by the windows.  A window meets at
// most two of those (one that started before it, one that starts inside it), so
// each window stores at most two partial results in the scratch array, and a last
// kernel adds a long row's partials in window order.  Every slot it reads is
// written earlier in the same call, so nothing in the scratch array has to start
// at zero.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "lpp_engine.h"

namespace {

constexpr int kNaWindow = 4096;           // entries per window
constexpr int kNaLong = 4096;             // longer rows use the windows
constexpr int kNaMaxWindows = 1 << 16;    // => at most 268,435,456 nonzeros
constexpr int kNaThreads = 256;
constexpr int kNaWarps = kNaThreads / 32;
// lanes per row by its length: one up to 4 entries, 4 up to 32, a warp up to
// 512, the block beyond (both in the window's block).  An FP64 warp instruction holds the pipe for 16
// clocks however many lanes are active, so a warp must not wait for one long
// row among short ones; lengths up to 4 are four fifths of a skewed LP's rows.
constexpr int kNaOne = 4, kNaShort = 32, kNaWarp = 512;

struct WindowPart {
    double2 act[2];   // (min, max) finite parts: [0] of the long row that started before the window,
    int2 ninf[2];     // [1] of the one that starts in it; infinite-term counts
    int32_t row[2];   // which row each slot belongs to (-1: unused)
    int32_t pad[2];
};
static_assert(sizeof(WindowPart) == 64, "4 MiB of scratch");

// The scratch of lpp_row_activity_noalloc: 4 MiB per device that loads the
// library, held until the process exits; shared by every call.
static __device__ __align__(256) WindowPart g_na_scratch[kNaMaxWindows];

struct NaArgs {
    int32_t m;
    int64_t nnz;
    const int32_t *rp, *ci;
    const double *val, *lb, *ub;
    long long huge_bits;  // |b| >= huge (or NaN) is infinite: one integer compare on the bits
    double *amin, *amax;
    int32_t *nmin, *nmax;
};

struct NaSum {
    double lo, hi;
    int nlo, nhi;
};

// entries b + 0, b + W, .. below e of a row, U loads and gathers in flight:
// the fused multiply-adds take them in order
template <int W, int U>
__device__ __forceinline__ void na_accumulate(const NaArgs &a, int32_t b, int32_t e, NaSum &s) {
    for (int32_t k0 = b; k0 < e; k0 += U * W) {
        int32_t j[U];
        double v[U], l[U], u[U];
#pragma unroll
        for (int q = 0; q < U; q++) {
            const bool in = k0 + q * W < e;
            j[q] = in ? a.ci[k0 + q * W] : -1;
            v[q] = in ? a.val[k0 + q * W] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < U; q++) {
            l[q] = j[q] >= 0 ? a.lb[j[q]] : 0.0;
            u[q] = j[q] >= 0 ? a.ub[j[q]] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < U; q++) {
            if (k0 + q * W >= e) break;
            const bool fl = (lpp::dbits(l[q]) & 0x7fffffffffffffffLL) < a.huge_bits;
            const bool fu = (lpp::dbits(u[q]) & 0x7fffffffffffffffLL) < a.huge_bits;
            const bool neg = lpp::is_neg(v[q]);
            const double bl = neg ? u[q] : l[q], bh = neg ? l[q] : u[q];
            if (neg ? fu : fl) s.lo = fma(v[q], bl, s.lo);
            else s.nlo++;
            if (neg ? fl : fu) s.hi = fma(v[q], bh, s.hi);
            else s.nhi++;
        }
    }
}

template <int W>
__device__ __forceinline__ void na_butterfly(NaSum &s) {
    const unsigned mask = lpp::group_mask<W>();
    s.lo = lpp::group_sum<W>(s.lo, mask);
    s.hi = lpp::group_sum<W>(s.hi, mask);
    s.nlo = lpp::group_sum<W>(s.nlo, mask);
    s.nhi = lpp::group_sum<W>(s.nhi, mask);
}

__device__ __forceinline__ void na_row(const NaArgs &a, int32_t r, const NaSum &s) {
    a.amin[r] = s.lo;
    a.amax[r] = s.hi;
    a.nmin[r] = s.nlo;
    a.nmax[r] = s.nhi;
}

// the block's sum of entries [b, e): warp butterflies, then the warps'
// (every thread must call it; thread 0 has the result)
__device__ __forceinline__ NaSum na_block(const NaArgs &a, int32_t b, int32_t e, NaSum *s_w) {
    NaSum s{0.0, 0.0, 0, 0};
    na_accumulate<kNaThreads, 4>(a, b + threadIdx.x, e, s);
    na_butterfly<32>(s);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = s;
    __syncthreads();
    NaSum w{0.0, 0.0, 0, 0};
    if (threadIdx.x < 32) {
        if (threadIdx.x < kNaWarps) w = s_w[threadIdx.x];
        na_butterfly<32>(w);
    }
    __syncthreads();
    return w;
}

// Row containing entry k, by a whole warp: the last row whose start is <= k
// (skips empty rows).  Each step probes 32 rows of the interval, so 2 M rows
// take five dependent loads instead of 21.
__device__ __forceinline__ int32_t na_row_of(const int32_t *rp, int32_t m, int64_t k) {
    const int lane = threadIdx.x & 31;
    int64_t lo = 0, hi = m;  // rp[lo] <= k < rp[hi]
    while (hi - lo > 1) {
        const int64_t p = lo + ((hi - lo) * (lane + 1)) / 33;
        const int c = __popc(__ballot_sync(0xffffffffu, rp[p] <= k));
        const int64_t l2 = c > 0 ? lo + ((hi - lo) * c) / 33 : lo;
        hi = c < 32 ? lo + ((hi - lo) * (c + 1)) / 33 : hi;
        lo = l2;
    }
    return (int32_t)lo;
}

// Rows of 33 to 4096 entries that start in the window [w0, w1), into own (at most
// kNaOwn of them); r0, r1: the rows of its first and last entry.  Few rows are
// looked at one by one; among many (most of them empty) a search finds those that
// hold a multiple of 32 entries, and the last row, which may hold none before w1.
constexpr int kNaOwn = (kNaWindow + kNaShort - 1) / kNaShort;
constexpr int32_t kNaScan = 8 * kNaThreads;
__device__ __forceinline__ void na_own_rows(const NaArgs &a, int64_t w0, int64_t w1, int32_t r0, int32_t r1,
                                            int32_t *own, int32_t *cnt) {
    const auto take = [&](int32_t r) {
        const int64_t b = a.rp[r], n = a.rp[r + 1] - b;
        if (b >= w0 && n > kNaShort && n <= kNaLong) own[atomicAdd(cnt, 1)] = r;
    };
    if (r1 - r0 < kNaScan) {
        for (int32_t r = r0 + (int32_t)threadIdx.x; r <= r1; r += kNaThreads) take(r);
        return;
    }
    const int64_t p = w0 + (int64_t)threadIdx.x * kNaShort;
    if (p < w1) {
        int32_t lo = r0, hi = r1;  // the last row that starts at or before p
        while (lo < hi) {
            const int32_t mid = lo + (hi - lo + 1) / 2;
            if (a.rp[mid] <= p) lo = mid;
            else hi = mid - 1;
        }
        if (a.rp[lo] > p - kNaShort) take(lo);  // p is its first multiple
    }
    if (threadIdx.x == kNaThreads - 1 && ((int64_t)a.rp[r1] + kNaShort - 1) / kNaShort * kNaShort >= w1) take(r1);
}

// window w of the entry array: the partials of the (at most two) long rows it
// meets, and the rows of 33 to 4096 entries that start in it
struct NaWindow {
    int32_t r[2], own[kNaOwn], cnt;
};
__device__ __forceinline__ void na_window(const NaArgs &a, WindowPart &p, int32_t w, NaSum *s_w, NaWindow &S) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t w0 = (int64_t)w * kNaWindow, w1 = min(a.nnz, w0 + kNaWindow);
    if (threadIdx.x == 0) S.cnt = 0;
    if (warp < 2) S.r[warp] = na_row_of(a.rp, a.m, warp == 0 ? w0 : w1 - 1);
    __syncthreads();
    na_own_rows(a, w0, w1, S.r[0], S.r[1], S.own, &S.cnt);
    for (int slot = 0; slot < 2; slot++) {
        const int32_t r = S.r[slot];
        const int64_t rb = a.rp[r], re = a.rp[r + 1];
        const bool use = re - rb > kNaLong && (slot == 0 ? rb < w0 : rb >= w0);
        if (threadIdx.x == 0) p.row[slot] = use ? r : -1;
        if (!use) continue;  // block-uniform
        const NaSum s = na_block(a, (int32_t)max(rb, w0), (int32_t)min(re, w1), s_w);
        if (threadIdx.x == 0) {
            p.act[slot] = make_double2(s.lo, s.hi);
            p.ninf[slot] = make_int2(s.nlo, s.nhi);
        }
    }
    __syncthreads();
    for (int i = warp; i < S.cnt; i += kNaWarps) {
        const int32_t r = S.own[i], b = a.rp[r], e = a.rp[r + 1];
        if (e - b > kNaWarp) continue;
        NaSum s{0.0, 0.0, 0, 0};
        na_accumulate<32, 4>(a, b + lane, e, s);
        na_butterfly<32>(s);
        if (lane == 0) na_row(a, r, s);
    }
    for (int i = 0; i < S.cnt; i++) {
        const int32_t r = S.own[i], b = a.rp[r], e = a.rp[r + 1];
        if (e - b <= kNaWarp) continue;  // block-uniform
        const NaSum s = na_block(a, b, e, s_w);
        if (threadIdx.x == 0) na_row(a, r, s);
    }
}

// Blocks [0, windows): the windows, first so that they run beside the rows; the
// other blocks: 256 rows each, those of at most 32 entries.
// Bound by the FP64 pipe (63% busy) and the latency of the two 8-byte bound
// gathers per entry: 20 M entries in 2 M skewed rows take 230 us, 2660 us
// with a warp per row (a median row of two entries used two of 32 lanes, and
// infinities were tested by FP64 compares).  No shared memory for the entries:
// a tile of them staged there, coalesced, took 510 us, because it leaves the
// L1 too few lines for the gathers in flight (4% hits instead of 23%).  With the
// rows of 33 to 4096 entries in the row blocks, 256 of them standing together ran
// on one SM: 3,000 rows of 4096 took 2460 us, now 128, a dense matrix of 1500 rows
// 1070, now 57.  The line at 32: with one at 64, 256 rows of 64 entries before
// 5,000 short ones took 67 us, not 45 (300 k rows of 33 entries 305, not 322).
__global__ void __launch_bounds__(kNaThreads, 5) k_na_rows(NaArgs a, WindowPart *scratch, int32_t windows) {
    __shared__ int2 s_mid[kNaWarps][32];  // a warp's rows of 5 to 32 entries: (lane of the row, first entry)
    __shared__ NaSum s_w[kNaWarps];
    __shared__ NaWindow s_win;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (blockIdx.x < (unsigned)windows) {
        na_window(a, scratch[blockIdx.x], (int32_t)blockIdx.x, s_w, s_win);
        return;
    }
    const int64_t rl = (int64_t)(blockIdx.x - windows) * kNaThreads + tid;
    const int32_t r = (int32_t)rl;
    int32_t b = 0, e = 0;
    if (rl < a.m) {
        b = a.rp[r];
        e = a.rp[r + 1];
    }
    const int32_t n = e - b;
    if (rl < a.m && n <= kNaOne) {
        NaSum s{0.0, 0.0, 0, 0};
        na_accumulate<1, 4>(a, b, e, s);
        na_row(a, r, s);
    }
    const unsigned mid = __ballot_sync(0xffffffffu, n > kNaOne && n <= kNaShort);
    if (n > kNaOne && n <= kNaShort) s_mid[warp][__popc(mid & ((1u << lane) - 1u))] = make_int2(lane, b);
    __syncwarp();
    const int nmid = __popc(mid);
    for (int i0 = 0; i0 < nmid; i0 += 8) {
        const int i = i0 + lane / 4;
        const int2 it = i < nmid ? s_mid[warp][i] : make_int2(0, 0);
        const int32_t eb = it.y, ee = eb + __shfl_sync(0xffffffffu, n, it.x);
        NaSum s{0.0, 0.0, 0, 0};
        if (i < nmid) na_accumulate<4, 4>(a, eb + (lane & 3), ee, s);
        na_butterfly<4>(s);
        if (i < nmid && (lane & 3) == 0) na_row(a, (int32_t)(rl - lane) + it.x, s);
    }
}

// one warp per window in which a long row starts: the row's partials, its
// windows lane-strided, then a butterfly
__global__ void __launch_bounds__(kNaThreads) k_na_long(NaArgs a, const WindowPart *scratch, int32_t windows) {
    const int32_t w = (int32_t)((blockIdx.x * (unsigned)kNaThreads + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (w >= windows) return;  // the same w in the whole warp
    const int32_t r = scratch[w].row[1];
    if (r < 0) return;
    const int32_t last = (a.rp[r + 1] - 1) / kNaWindow;
    NaSum s{0.0, 0.0, 0, 0};
    for (int32_t q = w + lane; q <= last; q += 32) {
        const int slot = q == w ? 1 : 0;
        const double2 d = scratch[q].act[slot];
        const int2 c = scratch[q].ninf[slot];
        s.lo += d.x;
        s.hi += d.y;
        s.nlo += c.x;
        s.nhi += c.y;
    }
    na_butterfly<32>(s);
    if (lane == 0) na_row(a, r, s);
}

// device address of g_na_scratch, looked up once per device
std::mutex g_na_mu;
void *g_na_ptr[256] = {};

}  // namespace

extern "C" lpp_status lpp_row_activity_noalloc(int32_t m, int32_t n, int64_t nnz, const int32_t *row_ptr,
                                               const int32_t *col_idx, const double *val, const double *lb,
                                               const double *ub, double huge, double *act_min, double *act_max,
                                               int32_t *ninf_min, int32_t *ninf_max, void *stream) {
    if (m < 0 || n < 0 || nnz < 0 || !(huge > 0))
        return lpp_noalloc_fail(LPP_ERR_INVALID, "lpp_row_activity_noalloc: negative size or huge <= 0");
    if (nnz > (int64_t)kNaMaxWindows * kNaWindow)
        return lpp_noalloc_fail(LPP_ERR_INVALID,
                                "lpp_row_activity_noalloc: nnz exceeds the fixed scratch (at most 268435456)");
    if (m == 0) return LPP_OK;
    if (!row_ptr || !act_min || !act_max || !ninf_min || !ninf_max || (nnz > 0 && (!col_idx || !val || !lb || !ub)))
        return lpp_noalloc_fail(LPP_ERR_INVALID, "lpp_row_activity_noalloc: NULL array");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return lpp_noalloc_fail(LPP_ERR_CUDA, cudaGetErrorString(e));
    if (dev < 0 || dev >= 256) return lpp_noalloc_fail(LPP_ERR_CUDA, "device ordinal out of range");
    void *scratch = nullptr;
    {
        std::lock_guard<std::mutex> g(g_na_mu);
        if (!g_na_ptr[dev]) {
            // set-up, once per device, with that device current: the array's
            // address, and both kernels loaded now (with lazy module
            // loading a kernel is otherwise loaded at its first launch, which
            // for the second is the first call with nnz > 4096)
            void *p = nullptr;
            e = cudaGetSymbolAddress(&p, g_na_scratch);
            cudaFuncAttributes fa;
            if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_na_rows);
            if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_na_long);
            if (e != cudaSuccess) return lpp_noalloc_fail(LPP_ERR_CUDA, cudaGetErrorString(e));
            g_na_ptr[dev] = p;
        }
        scratch = g_na_ptr[dev];
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    long long hb;
    std::memcpy(&hb, &huge, sizeof hb);
    NaArgs a{m, nnz, row_ptr, col_idx, val, lb, ub, hb, act_min, act_max, ninf_min, ninf_max};
    WindowPart *parts = static_cast<WindowPart *>(scratch);
    const int32_t windows = nnz > kNaShort ? (int32_t)((nnz + kNaWindow - 1) / kNaWindow) : 0;
    k_na_rows<<<(unsigned)(windows + (m + (int64_t)kNaThreads - 1) / kNaThreads), kNaThreads, 0, s>>>(a, parts,
                                                                                                  windows);
    if (nnz > kNaLong)
        k_na_long<<<(unsigned)((windows + kNaWarps - 1) / kNaWarps), kNaThreads, 0, s>>>(a, parts, windows);
    e = cudaGetLastError();
    if (e != cudaSuccess) return lpp_noalloc_fail(LPP_ERR_CUDA, cudaGetErrorString(e));
    return LPP_OK;
}
