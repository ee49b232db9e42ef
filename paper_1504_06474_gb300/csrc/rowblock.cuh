// rowblock.cuh -- y = A x by blocks of rows, the library's automatic choice
// when the caller asks for no tile shape and no variant of the segmented sum.
//
//   (r1) rowblock_kernel  a warp takes a group of rows: 32 rows, one per lane,
//                         or 32/G rows with G lanes each when rows are long.
//                         The values and columns of a group (of several short
//                         ones) are one contiguous range of the arrays, copied
//                         to shared memory by two bulk copies.
//   (r2) rowtail_kernel   groups of more entries than two stages hold (rows of
//                         thousands of entries and their neighbours; in FP64
//                         also smaller ones that one row fills), listed by
//                         (r1): a warp per row, or per piece of a very long
//                         row, straight from global memory.
//
// Why rows and not tiles of equal length: on this GPU one warp-wide FP64
// instruction occupies the FP64 pipe of an SM quarter for 76 cycles, however
// few lanes take part (measured), so 32 multiply-adds cost as much as
// streaming their 384 bytes and every extra FP64 addition of a cross-lane sum
// costs the same again.  A lane that owns a row needs no such additions, no
// descriptor, no partition, no repair of empty rows and no second pass over
// row_ptr; and lanes on neighbouring rows gather neighbouring x.  Groups whose
// row lengths are too uneven for that split their entries evenly over the
// lanes instead (a segmented sum inside the group).
//
// Measured (us a call among others; before: the three kernels of segsum.cuh).
// FP64: 27-point stencil 160^3 272 -> 239 (the FP64 pipe alone needs 207), R-MAT
// scale 22 with a 10^6-entry row 402 -> 327, banded half-width 31 (300,001 rows,
// plan) 64 -> 51, uniform rows of 0..40 entries (120,007 rows, axpby) 46 -> 22,
// rows of 1..8 entries and three of 500,000 92 -> 62, uniform 4096 rows 15 -> 7.
// FP32: stencil 101x97x103 62 -> 46, R-MAT scale 20 107 -> 89, 96 mixed matrices
// 516 -> 344; BF16 values: stencil 120x125x131 110 -> 72.
#pragma once
#include <cstdint>

#include "launch.cuh"
#include "rowshape.h"
#include "segsum.cuh"

namespace ssspmv {

// one matrix of a batch (filled on the device from the caller's descriptors by
// the batch set-up kernel)
struct RowMat {
    const void *val;
    const int32_t *col;
    const int32_t *row_ptr;
    const void *x;
    void *y;
    int32_t m, nnz;
    int32_t unit_base;  // the batch's number of its first unit
    int32_t nbig;       // see RowArgs
    int32_t cap;        // its shape: cap, and gs | us << 8 | piece << 16
    int32_t packed;
};
static_assert(sizeof(RowMat) == kRowMatBytes, "RowMat is one 64-byte record");

struct RowArgs {
    const int32_t *row_ptr;
    const int32_t *col;
    const void *val;
    const void *x;
    void *y;
    uint32_t *head;      // the workspace's header words
    int2 *ranges;        // {first row, rows}
    int2 *pieces;        // {row, piece}
    double *parts;       // sums of pieces
    uint32_t *arrived;   // per first piece of a row: its pieces summed so far
    int32_t max_ranges, max_pieces;
    int32_t m, nnz;
    int32_t nunits, nbig;  // units of rows, and how many of them of several groups
    RowShape shape;
    double alpha, beta;
    int32_t axpby;
    // batches: the matrices, the batch's units, and the matrix of each list entry
    const RowMat *mats = nullptr;
    int32_t count = 0;
    const int32_t *total_units = nullptr;
    int32_t *range_mat = nullptr, *piece_mat = nullptr;
};

// ---------------------------------------------------------------------------

// entry loop of one lane: n entries, the i-th at shared index i * G (G == 0:
// i * stride), added to acc; every lane has nmin or more, none more than nmax.
// ROT: the lane starts at its rot-th entry and wraps around (rot <= n).  A multiply-add that
// no lane needs is branched over: with every lane predicated off it
// would still hold the FP64 pipe for its 76 cycles (measured).
template <class P, int UN, int G, bool ROT>
__device__ __forceinline__ typename P::acc_t lane_dot(const typename P::val_t *vs,
                                                      const int32_t *cs,
                                                      const typename P::x_t *x, int n, int nmin,
                                                      int nmax, int stride, int rot, uint64_t pol,
                                                      typename P::acc_t acc)
{
    using X = typename P::x_t;
    const int st = G > 0 ? G : stride;
    // shared index of the lane's i-th entry
    auto at = [&](int i) { return ROT ? (i + rot < n ? i + rot : i + rot - n) * st : i * st; };
    int i = 0;
    for (; i + UN <= nmin; i += UN) {
        X xv[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) xv[u] = P::gather(x, cs[at(i + u)], pol);
#pragma unroll
        for (int u = 0; u < UN; ++u) acc = P::fma(vs[at(i + u)], xv[u], acc);
    }
    for (; i < nmax; i += UN) {
        X xv[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u)
            if (i + u < n) xv[u] = P::gather(x, cs[at(i + u)], pol);
#pragma unroll
        for (int u = 0; u < UN; ++u) {
            if (i + u >= nmax) break;
            if (i + u < n) acc = P::fma(vs[at(i + u)], xv[u], acc);
        }
    }
    return acc;
}

constexpr int kTurnUnits = 8192;  // fewer units are all taken by turns
constexpr int kUnitRowsMax = 128;
constexpr int kBatchRowWarps = 20;  // a batch's kernel needs 96 registers
// A kernel of its own for large matrices of very short rows: a stage of up to four
// groups whose rows have no more than kShortRow entries is worked off at once,
// where the general loop gathers for one group after the other, each a round trip
// of some 0.8 us for 32 rows.  20 million rows, FP64: of one entry 277 us and 181
// (the tiles 213), of 0 or 1 260 and 178 (209), of two 299 and 210 (285), of 1 to 3
// 314 and 228 (287); FP32 223 and 148 (197), 198 and 147 (200), 237 and 168 (241),
// 250 and 188 (245); 2 million of one entry 27.1 and 23.3; random columns from two
// entries on and R-MATs from 2 million rows on the same within 2%.  (Below: R-MATs
// of 0.5 and 1 million rows 2 to 5% slower, rows of one entry 7% faster.  In the
// general kernel the loop costs longer rows more than it gives these.)
constexpr int kShortRow = 4;
constexpr int32_t kShortRows = 1500000;  // rows from which on it is taken

struct alignas(16) RowScratch {
    uint64_t bar;
    uint64_t pad;
    uint32_t heads[32];
    uint8_t seg_row[kUnitRowsMax + 16];
    int32_t rp[kUnitRowsMax + 4];  // the unit's row pointers
};

// entries staged at [0, T): lane l sums [l*C, (l+1)*C), C odd (shared reads
// free of bank conflicts); sc->heads has a bit at each row start and at 0, in
// the order of sc->seg_row, and the rows cut between lanes are joined across
// them.  carry is the first row's sum so far; if the last row goes on past the
// stage (cont) its sum is returned instead of stored.  emit(row, sum) stores.
template <class P, class Emit>
__device__ __forceinline__ typename P::acc_t even_split(
    const typename P::val_t *vs, const int32_t *cs, const typename P::x_t *x, const RowScratch *sc,
    int32_t T, int32_t C, typename P::acc_t carry, bool cont, uint64_t pol, Emit &&emit)
{
    using X = typename P::x_t;
    using A = typename P::acc_t;
    constexpr int UN = P::kSplitBatch;
    const int lane = threadIdx.x & 31;
    const uint32_t hb = sc->heads[lane];
    const int c = __popc(hb);
    const int incl = warp_inclusive_scan(c, lane);
    const int idx0 = incl - c;
    const int nseg = __shfl_sync(FULL, incl, 31);
    auto row_of = [&](int seg) { return (int)sc->seg_row[seg & (kUnitRowsMax - 1)]; };
    int32_t n = T - lane * C;
    n = n < 0 ? 0 : (n > C ? C : n);
    vs += lane * C;
    cs += lane * C;
    A sum = P::zero(), pre = P::zero();
    int seg = idx0 - 1;
    X xa[UN];
    auto gather = [&](X (&xv)[UN], int i) {
#pragma unroll
        for (int k = 0; k < UN; ++k)
            if (i + k < n) xv[k] = P::gather(x, cs[i + k], pol);
    };
    auto fmas = [&](const X (&xv)[UN], int i) {
#pragma unroll
        for (int k = 0; k < UN; ++k) {
            if (i + k >= C) break;
            if ((hb >> (i + k)) & 1u) {  // closes the open segment
                if (seg >= idx0) emit(row_of(seg), sum);
                else pre = sum;
                ++seg;
                sum = (i + k == 0 && lane == 0) ? carry : P::zero();
            }
            if (i + k < n) sum = P::fma(vs[i + k], xv[k], sum);
        }
    };
#pragma unroll 1
    for (int i = 0; i < C; i += UN) {
        gather(xa, i);
        fmas(xa, i);
    }
    if (c == 0) pre = sum;  // no head: part of an earlier lane's segment
    const bool has = c > 0;
    const unsigned hm = __ballot_sync(FULL, has);
    const unsigned le = hm & ((lane == 31) ? FULL : ((2u << lane) - 1u));
    const int first = 31 - __clz(le);
    const int span = (int)__reduce_max_sync(FULL, (unsigned)(lane - first));
    A Cs = sum;
    if (span <= 4) {
        for (int d = 1; d <= span; ++d) {
            const A o = P::shfl_up(sum, d);
            if (lane - d >= first) Cs = P::add(Cs, o);
        }
    } else {
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const A o = P::shfl_up(Cs, d);
            if (lane - d >= first) Cs = P::add(Cs, o);
        }
    }
    const A Cprev = P::shfl_up(Cs, 1);
    if (has && lane > 0) emit(row_of(idx0 - 1), P::add(Cprev, pre));
    if (lane == 31 && !cont) emit(row_of(nseg - 1), Cs);
    return P::shfl(Cs, 31);
}

// a group that is not staged: its rows go to the lists (r2) works on.  Lane l
// holds row row0 + l of the group, len entries (0 past the group's rows).
static __device__ __noinline__ void list_group(const RowArgs &a, int32_t mat, int32_t pl,
                                               int32_t row0, int32_t rows, int32_t len)
{
    const int lane = threadIdx.x & 31;
    const bool valid = lane < rows;
    const bool isl = valid && len > (1 << pl);
    const int32_t plain = (valid && !isl) ? len : 0;
    const int32_t bucket = (warp_inclusive_scan(plain, lane) - plain) >> pl;
    const int32_t prev = __shfl_up_sync(FULL, bucket, 1);
    const bool lead = valid && (lane == 0 || bucket != prev);
    const unsigned leads = __ballot_sync(FULL, lead);
    const int32_t np = isl ? row_pieces(len, pl) : 0;
    const int32_t pincl = warp_inclusive_scan(np, lane);
    const int32_t total = __shfl_sync(FULL, pincl, 31);
    unsigned long long got = 0;
    if (lane == 0)
        got = atomicAdd(reinterpret_cast<unsigned long long *>(a.head + kWordLists),
                        ((unsigned long long)total << 32) | (unsigned)__popc(leads));
    got = __shfl_sync(FULL, got, 0);
    const uint32_t rbase = (uint32_t)got, pbase = (uint32_t)(got >> 32);
    if ((uint64_t)rbase + __popc(leads) > (uint32_t)a.max_ranges ||
        (uint64_t)pbase + (uint32_t)total > (uint32_t)a.max_pieces) {
        // more than any valid row_ptr can list
        if (lane == 0) atomicOr(a.head + kWordRowErr, SSSPMV_DEV_RANGE);
        return;
    }
    if (lead) {
        const unsigned above = lane == 31 ? 0u : leads & ~((2u << lane) - 1u);
        const int next = above ? __ffs(above) - 1 : rows;
        const uint32_t at = rbase + __popc(leads & ((1u << lane) - 1u));
        a.ranges[at] = make_int2(row0 + lane, next - lane);
        if (a.range_mat) a.range_mat[at] = mat;
    }
    unsigned todo = __ballot_sync(FULL, isl);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const int32_t n = __shfl_sync(FULL, np, src);
        const uint32_t at = pbase + __shfl_sync(FULL, pincl, src) - n;
        if (lane == 0) a.arrived[at] = 0u;
        for (int32_t p = lane; p < n; p += 32) {
            a.pieces[at + p] = make_int2(row0 + src, p);
            if (a.piece_mat) a.piece_mat[at + p] = mat;
        }
    }
}

// ---------------------------------------------------------------------------
// (r1)

// what is stored in y[row] for a row's sum v (alpha and beta: FP64 only)
template <class Y>
__device__ __forceinline__ Y row_value(const RowArgs &a, const Y *y, int32_t row, Y v)
{
    if constexpr (sizeof(Y) == sizeof(double))
        return scaled_store_value(y, row, v, a.alpha, a.beta, a.axpby);
    else return v;
}

// copies of the entries [b, e) into a warp's stage (all lanes call it); entry
// k lands at index k - (b & ~7)
template <class V>
__device__ __forceinline__ void stage_copy(unsigned char *st, int32_t col_off, uint64_t *bar,
                                           const V *val, const int32_t *col, int32_t nnz, int32_t b,
                                           int32_t e, uint64_t pol)
{
    const int lane = threadIdx.x & 31;
    const int32_t b8 = b & ~7;
    int32_t e8 = (e + 7) & ~7;
    if (e8 > nnz) e8 = nnz & ~7;  // the last entries of the arrays: below
    const int32_t n = e8 > b8 && e > b ? e8 - b8 : 0;
    if (lane == 0) {
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(bar, (uint32_t)n * (uint32_t)(sizeof(V) + 4));
        if (n > 0) {
            bulk_g2s(st, val + b8, (uint32_t)n * (uint32_t)sizeof(V), bar, pol);
            bulk_g2s(st + col_off, col + b8, (uint32_t)n * 4u, bar, pol);
        }
    }
    if (e > e8 && e > b) {
        const int32_t k = (e8 > b8 ? e8 : b8) + lane;
        if (k < e) {
            reinterpret_cast<V *>(st)[k - b8] = val[k];
            reinterpret_cast<int32_t *>(st + col_off)[k - b8] = col[k];
        }
    }
}

// Whether a stage of T entries in `groups` groups, whose longest lanes take n
// steps in all, keeps a lane per row (or G lanes), or splits its entries evenly
// (T / 32 steps and the joining of the cut rows).  Each group adds a step for the
// reductions that both ways make per group.  Against a longer lane of up to 2.5
// times the mean and 15 for FP32: rows of 0..40, 0..80 and 0..160 entries, 30
// million in all, FP32 139, 137 and 125 us and 123, 120 and 119 so, BF16 values
// 130, 127, 118 and 118, 114, 114; that rule for FP64: 136, 131, 128 and 156, 152,
// 137.  Without the step per group FP64 rows of 0..8 entries take 67 us instead of
// 64 (10 million); with two or more, of 0..20 143 instead of 137 (30 million).
__device__ __forceinline__ bool rows_even(int n, int T, int groups)
{
    return n <= (T >> 5) + (T >> 6) + 7 + groups;
}

// row pointer p as an index into [b, e], whatever row_ptr holds
__device__ __forceinline__ int32_t inside(int32_t p, int32_t b, int32_t e)
{
    return p < b ? b : (p > e ? e : p);
}

// the matrix that unit u of a batch belongs to: the last one of `count` that
// starts at or before it, `from` or a later one (all lanes call it).  The next
// 32 at once, then a search by 33 ways: a walk from one record to the next, which
// every warp makes past every matrix, took 2,198 us of 10,000 matrices of 1,000
// entries and 225 of 1,000 of 10,000; so 195 and 76 (the tiles: 188 and 66; 96
// mixed matrices: 336 us either way).
__device__ __forceinline__ int32_t find_matrix(const RowMat *mats, int32_t count, int32_t from,
                                               int32_t u)
{
    const int lane = threadIdx.x & 31;
    int32_t lo = from, hi = count, step = 1;
    while (hi - lo > 1) {
        const int32_t i = lo + (lane + 1) * step;
        const int n = __popc(__ballot_sync(FULL, i < hi && __ldg(&mats[i].unit_base) <= u));
        lo += n * step;
        if (n < 32 && lo + step < hi) hi = lo + step;
        step = (hi - lo + 31) >> 5;
    }
    return lo;
}

template <class P, bool MULTI, bool BATCHED = false, bool SHORT = false>
__global__ void __launch_bounds__((BATCHED ? kBatchRowWarps : P::kRowWarps) * 32, 1)
    rowblock_kernel(const RowArgs a, int32_t stage_bytes, int32_t col_off)
{
    using V = typename P::val_t;
    using X = typename P::x_t;
    using Y = typename P::y_t;
    using A = typename P::acc_t;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int32_t s_ticket;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char *const st = smem + warp * ((size_t)stage_bytes + sizeof(RowScratch));
    RowScratch *const sc = reinterpret_cast<RowScratch *>(st + stage_bytes);
    const V *const sv = reinterpret_cast<const V *>(st);
    const int32_t *const scol = reinterpret_cast<const int32_t *>(st + col_off);
    if (threadIdx.x == 0) s_ticket = 0;
    if (lane == 0) {
        mbar_init(&sc->bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    grid_dep_wait();  // everything read below may come from the kernel before
    grid_dep_trigger();

    // the current unit's matrix (in a batch: loaded again when it changes)
    const X *__restrict__ x = static_cast<const X *>(a.x);
    const V *__restrict__ val = static_cast<const V *>(a.val);
    const int32_t *__restrict__ col = a.col;
    Y *__restrict__ y = static_cast<Y *>(a.y);
    int32_t m = a.m, nnz = a.nnz, cap = a.shape.cap, piece = a.shape.piece;
    int gs = MULTI ? a.shape.gs : 0;
    auto load_matrix = [&](int32_t mi) {
        const RowMat *mm = a.mats + mi;
        val = static_cast<const V *>(ldg_ptr(&mm->val));
        x = static_cast<const X *>(ldg_ptr(&mm->x));
        y = static_cast<Y *>(ldg_ptr(const_cast<void *const *>(&mm->y)));
        col = ldg_ptr(&mm->col);
        m = __ldg(&mm->m);
        nnz = __ldg(&mm->nnz);
        cap = __ldg(&mm->cap);
        const int32_t p = __ldg(&mm->packed);
        gs = p & 255;
        piece = p >> 16;
    };
    const int32_t nunits = BATCHED ? __ldg(a.total_units) : a.nunits;
    // The first quarter of the units by turns (block b takes every gridDim.x-th
    // from the b-th on, its warps by a ticket in shared memory), the others by
    // a ticket of the whole grid: the blocks' shares of a power-law matrix
    // differ by a quarter of their time.  All of them by turns: R-MAT scale 22
    // 145 us, scale 20 FP32 53; half 123 and 51; a quarter 118 and 47; none
    // 118 and 49.  Small matrices would only wait for the ticket (120,007 rows
    // of 0..40 entries: 23 us, 24 with it), and a batch's even each other out
    // (342 us, 355 with half of them).
    const bool turns = BATCHED || nunits < kTurnUnits;
    const int64_t nstatic = turns ? INT64_MAX : nunits >> 2;
    const uint64_t pol_keep = policy_evict_last(), pol_stream = policy_evict_first();

    // the next unit of rows [r0, r0 + nr): several groups at a time first,
    // single ones towards the end; its row pointers are loaded into
    // registers, the lane's i-th being row_ptr[r0 + 32 i + lane]
    constexpr int NP = kUnitRowsMax / 32 + 1;
    struct Unit {
        int32_t r0, nr;
        int32_t mat;
        int32_t rp[NP];
    };
    int32_t at_mat = 0;  // a warp's tickets only grow, and with them the matrix
    auto next_unit = [&]() -> Unit {
        uint32_t t = 0;
        if (lane == 0) {
            const int64_t turn = (int64_t)atomicAdd(&s_ticket, 1) * gridDim.x + blockIdx.x;
            t = (uint32_t)(turn < nunits ? turn : nunits);
            if (!BATCHED && turn >= nstatic)
                t = (uint32_t)nstatic + atomicAdd(a.head + kWordUnitTicket, 1u);
        }
        t = __shfl_sync(FULL, t, 0);
        Unit q;
        q.r0 = -1;
        q.nr = 0;
        q.mat = 0;
        if (t >= (uint32_t)nunits) return q;
        int32_t u = (int32_t)t, um = m, ugs = gs, us = a.shape.us, nbig = a.nbig;
        const int32_t *row_ptr = a.row_ptr;
        if constexpr (BATCHED) {
            at_mat = find_matrix(a.mats, a.count, at_mat, u);
            const RowMat *mm = a.mats + at_mat;
            row_ptr = ldg_ptr(&mm->row_ptr);
            um = __ldg(&mm->m);
            u -= __ldg(&mm->unit_base);
            nbig = __ldg(&mm->nbig);
            const int32_t p = __ldg(&mm->packed);
            ugs = p & 255;
            us = (p >> 8) & 255;
            q.mat = at_mat;
        }
        const int32_t rows = 32 >> ugs, big = rows << us;
        if (u < nbig) {
            q.r0 = u * big;
            q.nr = big;
        } else {
            q.r0 = nbig * big + (u - nbig) * rows;
            q.nr = rows;
        }
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const int32_t r = q.r0 + 32 * i + lane;
            if (32 * i <= q.nr) q.rp[i] = __ldg(row_ptr + (r < um ? r : um));
        }
        return q;
    };
    auto store = [&](int32_t row, A v) {
        y[row] = row_value(a, y, row, P::out(v));
    };

    // One stage per warp, and as many warps as shared memory holds: a warp
    // waits for its copy while the others compute.  The row pointers of the
    // next unit are loaded a unit ahead.
    uint32_t phase = 0;  // parity of the stage's next completion
    Unit cur = next_unit();
    const int32_t *const rp = sc->rp;
    int32_t mat = -1;
    while (cur.nr > 0) {
        if (BATCHED && cur.mat != mat) load_matrix(mat = cur.mat);
        const int32_t rows = 32 >> gs;  // per group
#pragma unroll
        for (int i = 0; i < NP; ++i)
            if (32 * i + lane <= cur.nr) sc->rp[32 * i + lane] = cur.rp[i];
        __syncwarp();
        Unit nxt;
        nxt.nr = -1;  // not asked for yet
        const int32_t b = inside(rp[0], 0, nnz), e = inside(rp[cur.nr], b, nnz);
        int32_t j = 0;      // the next group's first row in the unit
        int32_t at = -1;    // (a group larger than the stage) its next entry
        A carry = P::zero();
#pragma unroll 1
        while (j < cur.nr) {
            // log2 of the lanes per row in this pass, and its rows: a group's, or
            // half of one's
            const bool second = MULTI && (j & (rows - 1)) != 0;
            int gl = gs + second;
            int32_t rl = 32 >> gl;
            const int32_t g0 = inside(rp[j], b, e);
            int32_t ge = inside(rp[j + rl], g0, e), T = ge - g0;
            // Listed: a group of too many entries, or (FP64) one that does not fit the
            // stage and whose longest row has half of its entries: the two stages of
            // such a group hold up its unit, and at the end of the launch all.  1,000
            // rows of 1,000 entries in 166,666 of 4.5 on average 31 us, and listed 22,
            // in 1.7 million 72 and 61; the row lengths of a Pareto law over 2,000 to
            // 16,000 rows 18 to 23 us and 15 to 19.  (100 such rows in 5 million: 136
            // and 144.  In FP32, where single and batched products have to agree, the
            // test alone made 27-point stencils 3% slower.)
            if (T > cap && !second) {
                bool list = T > 2 * cap && (!MULTI || T > row_most(nnz, gs, cap));
                if (!list && (sizeof(V) == 8 || MULTI) && gs < 5) {
                    const int32_t rs = rp[j + (lane >> gs)], re = rp[j + (lane >> gs) + 1];
                    const int32_t longest = (int32_t)__reduce_max_sync(FULL, (unsigned)(re - rs));
                    list = sizeof(V) == 8 && longest >= T - longest;
                    // a group of rows of about the same length that does not fit the
                    // stage goes by halves of its rows with twice the lanes for each,
                    // not by even parts of its entries (diagonal blocks of 32 to 64
                    // rows, 28 million entries: FP64 94 us -> 75, FP32 80 -> 54, BF16
                    // values 80 -> 54; of 32 to 230: 88 -> 78, 71 -> 58, 71 -> 57.
                    // Uneven groups by halves too: R-MAT of edge factor 32 in FP32 15%
                    // slower; more lanes per row from the mean: bands up to 30% slower)
                    if (MULTI && !list && gs > 0 &&
                        rows_even((longest + (1 << gs) - 1) >> gs, T, 1)) {
                        ++gl;
                        rl >>= 1;
                        ge = inside(rp[j + rl], g0, e);
                        T = ge - g0;
                    }
                }
                if (list) {
                    const int32_t l = lane < rows ? lane : 0;
                    const int32_t rs = inside(rp[j + l], g0, ge);
                    const int32_t re = inside(rp[j + l + 1], rs, ge);
                    const int32_t left = m - (cur.r0 + j);
                    list_group(a, cur.mat, piece, cur.r0 + j, left < rows ? left : rows,
                               lane < rows ? re - rs : 0);
                    j += rows;
                    continue;
                }
            }
            const int sub = lane & ((1 << gl) - 1);
            const int lrow = lane >> gl;  // the lane's row
            // the entries [ts, te) of the rows [j, jn): this group and those
            // after it that fit with it; or an even part of a group (of a row)
            // that does not fit by itself
            int32_t ts = g0, te = ge, jn = j + rl;
            if (T > cap) {
                const int32_t parts = (T + cap - 1) / cap;
                const int32_t len = ((T + parts - 1) / parts + 7) & ~7;
                ts = at < 0 ? g0 : at;
                te = ts + len < ge ? ts + len : ge;
            } else if (rl == rows) {
                while (jn < cur.nr) {
                    const int32_t t = inside(rp[jn + rows], te, e);
                    if (t - g0 > cap) break;
                    te = t;
                    jn += rows;
                }
            }
            if (!BATCHED && te == ts) {  // rows without entries: nothing to copy
                for (int32_t k = j + lane; k < jn; k += 32)
                    if (cur.r0 + k < m) store(cur.r0 + k, P::zero());
                j = jn;
                continue;
            }
            __syncwarp();  // every lane is done with the copy before
            stage_copy(st, col_off, &sc->bar, val, col, nnz, ts, te, pol_stream);
            if (nxt.nr < 0) nxt = next_unit();
            // how the rows share the lanes, while the copy is on its way
            int32_t steps = 0;
            bool even = false;
            if (T <= cap) {
                int groups = 0;
                for (int32_t k = j; k < jn; k += rl, ++groups) {
                    const int32_t rs = inside(rp[k + lrow], ts, te);
                    const int32_t n = inside(rp[k + lrow + 1], rs, te) - rs - sub;
                    steps += (int32_t)__reduce_max_sync(
                        FULL, (unsigned)(MULTI ? (n + (1 << gl) - 1) >> gl : n));
                }
                even = rows_even(steps, te - ts, groups);
            } else if (MULTI && rl == 1) {
                steps = (te - ts + 31) >> 5;
                even = true;  // a part of one long row
            }
            const int32_t Tp = te - ts;
            const int32_t C = ((Tp + 31) >> 5) | 1;
            bool cont = false;
            if (!even) {
                sc->heads[lane] = 0u;
                __syncwarp();
                const uint32_t inv = 65535u / (uint32_t)C + 1u;  // exact: p * C < 2^16
                int32_t base = 0;
                for (int32_t k = j; k < jn; k += rl) {
                    const int32_t r0 = rp[k + lrow], r1 = rp[k + lrow + 1];
                    const int32_t rs = inside(r0, ts, te), re = inside(r1, rs, te);
                    const bool holder = sub == 0 && re > rs;
                    const unsigned hold = __ballot_sync(FULL, holder);
                    if (holder) {
                        const int rank = base + __popc(hold & ((1u << lane) - 1u));
                        const uint32_t p = (uint32_t)(rs - ts);
                        const uint32_t own = (p * inv) >> 16;
                        sc->seg_row[rank & (kUnitRowsMax - 1)] = (uint8_t)(k + lrow);
                        atomicOr(&sc->heads[own], 1u << (p - own * (uint32_t)C));
                    }
                    base += __popc(hold);
                    // a row that goes on past the stage
                    cont = cont || __any_sync(FULL, holder && re == te && r1 > te && te < ge);
                    // empty rows, once
                    if (sub == 0 && r1 <= r0 && cur.r0 + k + lrow < m &&
                        (T <= cap || te == ge))
                        store(cur.r0 + k + lrow, P::zero());
                }
            }
            if (!mbar_wait_bounded(&sc->bar, phase)) {
                if (lane == 0) atomicOr(a.head + kWordRowErr, SSSPMV_DEV_TIMEOUT);
                mbar_wait_bounded(&sc->bar, phase);  // once more before the stage goes
                return;
            }
            phase ^= 1u;
            __syncwarp();
            const int32_t off = ts & 7;  // the first entry's shared index
            bool done = false;
            if constexpr (SHORT) {
                // up to four groups at once, so that their gathers overlap
                constexpr int GM = kUnitRowsMax / 32;
                int first[GM], n[GM], longest = 0;
#pragma unroll
                for (int g = 0; g < GM; ++g) {
                    const int32_t r = j + 32 * g < jn ? j + 32 * g + lane : j;
                    const int32_t rs = inside(rp[r], ts, te);
                    n[g] = j + 32 * g < jn ? inside(rp[r + 1], rs, te) - rs : 0;
                    first[g] = rs - ts + off;
                    longest = n[g] > longest ? n[g] : longest;
                }
                const int nmax = (int)__reduce_max_sync(FULL, (unsigned)longest);
                if (even && nmax <= kShortRow) {
                    A acc[GM];
#pragma unroll
                    for (int g = 0; g < GM; ++g) acc[g] = P::zero();
                    for (int i = 0; i < nmax; ++i) {
                        X xv[GM];
#pragma unroll
                        for (int g = 0; g < GM; ++g)
                            if (i < n[g]) xv[g] = P::gather(x, scol[first[g] + i], pol_keep);
#pragma unroll
                        for (int g = 0; g < GM; ++g)
                            if (i < n[g]) acc[g] = P::fma(sv[first[g] + i], xv[g], acc[g]);
                    }
#pragma unroll
                    for (int g = 0; g < GM; ++g) {
                        const int32_t r = j + 32 * g + lane;
                        if (j + 32 * g < jn && cur.r0 + r < m) store(cur.r0 + r, acc[g]);
                    }
                    done = true;
                }
            }
            if (done) {
                // stored above
            } else if (even) {
                for (int32_t k = j; k < jn; k += rl) {
                    const int32_t rs = inside(rp[k + lrow], ts, te);
                    const int32_t len = inside(rp[k + lrow + 1], rs, te) - rs;
                    const int32_t n = MULTI ? (len - sub + (1 << gl) - 1) >> gl : len;
                    // (of a single group: counted above)
                    const int32_t nmax = jn == j + rl
                                             ? steps
                                             : (int32_t)__reduce_max_sync(FULL, (unsigned)n);
                    const int32_t nmin = (int32_t)__reduce_min_sync(FULL, (unsigned)n);
                    const int32_t first = rs - ts + off + sub;
                    // rows that start in a few banks only (lengths that are a
                    // multiple of four): each lane starts elsewhere in its row,
                    // or 8 to 32 lanes would read one bank at every step
                    const unsigned banks =
                        __reduce_or_sync(FULL, n > 0 ? 1u << (first & 31) : 0u);
                    A acc;
                    if (__popc(banks) <= 8 && nmax >= 8)
                        acc = lane_dot<P, P::kLaneBatch, MULTI ? 0 : 1, true>(
                            sv + first, scol + first, x, n, nmin, nmax, 1 << gl,
                            n > 0 ? lrow % n : 0, pol_keep, MULTI ? carry : P::zero());
                    else
                        acc = lane_dot<P, P::kLaneBatch, MULTI ? 0 : 1, false>(
                            sv + first, scol + first, x, n, nmin, nmax, 1 << gl, 0, pol_keep,
                            MULTI ? carry : P::zero());
                    if (MULTI && te < ge) {  // a part of one long row: lane by lane
                        carry = acc;
                        continue;
                    }
                    if (MULTI) carry = P::zero();
                    if (MULTI)
                        for (int d = 1; d < (1 << gl); d <<= 1)
                            acc = P::add(acc, P::shfl(acc, lane ^ d));
                    if (sub == 0 && cur.r0 + k + lrow < m) store(cur.r0 + k + lrow, acc);
                }
            } else if (Tp > 0) {
                const A last = even_split<P>(sv + off, scol + off, x, sc, Tp, C, carry, cont,
                                             pol_keep, [&](int r, A v) { store(cur.r0 + r, v); });
                carry = cont ? last : P::zero();
            }
            at = te < ge && T > cap ? te : -1;
            if (at < 0) j = jn;
        }
        if (nxt.nr < 0) nxt = next_unit();
        __syncwarp();  // the stage and the row pointers are free
        cur = nxt;
    }
}

// ---------------------------------------------------------------------------
// (r2): works off the lists.  No shared memory, so that L1 keeps as much of x
// as it can: the listed rows hold most entries of a power-law matrix, whose
// gathers meet in the same few lines (R-MAT scale 22, the listed 48 M entries:
// 210 us; staged in shared memory like (r1)'s, 272 to 400 us with 12 to 16
// warps, following the L1 that was left).

constexpr int kTailThreads = 256;
// Below this many entries two blocks per SM with eight entries per lane at a time,
// from there on three with four.  Few very long rows in many short ones want the
// former at any size measured (8 million entries, 3 rows of 500,000: 58 us and 65;
// 12 million: 75 and 82), as do all matrices up to 5 million (R-MAT scale 16 of
// edge factor 16 19 us and 22, longrows of 4 million 38 and 44); power laws above
// 5.5 million the latter (R-MAT of 8 to 12 million 65 to 100 us and 61 to 93, of
// 66 million 330 and 309; FP32 289 and 266).
constexpr int32_t kTailWide = 15000000;
constexpr int kTailShort = 24;    // rows up to this long: one lane each

template <class T>
__device__ __forceinline__ T ldg_stream(const T *p)
{
    return __ldcs(p);
}
__device__ __forceinline__ __nv_bfloat16 ldg_stream(const __nv_bfloat16 *p)
{
    return __ushort_as_bfloat16(__ldcs(reinterpret_cast<const unsigned short *>(p)));
}

// sums of four rows over the warp, the rows' vectors given one at a time
// (add), with 6 additions instead of 20: after two rows the lower half warp
// holds the first's and the upper half the second's, after four each quarter
// holds one row's.
template <class P>
struct FourRows {
    using A = typename P::acc_t;
    A one, two;
    __device__ __forceinline__ A fold(A lo, A hi, int bit, int lane)
    {
        const bool up = lane & bit;
        return P::add(up ? hi : lo, P::shfl(up ? lo : hi, lane ^ bit));
    }
    __device__ __forceinline__ void add(int q, A v, int lane)
    {
        if (q == 0) one = v;
        else if (q == 1) two = fold(one, v, 16, lane);
        else if (q == 2) one = v;
        else one = fold(one, v, 16, lane);
    }
    // lanes with bit 8 clear hold rows 0 and 1, the others rows 2 and 3
    __device__ __forceinline__ A sum(int lane)
    {
        A t = fold(two, one, 8, lane);
#pragma unroll
        for (int d = 4; d >= 1; d >>= 1) t = P::add(t, P::shfl(t, lane ^ d));
        return t;
    }
};

// lane 0's sum of piece w of row it.x (len entries) is in; the warp that
// brings the row's last piece adds the pieces up, in a fixed order
template <class P>
__device__ __noinline__ void finish_piece(const RowArgs &a, typename P::y_t *y, int32_t pl,
                                          uint32_t w, int2 it, int32_t len, double sum)
{
    using Y = typename P::y_t;
    const int lane = threadIdx.x & 31;
    const int32_t n = row_pieces(len, pl);
    const uint32_t first = w - (uint32_t)it.y;
    uint32_t seen = 0;
    if (lane == 0) {
        __stcg(a.parts + w, sum);
        __threadfence();
        seen = atomicAdd(a.arrived + first, 1u);
    }
    seen = __shfl_sync(FULL, seen, 0);
    if (seen + 1u != (uint32_t)n) return;
    __threadfence();
    double t = 0.0;
    for (int32_t p = lane; p < n; p += 32) t += __ldcg(a.parts + first + p);
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) t += __shfl_xor_sync(FULL, t, d);
    if (lane == 0) {
        y[it.x] = row_value(a, y, it.x, (Y)t);
    }
}

template <class P, int UN, int BLOCKS, bool BATCHED = false>
__global__ void __launch_bounds__(kTailThreads, BLOCKS) rowtail_kernel(const RowArgs a)
{
    using V = typename P::val_t;
    using X = typename P::x_t;
    using Y = typename P::y_t;
    using A = typename P::acc_t;
    grid_dep_wait();
    uint32_t nr = *(volatile const uint32_t *)(a.head + kWordLists);
    uint32_t np = *(volatile const uint32_t *)(a.head + kWordLists + 1);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.head[kWordUnitTicket] = 0u;  // (r1)'s
        // (r1)'s error bits become the call's (beside a batch's set-up's).  They
        // have a word of their own because no block of (r1) could clear the
        // call's word before all the others may set a bit in it.
        const uint32_t bits = *(volatile const uint32_t *)(a.head + kWordRowErr);
        a.head[kWordErr] = BATCHED ? a.head[kWordErr] | bits : bits;
        a.head[kWordRowErr] = 0u;
    }
    if (nr + np == 0u) return;  // every row was staged
    // (an invalid row_ptr may have been refused more than the lists hold)
    nr = nr > (uint32_t)a.max_ranges ? 0u : nr;
    np = np > (uint32_t)a.max_pieces ? 0u : np;
    const int lane = threadIdx.x & 31;
    const V *__restrict__ val = static_cast<const V *>(a.val);
    const X *__restrict__ x = static_cast<const X *>(a.x);
    const int32_t *__restrict__ col = a.col;
    const int32_t *__restrict__ row_ptr = a.row_ptr;
    Y *y = static_cast<Y *>(a.y);
    int32_t m = a.m, nnz = a.nnz;
    int pl = a.shape.piece;
    const uint64_t pol = policy_evict_last();
    auto rp = [&](int32_t r) {
        const int32_t p = __ldg(row_ptr + r);
        return p < 0 ? 0 : (p > nnz ? nnz : p);
    };
    const uint32_t warps = gridDim.x * (kTailThreads / 32);
    // The last ranges, half as many as there are warps, are shared by four
    // warps each (eight if there are few), or most warps would wait for a few
    // at the end (FP32, R-MAT scale 20: 56 us if none are shared, 52 so, 54 if
    // as many as warps are, 62 if those by eight).
    const uint32_t nsub = 8 * nr <= warps ? 8 : 4;
    const uint32_t whole = nr > warps / 2 ? nr - warps / 2 : 0u;
    // the first piece of work by the warp's place, the others by ticket
    uint32_t w = blockIdx.x * (kTailThreads / 32) + (threadIdx.x >> 5);
    const uint32_t total = np + whole + (nr - whole) * nsub;
    // (drawing the next ticket early gave the last ones to busy warps: 56 -> 64 us)
    auto next = [&]() -> uint32_t {
        uint32_t t = 0;
        if (lane == 0) t = warps + atomicAdd(a.head + kWordTailTicket, 1u);
        return __shfl_sync(FULL, t, 0);
    };
    for (; w < total; w = next()) {
        // the entries [s, e) of the lane's row, row0 + lane; a piece of a very
        // long row: lane 0's
        const bool piece = w < np;
        const bool shared = w >= np + whole;
        const uint32_t ri = shared ? whole + (w - np - whole) / nsub : w - np;
        const uint32_t sub = shared ? (w - np - whole) & (nsub - 1) : 0u;
        const int2 it = piece ? a.pieces[w] : a.ranges[ri];
        if constexpr (BATCHED) {
            const RowMat *mm = a.mats + (piece ? a.piece_mat[w] : a.range_mat[ri]);
            val = static_cast<const V *>(ldg_ptr(&mm->val));
            x = static_cast<const X *>(ldg_ptr(&mm->x));
            y = static_cast<Y *>(ldg_ptr(const_cast<void *const *>(&mm->y)));
            col = ldg_ptr(&mm->col);
            row_ptr = ldg_ptr(&mm->row_ptr);
            m = __ldg(&mm->m);
            nnz = __ldg(&mm->nnz);
            pl = __ldg(&mm->packed) >> 16;
        }
        // (whatever the lists hold, nothing outside the arrays is touched)
        const bool in = (piece ? lane == 0 : lane < it.y) &&
                        (uint32_t)it.x + (uint32_t)lane < (uint32_t)m;
        int32_t s = in ? rp(it.x + lane) : 0, e = in ? rp(it.x + lane + 1) : 0;
        const int32_t row_len = e - s;
        unsigned todo;
        if (piece) {
            const bool mine = (uint32_t)it.y <= w && it.y < row_pieces(row_len, pl);
            s += mine ? it.y << pl : 0;
            e = piece_end(s, e, pl);
            todo = __ballot_sync(FULL, lane == 0 && mine);
        } else {
            const bool isshort = in && row_len <= kTailShort;
            if (sub == 0) {
                // short rows: one lane each
                const int32_t n = isshort && row_len > 0 ? row_len : 0;
                const int32_t nmax = (int32_t)__reduce_max_sync(FULL, (unsigned)n);
                A acc = P::zero();
#pragma unroll 1
                for (int32_t i = 0; i < nmax; i += 4) {
                    X xv[4];
                    V v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (i + u < n) {
                            xv[u] = P::gather(x, __ldg(col + s + i + u), pol);
                            v[u] = val[s + i + u];
                        }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (i + u >= nmax) break;
                        if (i + u < n) acc = P::fma(v[u], xv[u], acc);
                    }
                }
                if (isshort)
                    y[it.x + lane] = row_value(a, y, it.x + lane, P::out(acc));
            }
            todo = __ballot_sync(FULL, in && !isshort && row_len <= (1 << pl));
        }
        // the longer rows, every nsub-th from the sub-th on, 32 * UN entries at a
        // time: the values and columns of a block of entries, be it the row's
        // or the next row's, are loaded while the block before it gathers
        if (shared) {
            unsigned mine = 0;
            for (uint32_t k = 0; todo; ++k, todo &= todo - 1)
                if ((k & (nsub - 1)) == sub) mine |= todo & -todo;
            todo = mine;
        }
        int32_t k = 0, n = 0;  // the block's first entry, and the row's entries from there on
        int f = 0;             // its row
        auto advance = [&]() -> bool {
            k += 32 * UN;
            n -= 32 * UN;
            if (n > 0) return true;
            if (!todo) return false;
            f = __ffs(todo) - 1;
            todo &= todo - 1;
            k = __shfl_sync(FULL, s, f);
            n = __shfl_sync(FULL, e, f) - k;
            return true;
        };
        int32_t c[UN];
        V v[UN];
        auto load = [&]() {
#pragma unroll
            for (int u = 0; u < UN; ++u)
                if (lane + 32 * u < n) {
                    c[u] = ldg_stream(col + k + lane + 32 * u);
                    v[u] = ldg_stream(val + k + lane + 32 * u);
                }
        };
        bool more = advance();
        if (more) load();
        FourRows<P> r4;
        A acc = P::zero();
        int q = 0;
        int32_t src = -1;  // the row whose sum the lane gets to hold
#pragma unroll 1
        while (more) {
            const int32_t left = n;
            const int row = f;
            X xv[UN];
            V vv[UN];
#pragma unroll
            for (int u = 0; u < UN; ++u) {
                if (lane + 32 * u < left) xv[u] = P::gather(x, c[u], pol);
                vv[u] = v[u];
            }
            more = advance();
            if (more) load();
#pragma unroll
            for (int u = 0; u < UN; ++u) {
                if (32 * u >= left) break;  // the same for the whole warp
                if (lane + 32 * u < left) acc = P::fma(vv[u], xv[u], acc);
            }
            if (left > 32 * UN) continue;
            // the row is complete
            if (q == (((lane >> 4) & 1) | ((lane >> 2) & 2))) src = row;
            r4.add(q, acc, lane);
            acc = P::zero();
            ++q;
            if (q < 4 && more) continue;
            for (; q < 4; ++q) r4.add(q, acc, lane);
            const A t = r4.sum(lane);
            if (piece) {
                finish_piece<P>(a, y, pl, w, it, __shfl_sync(FULL, row_len, 0), P::to_f64(t));
            } else if ((lane & 7) == 0 && src >= 0) {
                const int32_t r = it.x + src;
                y[r] = row_value(a, y, r, P::out(t));
            }
            q = 0;
            src = -1;
        }
    }
    // the last block leaves the list words as it found them: zero
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(a.head + kWordTailDone, 1u) == gridDim.x - 1u) {
            a.head[kWordLists] = 0u;
            a.head[kWordLists + 1] = 0u;
            a.head[kWordTailTicket] = 0u;
            a.head[kWordTailDone] = 0u;
        }
    }
}

// ---------------------------------------------------------------------------
// host side

// whether the lists of this call's row blocks fit the workspace of its layout
inline bool row_lists_fit(int32_t nnz, const RowShape &s, const Layout &l)
{
    return row_lists(nnz, s.cap, s.piece).bytes <= l.total - l.off_tile_offset;
}

struct StageShape {
    int32_t bytes, col_off, warps;
};

// a warp's stage for `cap` entries, and how many warps shared memory holds
template <class P>
StageShape stage_shape(int32_t cap, int32_t budget)
{
    StageShape s;
    const int32_t entries = cap + 8;
    s.col_off = (entries * (int32_t)sizeof(typename P::val_t) + 15) & ~15;
    s.bytes = (s.col_off + entries * 4 + 127) & ~127;
    s.warps = budget / (s.bytes + (int32_t)sizeof(RowScratch));
    return s;
}

template <class K>
cudaError_t allow_smem(K kernel, int (&done)[64])
{
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = 1;
    return e;
}

template <class P, bool MULTI, bool BATCHED = false, bool SHORT = false>
int launch_rowblock(const Call &c, const RowArgs &a)
{
    static int done[64] = {0};
    cudaError_t e = allow_smem(rowblock_kernel<P, MULTI, BATCHED, SHORT>, done);
    if (e != cudaSuccess) return record_cuda_error(e);
    // A gather that misses L1 holds one of its lines until it is served, so L1
    // has to be large enough for the gathers in flight: with all of shared
    // memory in stages (28 KB of L1) random columns ran at 137 G gathers/s,
    // with 194 KB (60 KB) at 205, with 162 KB (92 KB) at 230; a stencil, whose
    // lanes share lines, prefers warps (160^3: 235, 250 and 271 us).  The
    // larger L1 for rows of up to four entries, which are graphs more often
    // than grids.
    const int32_t budget = ((int64_t)a.nnz > 4 * (int64_t)a.m ? 194 : 162) * 1024;
    const StageShape s = stage_shape<P>(a.shape.cap, budget);
    constexpr int32_t most = BATCHED ? kBatchRowWarps : P::kRowWarps;
    int32_t warps = s.warps < most ? s.warps : most;
    const int sms = device_sm_count();
    const unsigned grid = (unsigned)(a.nunits < sms ? a.nunits : sms);
    const int32_t need = (int32_t)((a.nunits + (int64_t)grid - 1) / grid);
    if (warps > need) warps = need;
    e = launch_dependent(rowblock_kernel<P, MULTI, BATCHED, SHORT>, grid, (unsigned)warps * 32,
                         (size_t)warps * (s.bytes + sizeof(RowScratch)), c.stream, a, s.bytes,
                         s.col_off);
    return e == cudaSuccess ? SSSPMV_OK : record_cuda_error(e);
}

// (r2) with at most one wave of blocks: a warp per listed range or piece
template <class P, int UN, int BLOCKS, bool BATCHED = false>
int launch_rowtail(const Call &c, const RowArgs &a)
{
    auto k2 = rowtail_kernel<P, UN, BLOCKS, BATCHED>;
    static int blocks[64] = {0};  // resident per SM
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    if (blocks[dev] <= 0) {
        int n = 0;
        if (cudaFuncSetAttribute(k2, cudaFuncAttributePreferredSharedMemoryCarveout, 0) !=
                cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k2, kTailThreads, 0) !=
                cudaSuccess ||
            n < 1) {
            (void)cudaGetLastError();
            n = 1;
        }
        blocks[dev] = n;
    }
    // (few ranges are shared by up to eight warps each)
    const int64_t work = 8 * (int64_t)a.max_ranges + a.max_pieces;
    int64_t grid = (int64_t)blocks[dev] * device_sm_count();
    const int64_t need = (work + kTailThreads / 32 - 1) / (kTailThreads / 32);
    if (grid > need) grid = need;
    const cudaError_t e = launch_dependent(k2, (unsigned)grid, kTailThreads, 0, c.stream, a);
    return e == cudaSuccess ? SSSPMV_OK : record_cuda_error(e);
}

// y = A x by row blocks: (r1) and (r2).  The header's list words are zero when
// it starts and when it ends.
template <class P>
int run_rowblock(const Call &c)
{
    cudaError_t e = cudaSuccess;
    if (c.ev && (e = cudaEventRecord(c.ev[0], c.stream)) != cudaSuccess)
        return record_cuda_error(e);
    if (c.ev && (e = cudaEventRecord(c.ev[1], c.stream)) != cudaSuccess)
        return record_cuda_error(e);
    RowArgs a;
    a.shape = row_shape(c.m, c.nnz, (int32_t)sizeof(typename P::val_t));
    const RowLists rl = row_lists(c.nnz, a.shape.cap, a.shape.piece);
    unsigned char *lists = c.ws + c.lay.off_tile_offset;
    a.row_ptr = c.row_ptr;
    a.col = c.col;
    a.val = c.val;
    a.x = c.x;
    a.y = c.y;
    a.head = reinterpret_cast<uint32_t *>(c.ws + c.lay.off_err);
    a.ranges = reinterpret_cast<int2 *>(lists + rl.off_ranges);
    a.pieces = reinterpret_cast<int2 *>(lists + rl.off_pieces);
    a.parts = reinterpret_cast<double *>(lists + rl.off_parts);
    a.arrived = reinterpret_cast<uint32_t *>(lists + rl.off_arrived);
    a.max_ranges = (int32_t)rl.ranges;
    a.max_pieces = (int32_t)rl.pieces;
    a.m = c.m;
    a.nnz = c.nnz;
    const RowUnits units = row_units(c.m, c.nnz, a.shape);
    a.nbig = units.nbig;
    a.nunits = units.nunits;
    a.alpha = c.alpha;
    a.beta = c.beta;
    a.axpby = c.axpby;
    int rc = SSSPMV_OK;
    if (a.shape.gs > 0) rc = launch_rowblock<P, true>(c, a);
    else if (c.m >= kShortRows && (int64_t)c.nnz <= 3 * (int64_t)c.m)
        rc = launch_rowblock<P, false, false, true>(c, a);
    else rc = launch_rowblock<P, false>(c, a);
    if (rc) return rc;
    if (c.ev && (e = cudaEventRecord(c.ev[2], c.stream)) != cudaSuccess)
        rc = record_cuda_error(e);
    if (!rc) rc = c.nnz < kTailWide ? launch_rowtail<P, 8, 2>(c, a) : launch_rowtail<P, 4, 3>(c, a);
    if (rc) {
        // (r1) has run and (r2) will not (its first launch loads it, and may find
        // no memory): the counters (r1) leaves must not meet the next call
        (void)cudaMemsetAsync(a.head, 0, kHeaderBytes, c.stream);
        return rc;
    }
    if (c.ev && (e = cudaEventRecord(c.ev[3], c.stream)) != cudaSuccess)
        return record_cuda_error(e);
    e = cudaGetLastError();
    return e == cudaSuccess ? SSSPMV_OK : record_cuda_error(e);
}

}  // namespace ssspmv
