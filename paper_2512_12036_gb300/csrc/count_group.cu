// Intermediate-product counting (Algorithm 1), row grouping (Section III-B)
// and the row-pointer scan of the allocation phase.
#include "internal.h"

namespace spg {

// ---------------------------------------------------------------------------
// Small utilities
// ---------------------------------------------------------------------------

template <typename T>
__global__ void k_sum_to(const T* x, long long n, long long* out) {
    __shared__ long long red[33];
    long long acc = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        acc += (long long)x[i];
    acc = block_sum(acc, red);
    if (threadIdx.x == 0 && acc != 0) atomicAdd((unsigned long long*)out, (unsigned long long)acc);
}

__global__ void k_zero_total(Ctl* ctl, int which) { ctl->totals[which] = 0; }

// ---------------------------------------------------------------------------
// Algorithm 1, balanced over nonzeros: each block takes a tile of A's stored
// entries, so a row of 60k entries costs the same as 60k rows of one entry.
// The lengths of the selected B rows are gathered (eight in flight per
// thread) and scanned over the tile; a row's count is then a difference of
// two prefixes, written directly when the row lies inside the tile and added
// otherwise. (A binary search for the row of every entry and segmented warp
// sums took 111 us on 11.5M entries of 589,000 rows; 69 us now.)
// ---------------------------------------------------------------------------

constexpr int kCountThreads = 256;
constexpr int kCountItems = 8;
constexpr int kCountTile = kCountThreads * kCountItems;

// The last row in [0, hi] that starts at or before entry j, by one warp: 32
// probes a step.
__device__ __forceinline__ int row_of(const int* rpt, long long j, int hi) {
    const int lane = lane_id();
    int lo = 0;
    while (lo < hi) {
        const int step = (hi - lo + 33) / 33;    // 33 steps cover [lo, hi]
        const int p = lo + (lane + 1) * step;
        const int c = __popc(__ballot_sync(kFull, p <= hi && (long long)rpt[p <= hi ? p : hi] <= j));
        lo += c * step;
        hi = min(hi, lo + step - 1);
    }
    return lo;
}

__global__ void __launch_bounds__(kCountThreads) k_ip_count(CsrDev A, CsrDev B, long long* ip,
                                                            Ctl* ctl) {
    __shared__ int s_r[2];
    __shared__ int s_len[kCountTile + kCountTile / 32];          // (padded: thread t reads 8t ..)
    __shared__ unsigned long long s_pre[kCountTile + 1];
    __shared__ unsigned long long scratch[33];
    const int m = A.rows;
    const long long J0 = A.rpt[0], J1 = A.rpt[m];
    if (J0 < 0 || J1 < J0 || J1 > A.nnz) {
        if (blockIdx.x == 0 && threadIdx.x == 0) set_status(ctl, ST_INVALID);
        return;
    }
    const long long jb = J0 + (long long)blockIdx.x * kCountTile;
    if (jb >= J1) return;
    const long long je = jb + kCountTile < J1 ? jb + kCountTile : J1;
    const int t = threadIdx.x;
    // the tile's first and last row, searched while the lengths are gathered
    if ((t >> 5) < 2) {
        const int r = row_of(A.rpt, (t >> 5) == 0 ? jb : je - 1, m - 1);
        if (lane_id() == 0) s_r[t >> 5] = r;
    }
    int len[kCountItems];
#pragma unroll
    for (int q = 0; q < kCountItems; ++q) {
        const long long j = jb + q * kCountThreads + t;
        int bs;
        len[q] = 0;
        if (j < je) a_entry(A, B, (int)j, bs, len[q], ctl);
    }
#pragma unroll
    for (int q = 0; q < kCountItems; ++q) {
        const int p = q * kCountThreads + t;
        s_len[p + (p >> 5)] = len[q];
    }
    __syncthreads();
    unsigned long long sum = 0;
#pragma unroll
    for (int q = 0; q < kCountItems; ++q) {
        const int p = t * kCountItems + q;
        len[q] = s_len[p + (p >> 5)];
        sum += (unsigned)len[q];
    }
    unsigned long long tot;
    unsigned long long run = block_excl_scan_u64(sum, scratch, &tot);
#pragma unroll
    for (int q = 0; q < kCountItems; ++q) {
        s_pre[t * kCountItems + q] = run;
        run += (unsigned)len[q];
    }
    if (t == kCountThreads - 1) s_pre[kCountTile] = run;
    __syncthreads();
    const int r1 = s_r[1];
    for (int r = s_r[0] + t; r <= r1; r += kCountThreads) {
        const long long s = A.rpt[r], e = A.rpt[r + 1];
        // (row pointers out of order were flagged; they stay inside the tile here)
        const long long a = s > jb ? (s < je ? s : je) : jb, b = e < je ? (e > a ? e : a) : je;
        const unsigned long long v = s_pre[b - jb] - s_pre[a - jb];
        if (s >= jb && e <= je) ip[r] = (long long)v;
        else if (v != 0) atomicAdd((unsigned long long*)&ip[r], v);
    }
    if (t == 0 && tot != 0) atomicAdd((unsigned long long*)&ctl->totals[0], tot);
}

// One pass over the rows before the count: zero counts, both operands' row
// pointers checked, the total reset.
__global__ void k_count_prep(CsrDev A, CsrDev B, long long* ip, Ctl* ctl) {
    const long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long step = (long long)gridDim.x * blockDim.x;
    if (i0 == 0) ctl->totals[0] = 0;
    bool bad = false;
    for (long long i = i0; i < A.rows; i += step) {
        const int s = A.rpt[i], e = A.rpt[i + 1];
        bad |= s < 0 || e < s || (long long)e > A.nnz;
        ip[i] = 0;
    }
    for (long long i = i0; i < B.rows; i += step) {
        const int s = B.rpt[i], e = B.rpt[i + 1];
        bad |= s < 0 || e < s || (long long)e > B.nnz;
    }
    if (bad) set_status(ctl, ST_INVALID);
}

// Row pointers must be monotone and inside [0, nnz].
__global__ void k_check_rpt(CsrDev M, Ctl* ctl) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < M.rows;
         i += (long long)gridDim.x * blockDim.x) {
        const int s = M.rpt[i], e = M.rpt[i + 1];
        if (s < 0 || e < s || (long long)e > M.nnz) set_status(ctl, ST_INVALID);
    }
}

void launch_check_rpt(const spgemm_plan* p, const CsrDev& M, const WsPtrs& w, cudaStream_t s) {
    if (M.rows == 0) return;
    const int blocks = (M.rows + 255) / 256 < 4096 ? (M.rows + 255) / 256 : 4096;
    SPG_LAUNCH(p, K_CHECK_RPT, s, k_check_rpt<<<blocks, 256, 0, s>>>(M, w.ctl));
}

void launch_ip_count(const spgemm_plan* p, const CsrDev& A, const CsrDev& B, long long* ip,
                     const WsPtrs& w, cudaStream_t s) {
    if (A.rows == 0) return;
    const int rows = A.rows > B.rows ? A.rows : B.rows;
    const int blocks = (rows + 255) / 256 < 4096 ? (rows + 255) / 256 : 4096;
    SPG_LAUNCH(p, K_CHECK_RPT, s, k_count_prep<<<blocks, 256, 0, s>>>(A, B, ip, w.ctl));
    if (A.nnz > 0) {
        const long long tiles = (A.nnz + kCountTile - 1) / kCountTile;
        SPG_LAUNCH(p, K_IP_COUNT, s, k_ip_count<<<(unsigned)tiles, kCountThreads, 0, s>>>(A, B, ip, w.ctl));
    }
}

void launch_nnz_total(const spgemm_plan* p, const int* row_nnz, int n, const WsPtrs& w, cudaStream_t s) {
    SPG_LAUNCH(p, K_ZERO, s, k_zero_total<<<1, 1, 0, s>>>(w.ctl, 1));
    if (n > 0) SPG_LAUNCH(p, K_SUM, s, k_sum_to<int><<<256, 256, 0, s>>>(row_nnz, n, &w.ctl->totals[1]));
}

// ---------------------------------------------------------------------------
// Row grouping. Every row gets a bin id; the map is a stable partition of
// the rows by bin (ascending bin, ascending row inside a bin), built from
// per-block histograms, one exclusive scan over (bin, block) and a scatter
// that ranks rows inside a warp with __match_any_sync. One pass of atomics
// in shared memory per block replaces the per-row global atomics that the
// paper names as the grouping phase's cost.
// ---------------------------------------------------------------------------

__device__ __forceinline__ int clampi(int x, int lo, int hi) { return x < lo ? lo : (x > hi ? hi : x); }

__device__ __forceinline__ int bin_of(const GroupArgs& g, int r, bool settle) {
    if (g.phase == 2) {
        const long long k = g.key[r];
        int b = 0;
        while (b < g.nthr && k >= g.thr[b]) ++b;
        return b;
    }
    if (g.phase == 3) {       // backward tiers, by nnz of row r of C
        const int nc = g.rptC[r + 1] - g.rptC[r];
        if (nc <= 0) return kSkipBin;
        if (g.bcols <= kBwdDenseCols) return BW_DENSE;
        if (nc <= kBwdWarpSlots / 2) return BW_WARP;
        if (nc <= kBwdBlockSlots / 2) return BW_BLOCK;
        return BW_PANEL;
    }
    const int row = g.row_begin + r;
    const long long ip = g.ip[row];
    const int na = g.rptA[row + 1] - g.rptA[row];
    const spgemm_opts& o = g.opts;
    if (g.phase == 0) {
        // settled here, but for a row of one product that the accumulation phase
        // takes in the narrow tier: that one reads the row's bitmap, which only
        // the allocation phase's narrow tier writes
        if (ip < 1 || (ip == 1 && (na <= o.esc_max || g.bcols > kNarrowCols))) {
            if (settle) g.row_nnz[row] = ip < 0 ? 0 : (int)ip;
            return kSkipBin;
        }
        if (ip <= o.esc_max && na <= o.esc_max) return SB_ESC;
        if (g.bcols <= kNarrowCols && ip <= narrow_max_ip(o)) return SB_NARROW;
        if (ip <= sort_max_ip(o.warp_max_ip / 2)) return ip <= sort_max_ip(o.warp_max_ip / 2) / 2 ? SB_SORTA : SB_SORTB;
        if (ip <= o.warp_max_ip) return SB_WARP;
        const int L = log2_ceil_ll(ip);
        if (ip <= o.block_max_ip) {
            const int Lmax = log2_ceil_ll(o.block_max_ip);
            return SB_BLOCK0 + clampi(Lmax - L, 0, SB_BLOCK_N - 1);
        }
        return SB_DENSE0 + clampi(46 - L, 0, SB_DENSE_N - 1);
    }
    const int nnz = g.rptC[r + 1] - g.rptC[r];
    if (nnz <= 0) return kSkipBin;
    const bool f64 = na > o.fp32_max_terms && ip > o.fp32_max_terms;
    if (ip <= o.esc_max && na <= o.esc_max) return NB_ESC;
    if (g.bcols <= kNarrowCols && ip <= narrow_max_ip(o)) return f64 ? NB_NARROW64 : NB_NARROW32;
    if (ip <= sort_max_ip(o.warp_max_nnz) && g.bcols < kSortCols) {
        if (ip <= sort_max_ip(o.warp_max_nnz) / 2) return f64 ? NB_SORT64A : NB_SORT32A;
        return f64 ? NB_SORT64B : NB_SORT32B;
    }
    if (ip <= 16ll * o.warp_max_nnz) {
        if (nnz <= o.warp_max_nnz / 2) return f64 ? NB_WARP64S : NB_WARP32S;
        if (nnz <= o.warp_max_nnz) return f64 ? NB_WARP64 : NB_WARP32;
        // fp32 rows of up to twice that stay with one warp: a block's barriers
        // cost a row of this size more than the longer sort of one warp
        // (131,072 rows of 1,075 products, 600-900 entries: 4,562 us by
        // 512-thread blocks, 3,827 us by warps)
        if (!f64 && nnz <= 2 * o.warp_max_nnz && nnz <= o.block_max_nnz) return NB_WARP32L;
    }
    if (nnz <= block_small_nnz(o)) return f64 ? NB_BLOCK64S : NB_BLOCK32S;
    if (nnz <= block_mid_nnz(o)) return f64 ? NB_BLOCK64M : NB_BLOCK32M;
    if (nnz <= o.block_max_nnz) return f64 ? NB_BLOCK64 : NB_BLOCK32;
    if (!f64 && nnz <= g.bits_cap) return NB_BITS32;
    const int L = log2_ceil_ll(ip);
    return (f64 ? NB_DENSE64_0 : NB_DENSE32_0) + clampi(kDenseTopLog - L, 0, NB_DENSE_N - 1);
}

__global__ void __launch_bounds__(kBinRows) k_group_hist(GroupArgs g, int nblk, int* blk_counts) {
    __shared__ int hist[kNumBins];
    if (threadIdx.x < kNumBins) hist[threadIdx.x] = 0;
    __syncthreads();
    const int r = blockIdx.x * kBinRows + threadIdx.x;
    if (r < g.n) atomicAdd(&hist[bin_of(g, r, true)], 1);
    __syncthreads();
    if (threadIdx.x < kNumBins) blk_counts[threadIdx.x * nblk + blockIdx.x] = hist[threadIdx.x];
}

// A block per bin: exclusive scan of the bin's block counts in place and the
// bin's rows into ctl->bin_rows (one block over all 64 bins was a chain of 72
// barriers for 1,150 row blocks, 27 us; under 3 us now).
constexpr int kGroupScanThreads = 256;

__global__ void __launch_bounds__(kGroupScanThreads) k_group_scan(int nblk, int* blk_counts, Ctl* ctl) {
    __shared__ int scratch[33];
    int* counts = blk_counts + (long long)blockIdx.x * nblk;
    int carry = 0;
    for (int base = 0; base < nblk; base += kGroupScanThreads) {
        const int i = base + threadIdx.x;
        const int v = i < nblk ? counts[i] : 0;
        int tot;
        const int ex = block_excl_scan(v, scratch, &tot);
        if (i < nblk) counts[i] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0) ctl->bin_rows[blockIdx.x] = carry;
    // (the scatter, which follows, sets the flags)
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->dense_wide = ctl->dense_uncached = 0;
}

// Bin starts from the bins' row counts, by one warp: base[b] for every bin in
// shared memory and, from one block of the launch, ctl->bin_off (offsets_out
// for the public grouping call) and the tiers' row counters.
__device__ __forceinline__ void group_bases(const int* rows, int* base, bool write, Ctl* ctl,
                                            int* offsets_out, int ngroups) {
    const int lane = lane_id();
    const int a = rows[2 * lane], b = rows[2 * lane + 1];
    const int incl = warp_incl_scan(a + b), ex = incl - a - b;
    base[2 * lane] = ex;
    base[2 * lane + 1] = ex + a;
    if (!write) return;
    ctl->bin_off[2 * lane] = ex;
    ctl->bin_off[2 * lane + 1] = ex + a;
    if (lane == 31) ctl->bin_off[kNumBins] = incl;
    if (lane < kMaxTiers) ctl->work[lane] = 0;
    if (offsets_out) {
        const int total = __shfl_sync(kFull, incl, 31);
        for (int q = 0; q < 2; ++q) {
            const int g = 2 * lane + q;
            if (g <= ngroups) offsets_out[g] = g == ngroups ? total : (q ? ex + a : ex);
        }
    }
}

// accumulation: flag an fp32 dense row too wide for the rank-compacted
// kernel, so the fallback kernel runs only when it has rows, and an
// fp64-bound dense row without a cached bitmap, so the kernel for those runs
// only when there are some
__device__ __forceinline__ void group_flags(const GroupArgs& g, int r, int b, Ctl* ctl) {
    if (g.phase != 1 || b < 0) return;
    // (no tier is launched for rows of more entries than B has columns)
    if (g.rptC[r + 1] - g.rptC[r] > g.bcols) set_status(ctl, ST_INTERNAL);
    if (b >= NB_DENSE32_0 && b < NB_DENSE32_0 + NB_DENSE_N) {
        const int row = g.row_begin + r;
        if (g.rptA[row + 1] - g.rptA[row] > kRankTileEntries) ctl->dense_wide = 1;
    }
    if (b >= NB_DENSE64_0 && b < NB_DENSE64_0 + NB_DENSE_N &&
        (g.rc_slot == nullptr || g.rc_slot[g.row_begin + r] < 0))
        ctl->dense_uncached = 1;
}

__global__ void __launch_bounds__(kBinRows) k_group_scatter(GroupArgs g, int nblk,
                                                            const int* blk_counts, int* map,
                                                            Ctl* ctl, int* offsets_out,
                                                            int ngroups) {
    __shared__ int wcount[kBinRows / 32][kNumBins];
    __shared__ int base[kNumBins];
    const int warp = threadIdx.x >> 5;
    if (warp == 0) group_bases(ctl->bin_rows, base, blockIdx.x == 0, ctl, offsets_out, ngroups);
    for (int i = threadIdx.x; i < (kBinRows / 32) * kNumBins; i += blockDim.x)
        (&wcount[0][0])[i] = 0;
    __syncthreads();
    const int r = blockIdx.x * kBinRows + threadIdx.x;
    const int b = r < g.n ? bin_of(g, r, false) : -1;
    group_flags(g, r, b, ctl);
    const unsigned peers = __match_any_sync(kFull, b);
    const int rank = __popc(peers & lanemask_lt());
    if (b >= 0 && rank == 0) wcount[warp][b] = __popc(peers);
    __syncthreads();
    if (threadIdx.x < kNumBins) {
        int acc = 0;
        for (int w = 0; w < kBinRows / 32; ++w) {
            const int c = wcount[w][threadIdx.x];
            wcount[w][threadIdx.x] = acc;
            acc += c;
        }
    }
    __syncthreads();
    if (b >= 0) map[base[b] + blk_counts[(long long)b * nblk + blockIdx.x] + wcount[warp][b] + rank] = r;
}

// The whole grouping of up to kGroupSmallRows rows in one block, thread t
// taking rows t, t + 1024, ...: one launch instead of three, which is what a
// small product waits for. Same map: rows of a bin in ascending order.
constexpr int kGroupSmallRows = 8 * kBinRows;

__global__ void __launch_bounds__(kBinRows) k_group_small(GroupArgs g, int* map, Ctl* ctl,
                                                          int* offsets_out, int ngroups) {
    constexpr int kChunks = kGroupSmallRows / kBinRows;
    __shared__ int wcount[kBinRows / 32][kNumBins];
    __shared__ int base[kNumBins], total[kNumBins];
    const int t = threadIdx.x, warp = t >> 5;
    int bins[kChunks];
    if (t < kNumBins) total[t] = 0;
    __syncthreads();
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
        const int r = c * kBinRows + t;
        bins[c] = -1;
        if (c * kBinRows < g.n) {                     // block-uniform
            if (r < g.n) bins[c] = bin_of(g, r, true);
            const unsigned peers = __match_any_sync(kFull, bins[c]);
            if (bins[c] >= 0 && (peers & lanemask_lt()) == 0) atomicAdd(&total[bins[c]], __popc(peers));
        }
    }
    __syncthreads();
    if (warp == 0) group_bases(total, base, true, ctl, offsets_out, ngroups);
    if (t == 32) ctl->dense_wide = ctl->dense_uncached = 0;
    __syncthreads();                                 // (flags are reset before they are set)
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
        if (c * kBinRows >= g.n) break;              // block-uniform
        for (int i = t; i < (kBinRows / 32) * kNumBins; i += kBinRows) (&wcount[0][0])[i] = 0;
        __syncthreads();
        const int r = c * kBinRows + t, b = bins[c];
        group_flags(g, r, b, ctl);
        const unsigned peers = __match_any_sync(kFull, b);
        const int rank = __popc(peers & lanemask_lt());
        if (b >= 0 && rank == 0) wcount[warp][b] = __popc(peers);
        __syncthreads();
        if (t < kNumBins) {
            int acc = base[t];
            for (int w = 0; w < kBinRows / 32; ++w) {
                const int n = wcount[w][t];
                wcount[w][t] = acc;
                acc += n;
            }
            base[t] = acc;
        }
        __syncthreads();
        if (b >= 0) map[wcount[warp][b] + rank] = r;
        __syncthreads();
    }
}

void launch_group(const spgemm_plan* p, const GroupArgs& g, const WsPtrs& w, int* map_out,
                  int* offsets_out, cudaStream_t s) {
    const int nblk = (g.n + kBinRows - 1) / kBinRows;
    if (g.n <= kGroupSmallRows) {
        SPG_LAUNCH(p, K_GROUP_SCATTER, s,
                   k_group_small<<<1, kBinRows, 0, s>>>(g, map_out, w.ctl, offsets_out,
                                                        g.phase == 2 ? g.nthr + 1 : 0));
        return;
    }
    SPG_LAUNCH(p, K_GROUP_HIST, s, k_group_hist<<<nblk, kBinRows, 0, s>>>(g, nblk, w.blk_counts));
    SPG_LAUNCH(p, K_GROUP_SCAN, s,
               k_group_scan<<<kNumBins, kGroupScanThreads, 0, s>>>(nblk, w.blk_counts, w.ctl));
    SPG_LAUNCH(p, K_GROUP_SCATTER, s,
               k_group_scatter<<<nblk, kBinRows, 0, s>>>(g, nblk, w.blk_counts, map_out, w.ctl, offsets_out,
                                                         g.phase == 2 ? g.nthr + 1 : 0));
}

// ---------------------------------------------------------------------------
// Row pointers: exclusive scan of int32 counts with an int64 running total
// (reduce, scan of block sums, local scan). Overflow past INT32_MAX is
// flagged; the caller then works on blocks of rows.
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(1024) k_scan_part(const int* x, int n, long long* part) {
    __shared__ long long red[33];
    const long long base = (long long)blockIdx.x * kScanItems;
    long long acc = 0;
    for (int i = threadIdx.x; i < kScanItems; i += blockDim.x) {
        const long long q = base + i;
        if (q < n) acc += x[q];
    }
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

__device__ __forceinline__ long long block_excl_scan64(long long v, long long* scratch,
                                                       long long* total) {
    const int lane = lane_id(), warp = threadIdx.x >> 5, nwarps = (blockDim.x + 31) >> 5;
    long long incl = warp_incl_scan64(v);
    if (lane == 31) scratch[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        long long wv = lane < nwarps ? scratch[lane] : 0;
        long long wi = warp_incl_scan64(wv);
        scratch[lane] = wi - wv;
        if (lane == 31) scratch[32] = wi;
    }
    __syncthreads();
    const long long r = scratch[warp] + incl - v;
    *total = scratch[32];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(1024) k_scan_top(long long* part, int nscan, Ctl* ctl,
                                                   int* row_ptr, int n) {
    __shared__ long long scratch[33];
    long long carry = 0;
    for (int base = 0; base < nscan; base += blockDim.x) {
        const int i = base + threadIdx.x;
        const long long v = i < nscan ? part[i] : 0;
        long long tot;
        const long long ex = block_excl_scan64(v, scratch, &tot);
        if (i < nscan) part[i] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0) {
        part[nscan] = carry;
        ctl->totals[2] = carry;
        if (carry > 2147483647ll) set_status(ctl, ST_OVERFLOW);
        row_ptr[n] = (int)carry;
    }
}

__global__ void __launch_bounds__(1024) k_scan_final(const int* x, int n, const long long* part,
                                                     int* row_ptr) {
    __shared__ long long scratch[33];
    constexpr int kPer = kScanItems / 1024;
    const long long base = (long long)blockIdx.x * kScanItems + (long long)threadIdx.x * kPer;
    int v[kPer];
    long long sum = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        v[q] = base + q < n ? x[base + q] : 0;
        sum += v[q];
    }
    long long tot;
    long long ex = block_excl_scan64(sum, scratch, &tot) + part[blockIdx.x];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        if (base + q < n) row_ptr[base + q] = (int)ex;
        ex += v[q];
    }
}

// The three steps in one block for up to kScanSmall rows (one launch).
constexpr int kScanSmall = 4 * kScanItems;

__global__ void __launch_bounds__(1024) k_scan_small(const int* x, int n, Ctl* ctl, int* row_ptr) {
    __shared__ long long scratch[33];
    constexpr int kPer = kScanItems / 1024;
    long long carry = 0;
    for (int b0 = 0; b0 < n; b0 += kScanItems) {
        const int base = b0 + (int)threadIdx.x * kPer;
        int v[kPer];
        long long sum = 0;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            v[q] = base + q < n ? x[base + q] : 0;
            sum += v[q];
        }
        long long tot;
        long long ex = carry + block_excl_scan64(sum, scratch, &tot);
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            if (base + q < n) row_ptr[base + q] = (int)ex;
            ex += v[q];
        }
        carry += tot;
    }
    if (threadIdx.x == 0) {
        ctl->totals[2] = carry;
        if (carry > 2147483647ll) set_status(ctl, ST_OVERFLOW);
        row_ptr[n] = (int)carry;
    }
}

void launch_row_ptr(const spgemm_plan* p, const int* row_nnz, int n, const WsPtrs& w,
                    int* row_ptr, cudaStream_t s) {
    if (n <= kScanSmall) {
        SPG_LAUNCH(p, K_SCAN_TOP, s, k_scan_small<<<1, 1024, 0, s>>>(row_nnz, n, w.ctl, row_ptr));
        return;
    }
    const int nscan = (n + kScanItems - 1) / kScanItems;
    if (nscan > 0)
        SPG_LAUNCH(p, K_SCAN_PART, s, k_scan_part<<<nscan, 1024, 0, s>>>(row_nnz, n, w.scan_part));
    SPG_LAUNCH(p, K_SCAN_TOP, s,
               k_scan_top<<<1, 1024, 0, s>>>(w.scan_part, nscan, w.ctl, row_ptr, n));
    if (nscan > 0)
        SPG_LAUNCH(p, K_SCAN_FINAL, s,
                   k_scan_final<<<nscan, 1024, 0, s>>>(row_nnz, n, w.scan_part, row_ptr));
}

}  // namespace spg
