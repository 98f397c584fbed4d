// Narrow tiers: B with at most kNarrowCols columns (the GNN feature
// matrices), rows of up to narrow_max_ip products, one warp per row, both
// phases.
//
// Allocation phase: a row's columns are the union of its B rows' columns, so
// when A has enough entries to pay for it B's rows are first turned into
// bitmaps (one pass over B's columns) and a row of C is the OR of one bitmap
// per A entry: 32 bytes an entry at 256 columns where the products' columns
// are 4 bytes each. Otherwise the products are marked one by one. C's bitmap is
// kept for the accumulation phase where the workspace has room for it (the
// place of the dense tiers' tables, 20 bytes per entry of B); without it that
// phase marks a row's products again. The two phases' narrow tiers hold the
// same rows, down to a row of one product among many A entries: the grouping
// rules have to agree, or a row would read a bitmap that nobody wrote.
//
// Accumulation phase: a dense accumulator over B's columns per warp. A B row
// without a repeated column touches every accumulator at most once, so its
// entries are added without atomics, one A entry after the other, which also
// fixes the order of every sum. C's bitmap then gives each column its place:
// 32 columns a step, coalesced stores.
#include "internal.h"

namespace spg {

constexpr int kNarrowThreads = 256;
constexpr int kNarrowUnroll = 4;     // A entries whose products are in flight (2 / 4 / 8 -> 943 / 738 / 892 us)

// Bitmaps of B's rows (nw words each); a row that repeats a column sets
// ctl->narrow_dup. Four rows are in flight per warp: the row pointers of 32
// rows are read at once and the columns of four rows before they are marked.
__global__ void __launch_bounds__(kNarrowThreads) k_narrow_build(CsrDev B, int nw, unsigned* bits,
                                                                 Ctl* ctl) {
    constexpr int kRows = 4;
    __shared__ unsigned s_bm[kNarrowThreads / 32][kRows][32];
    unsigned(*bm)[32] = s_bm[threadIdx.x >> 5];
    const int lane = lane_id();
    const long long gw = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    bool dup = false;
#pragma unroll
    for (int u = 0; u < kRows; ++u) bm[u][lane] = 0u;
    __syncwarp();
    for (long long r0 = gw * 32; r0 < B.rows; r0 += nwarps * 32) {
        int s = 0, e = 0;
        if (r0 + lane < B.rows) row_extent(B, (int)(r0 + lane), s, e, ctl);
        const int rows = B.rows - r0 < 32 ? (int)(B.rows - r0) : 32;
        for (int q = 0; q < rows; q += kRows) {
            int qs[kRows], qe[kRows], c[kRows];
#pragma unroll
            for (int u = 0; u < kRows; ++u) {
                qs[u] = __shfl_sync(kFull, s, (q + u) & 31);
                qe[u] = __shfl_sync(kFull, e, (q + u) & 31);
                if (q + u >= rows) qe[u] = qs[u];
                c[u] = qs[u] + lane < qe[u] ? B.col[qs[u] + lane] : -1;
            }
#pragma unroll
            for (int u = 0; u < kRows; ++u)
                for (int t = qs[u] + lane; t < qe[u]; t += 32) {
                    const int col = t == qs[u] + lane ? c[u] : B.col[t];
                    if ((unsigned)col < (unsigned)B.cols) {
                        const unsigned bit = 1u << (col & 31);
                        dup |= (atomicOr(&bm[u][col >> 5], bit) & bit) != 0u;
                    } else {
                        set_status(ctl, ST_INVALID);
                    }
                }
            __syncwarp();
#pragma unroll
            for (int u = 0; u < kRows; ++u) {
                if (lane < nw && q + u < rows) bits[(r0 + q + u) * nw + lane] = bm[u][lane];
                bm[u][lane] = 0u;
            }
            __syncwarp();
        }
    }
    if (__any_sync(kFull, dup) && lane == 0) ctl->narrow_dup = 1;
}

// Row of C as the OR of its B rows' bitmaps. The warp takes 32 >> lg A
// entries a step, 1 << lg lanes (at least nw) per bitmap.
__global__ void __launch_bounds__(kNarrowThreads) k_sym_narrow_or(CsrDev A, int b_rows, int nw, int lg,
                                                                  const unsigned* bbits,
                                                                  unsigned* cbits, const int* map,
                                                                  Ctl* ctl, int* row_nnz, int bin) {
    const int lane = lane_id();
    const int begin = ctl->bin_off[bin], end = ctl->bin_off[bin + 1];
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int per = 32 >> lg, slot = lane >> lg, word = lane & ((1 << lg) - 1);
    int r_next = begin + gw < end ? map[begin + gw] : 0;
    for (int idx = begin + gw; idx < end; idx += nwarps) {
        const int row = r_next;
        if (idx + nwarps < end) r_next = map[idx + nwarps];
        int rs, re;
        row_extent(A, row, rs, re, ctl);
        unsigned acc = 0u;
        for (int base = rs; base < re; base += 32) {
            int k = -1;
            if (base + lane < re) {
                k = A.col[base + lane];
                if ((unsigned)k >= (unsigned)b_rows) {
                    set_status(ctl, ST_INVALID);
                    k = -1;
                }
            }
            const int n = re - base < 32 ? re - base : 32;
#pragma unroll 4
            for (int q = 0; q < n; q += per) {
                const int kq = __shfl_sync(kFull, k, q + slot);      // (q + slot <= 31)
                if (kq >= 0 && word < nw) acc |= bbits[(long long)kq * nw + word];
            }
        }
        for (int o = 1 << lg; o < 32; o <<= 1) acc |= __shfl_xor_sync(kFull, acc, o);
        const int nnz = __reduce_add_sync(kFull, lane < nw ? __popc(acc) : 0);
        if (lane < nw) cbits[(long long)row * nw + lane] = acc;
        if (lane == 0) row_nnz[row] = nnz;
    }
}

// Row of C by marking every product (A too short to pay for B's bitmaps).
__global__ void __launch_bounds__(kNarrowThreads) k_sym_narrow(CsrDev A, CsrDev B, int nw,
                                                               unsigned* cbits, const int* map,
                                                               Ctl* ctl, int* row_nnz, int bin) {
    __shared__ unsigned s_bm[kNarrowThreads / 32][32];
    unsigned* bm = s_bm[threadIdx.x >> 5];
    const int lane = lane_id();
    bm[lane] = 0u;
    __syncwarp();
    const int begin = ctl->bin_off[bin], end = ctl->bin_off[bin + 1];
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int idx = begin + gw; idx < end; idx += nwarps) {
        const int row = map[idx];
        int rs, re;
        row_extent(A, row, rs, re, ctl);
        warp_expand_ahead<kWarpAhead, false>(
            A, B, rs, re, ctl, [&](int t) { return B.col[t]; },
            [&](int c, float, unsigned) {
                if ((unsigned)c < (unsigned)B.cols) atomicOr(&bm[c >> 5], 1u << (c & 31));
                else set_status(ctl, ST_INVALID);
            });
        __syncwarp();
        const unsigned word = bm[lane];
        bm[lane] = 0u;
        const int nnz = __reduce_add_sync(kFull, __popc(word));
        if (cbits != nullptr && lane < nw) cbits[(long long)row * nw + lane] = word;
        if (lane == 0) row_nnz[row] = nnz;
        __syncwarp();
    }
}

// What bounds it: instruction issue and the shared-memory round trip of every
// A entry. 589,000 rows of 612 products over 256 columns: 2,013 us with
// atomics, a bitmap marked per product and each lane emitting its own word (8
// of 32 lanes, scattered stores), 752 us now.
// kBits: C's bitmaps are there (without them the row is marked here, in a
// kernel of its own: in one kernel that code cost the other rows 752 -> 770 us
// on 1,024 subgraphs of 256 features).
template <typename Acc, bool kBits>
__global__ void __launch_bounds__(kNarrowMaxWarps * 32) k_num_narrow(CsrDev A, CsrDev B,
                                                                     const int* map, Ctl* ctl,
                                                                     const int* rptC, int row_begin,
                                                                     int* colC, float* valC, int bin,
                                                                     int nw, const unsigned* cbits) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int warp = threadIdx.x >> 5, lane = lane_id();
    Acc* dense = reinterpret_cast<Acc*>(sm_raw) + warp * nw * 32;
    __shared__ unsigned s_bm[kBits ? 1 : kNarrowMaxWarps][32];
    unsigned* bm = s_bm[kBits ? 0 : warp];
    if (!kBits) bm[lane] = 0u;
    for (int c = lane; c < nw * 32; c += 32) dense[c] = Acc(0);
    __syncwarp();
    const int begin = ctl->bin_off[bin], end = ctl->bin_off[bin + 1];
    if (begin >= end) return;
    const bool dup = ctl->narrow_dup != 0;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    int r_next = begin + gw < end ? map[begin + gw] : 0;
    for (int idx = begin + gw; idx < end; idx += nwarps) {
        const int r = r_next;
        if (idx + nwarps < end) r_next = map[idx + nwarps];
        const int row = row_begin + r;
        const int out = rptC[r];
        const int nnz_row = rptC[r + 1] - out;
        int rs, re;
        row_extent(A, row, rs, re, ctl);
        unsigned word = 0u;
        if (kBits) {
            if (lane < nw) word = cbits[(long long)row * nw + lane];
        } else {
            warp_expand_ahead<kWarpAhead, false>(
                A, B, rs, re, ctl, [&](int t) { return B.col[t]; },
                [&](int c, float, unsigned) {
                    if ((unsigned)c < (unsigned)B.cols) atomicOr(&bm[c >> 5], 1u << (c & 31));
                });
            __syncwarp();
            word = bm[lane];
            bm[lane] = 0u;
        }
        for (int base = rs; base < re; base += 32) {
            const int j = base + lane;
            int bs = 0, len = 0;
            float a = 0.f;
            if (j < re) {
                a_entry(A, B, j, bs, len, ctl);
                a = A.val[j];
            }
            const int n = re - base < 32 ? re - base : 32;
            // an entry's products on the lanes, unless entries are so short
            // that most lanes would idle
            const int most = __reduce_max_sync(kFull, len);
            const bool entries = !dup && (most >= kLongRow || __reduce_add_sync(kFull, len) >= 12 * n);
            if (!entries) {
                warp_expand_ahead<kWarpAhead, true>(
                    A, B, base, base + n, ctl,
                    [&](int t) { return make_int2(B.col[t], __float_as_int(B.val[t])); },
                    [&](int2 cv, float av, unsigned) {
                        if ((unsigned)cv.x < (unsigned)B.cols)
                            atomicAdd(&dense[cv.x], (Acc)av * (Acc)__int_as_float(cv.y));
                    });
                __syncwarp();
                continue;
            }
            for (int q = 0; q < n; q += kNarrowUnroll) {
                int qs[kNarrowUnroll], ql[kNarrowUnroll], c[kNarrowUnroll];
                float qa[kNarrowUnroll], v[kNarrowUnroll];
#pragma unroll
                for (int u = 0; u < kNarrowUnroll; ++u) {
                    qs[u] = __shfl_sync(kFull, bs, (q + u) & 31);
                    ql[u] = __shfl_sync(kFull, len, (q + u) & 31);
                    qa[u] = __shfl_sync(kFull, a, (q + u) & 31);
                    if (q + u >= n) ql[u] = 0;
                    c[u] = -1;
                    v[u] = 0.f;
                    if (lane < ql[u]) {
                        c[u] = B.col[qs[u] + lane];
                        v[u] = B.val[qs[u] + lane];
                    }
                }
                if (most <= 32) {                            // warp-uniform: no loops
#pragma unroll
                    for (int u = 0; u < kNarrowUnroll; ++u) {
                        if ((unsigned)c[u] < (unsigned)B.cols) dense[c[u]] += (Acc)qa[u] * (Acc)v[u];
                        __syncwarp();
                    }
                    continue;
                }
#pragma unroll
                for (int u = 0; u < kNarrowUnroll; ++u) {
                    if ((unsigned)c[u] < (unsigned)B.cols) dense[c[u]] += (Acc)qa[u] * (Acc)v[u];
                    for (int t = 32 + lane; t - lane < ql[u]; t += 32) {     // warp-uniform trips
                        if (t < ql[u]) {
                            const int ct = B.col[qs[u] + t];
                            if ((unsigned)ct < (unsigned)B.cols)
                                dense[ct] += (Acc)qa[u] * (Acc)B.val[qs[u] + t];
                        }
                    }
                    __syncwarp();
                }
            }
        }
        const int cnt = __popc(word);
        const int incl = warp_incl_scan(cnt);
        const int before = incl - cnt;
        if (lane == 31 && incl != nnz_row) set_status(ctl, ST_INTERNAL);
        for (int w = 0; w < nw; ++w) {
            const unsigned bits = __shfl_sync(kFull, word, w);
            const int pos = __shfl_sync(kFull, before, w) + __popc(bits & lanemask_lt());
            if ((bits >> lane) & 1u) {
                const int c = w * 32 + lane;
                if (pos < nnz_row) {
                    colC[out + pos] = c;
                    valC[out + pos] = (float)dense[c];
                }
                dense[c] = Acc(0);
            }
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------

void occupancy_narrow(spgemm_plan* p) {
    allow_max_dynamic_smem((const void*)k_num_narrow<float, true>, p);
    allow_max_dynamic_smem((const void*)k_num_narrow<double, true>, p);
    allow_max_dynamic_smem((const void*)k_num_narrow<float, false>, p);
    allow_max_dynamic_smem((const void*)k_num_narrow<double, false>, p);
}

__global__ void k_narrow_reset(Ctl* ctl, int dup) { ctl->narrow_dup = dup; }

void launch_sym_narrow(const spgemm_plan* p, const CsrDev& A, const CsrDev& B, const WsPtrs& w,
                       int* row_nnz, cudaStream_t s) {
    const int nw = (B.cols + 31) / 32;
    const int grid = p->num_sms * 8;
    // B's bitmaps cost a pass over B and save a pass over the products: worth
    // it unless A selects few of B's rows (B rows are then read about once)
    const bool build = w.nc_bits != nullptr && A.nnz >= B.rows / 2;
    SPG_LAUNCH(p, K_SYM_NARROW, s, k_narrow_reset<<<1, 1, 0, s>>>(w.ctl, build ? 0 : 1));
    if (build) {
        SPG_LAUNCH(p, K_SYM_NARROW, s, k_narrow_build<<<grid, kNarrowThreads, 0, s>>>(B, nw, w.nb_bits, w.ctl));
        int lg = 0;
        while ((1 << lg) < nw) ++lg;
        SPG_LAUNCH(p, K_SYM_NARROW, s,
                   k_sym_narrow_or<<<grid, kNarrowThreads, 0, s>>>(A, B.rows, nw, lg, w.nb_bits, w.nc_bits,
                                                                  w.map, w.ctl, row_nnz, SB_NARROW));
    } else {
        SPG_LAUNCH(p, K_SYM_NARROW, s,
                   k_sym_narrow<<<grid, kNarrowThreads, 0, s>>>(A, B, nw, w.nc_bits, w.map, w.ctl, row_nnz,
                                                               SB_NARROW));
    }
}

void launch_num_narrow(const spgemm_plan* p, bool f64, const CsrDev& A, const CsrDev& B, const WsPtrs& w,
                       const int* rptC, int row_begin, int* colC, float* valC, cudaStream_t s) {
    const int nw = (B.cols + 31) / 32;
    const int nwp = narrow_warps(p);
    const int grid = p->num_sms * (64 / nwp > 1 ? 64 / nwp : 1);
    const size_t smem = (size_t)nwp * nw * 32 * (f64 ? 8 : 4);
    auto go = [&](auto kernel, int bin) {
        SPG_LAUNCH(p, K_NUM_NARROW, s, kernel<<<grid, nwp * 32, smem, s>>>(
            A, B, w.map, w.ctl, rptC, row_begin, colC, valC, bin, nw, w.nc_bits));
    };
    if (w.nc_bits != nullptr) {
        if (f64) go(k_num_narrow<double, true>, NB_NARROW64);
        else go(k_num_narrow<float, true>, NB_NARROW32);
    } else {
        if (f64) go(k_num_narrow<double, false>, NB_NARROW64);
        else go(k_num_narrow<float, false>, NB_NARROW32);
    }
}

}  // namespace spg
