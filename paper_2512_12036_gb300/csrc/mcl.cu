// Markov-clustering matrix step (Algorithm 6) on the rows of M^T: after the
// expansion E = M^T * M^T (= (M*M)^T), each row of E (a column of M) is
// pruned (entries below theta dropped), cut to its k largest entries (ties
// to the smaller column), inflated (v^r) and normalised to sum 1.
//
// Keep/drop decisions are taken in fp32 on the value (order 0: prune and
// top-k first, then inflate) or on the fp32-rounded inflated value (order 1:
// inflate first). The k-th largest decision value is found by a radix
// selection over order-preserving 32-bit keys (four 8-bit digits, a
// 256-bin histogram each), so no sort is needed; kept entries keep their
// column order. Selection runs once: it leaves a row's kept entries' count and
// threshold key, 8 bytes in the row's places of row_ptr_out and the row map,
// for the writing pass, which filters by the key, stages the kept values in
// the output and inflates and normalises only those. (With the selection run
// again before writing, and pow inlined into unrolled loops beyond the
// instruction cache, 50,021 rows of 600 entries took 3,343 us; 511 us now.)
// Weights and the row sum are fp64; each output is rounded once to fp32.
// k < 0 keeps every entry that passes the threshold (a plain normalisation
// when theta <= 0 and r = 1).
#include "internal.h"

namespace spg {

constexpr int kMclWarpMax = 1024;     // rows up to this length: one warp, 32 keys per lane
constexpr int kMclThreads = 256;
constexpr int kMclStage = 6144;       // decision keys of a longer row kept in shared memory

struct MclParams {
    float theta;
    int k;
    double r;
    int order;
};

__device__ __forceinline__ unsigned ord_key(float x) {
    const unsigned b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// (out of line: inlined into unrolled loops, pow overran the instruction cache)
__device__ __noinline__ double mcl_pow(double d, double r) { return pow(d, r); }

__device__ __forceinline__ double mcl_weight(float v, double r) {
    const double d = (double)v;
    if (r == 2.0) return d * d;
    if (r == 1.0) return d;
    return mcl_pow(d, r);
}

// (the product of two fp32 numbers is exact in fp64, so rounding it to fp32
// is the fp32 product)
__device__ __forceinline__ float mcl_decide(float v, const MclParams& p) {
    if (p.order == 0 || p.r == 1.0) return v;
    return p.r == 2.0 ? __fmul_rn(v, v) : (float)mcl_weight(v, p.r);
}

__device__ __forceinline__ unsigned mcl_key(float v, const MclParams& p) {
    const float d = mcl_decide(v, p);
    return d >= p.theta ? ord_key(d) : 0u;       // 0: pruned
}

// ---------------------------------------------------------------------------
// Selection, rows of up to kMclWarpMax entries: one warp per row. The kept
// entries are those above a key, thr[row], and as many of the first ones equal
// to it as counts[row] lacks then. Longer rows are left to k_mcl_select_long,
// listed if there is a list.
__global__ void __launch_bounds__(kMclThreads) k_mcl_select(CsrDev E, MclParams prm, int* counts,
                                                            unsigned* thr, int* longer, Ctl* ctl) {
    constexpr int kPer = kMclWarpMax / 32;
    __shared__ int whist[kMclThreads / 32][256];
    const int lane = lane_id();
    int* hist = whist[threadIdx.x >> 5];
    const long long gw = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long row = gw; row < E.rows; row += nw) {
        int s, e;
        row_extent(E, (int)row, s, e, ctl);
        const int n = e - s;
        if (n > kMclWarpMax) {
            if (longer && lane == 0) longer[atomicAdd(&ctl->work[0], 1)] = (int)row;
            continue;
        }
        unsigned key[kPer];
        int cnt = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            key[i] = 0u;
            if (32 * i < n) {                                   // warp-uniform
                const int q = s + lane + 32 * i;
                if (q < e) key[i] = mcl_key(E.val[q], prm);
                cnt += key[i] != 0u;
            }
        }
        cnt = __reduce_add_sync(kFull, cnt);
        const bool cut = prm.k >= 0 && cnt > prm.k;
        unsigned K = 0u;                                        // (0: every unpruned entry)
        if (cut) {
            // the k-th largest key by radix selection, 8 bits a pass from the
            // top, on a per-warp 256-bin histogram
            unsigned prefix = 0u, pmask = 0u;
            int above = 0;
#pragma unroll 1
            for (int sh = 24; sh >= 0; sh -= 8) {
#pragma unroll
                for (int b = 0; b < 8; ++b) hist[lane + 32 * b] = 0;
                __syncwarp();
#pragma unroll
                for (int i = 0; i < kPer; ++i)
                    if (32 * i < n && key[i] != 0u && (key[i] & pmask) == prefix)
                        atomicAdd(&hist[(key[i] >> sh) & 255u], 1);
                __syncwarp();
                int dig, run_at;
                radix_digit256(hist, above, prm.k, dig, run_at);
                prefix |= (unsigned)dig << sh;
                pmask |= 255u << sh;
                above = run_at;
                const int inside = hist[dig];
                __syncwarp();
                if (above + inside == prm.k) {                  // the whole bin is kept
                    --prefix;
                    break;
                }
            }
            K = prefix;
        }
        if (lane == 0) {
            counts[row] = cut ? prm.k : cnt;
            thr[row] = K;
        }
    }
}

// Rows of more than kMclWarpMax entries, a block each, by a counter: from the
// list that k_mcl_select has left, or, where the workspace has no room for one,
// from chunks of rows that are looked through. Chunks are small where there are
// few rows, so that the blocks end together, and of a test per thread at most,
// so that a matrix without long rows costs few steps (50,021 rows, 15% of them
// long: the step takes 547 us with the list, 585 with chunks of 8).
__device__ __forceinline__ int mcl_chunk(int rows, int blocks) {
    int c = 8;
    while (c < kMclThreads && (long long)rows > (long long)c * blocks * 8) c *= 2;
    return c;
}

// (kList: kernels of their own, since one kernel for both took registers that
// left room for a block less on an SM: 97 + 119 us instead of 90 + 92.)
template <bool kList, class Row>
__device__ __forceinline__ void mcl_long_rows(const CsrDev& E, const int* longer, int tier, Ctl* ctl,
                                              Row&& each) {
    __shared__ int s_next;
    if constexpr (kList) {
        const int n = ctl->work[0];
        for (;;) {
            if (threadIdx.x == 0) s_next = atomicAdd(&ctl->work[tier], 1);
            __syncthreads();
            if (s_next >= n) break;
            const int row = longer[s_next];
            int s, e;
            row_extent(E, row, s, e, ctl);
            each(row, s, e);                         // (with barriers)
        }
    } else {
        __shared__ int s_s[kMclThreads], s_e[kMclThreads];
        const int chunk = mcl_chunk(E.rows, gridDim.x);
        const int t = threadIdx.x;
        for (;;) {
            if (t == 0) s_next = atomicAdd(&ctl->work[tier], 1);
            __syncthreads();
            const long long r0 = (long long)s_next * chunk;
            if (r0 >= E.rows) break;
            bool any = false;
            if (t < chunk) {
                int s = 0, e = 0;
                if (r0 + t < E.rows) row_extent(E, (int)(r0 + t), s, e, ctl);
                any = e - s > kMclWarpMax;
                s_s[t] = s;
                s_e[t] = any ? e : s;
            }
            if (__syncthreads_or(any))
                for (int q = 0; q < chunk; ++q)
                    if (s_e[q] > s_s[q]) each((int)(r0 + q), s_s[q], s_e[q]);  // (block-uniform)
            __syncthreads();
        }
    }
}

// Selection of the long rows: a row's keys in shared memory (rows of up to
// kMclStage entries; longer ones compute them again each pass).
template <bool kList>
__global__ void __launch_bounds__(kMclThreads) k_mcl_select_long(CsrDev E, MclParams prm, int* counts,
                                                                 unsigned* thr, const int* longer, Ctl* ctl) {
    __shared__ int red[33];
    __shared__ int hist[256];
    __shared__ int s_dig, s_above, s_whole;
    __shared__ unsigned skey[kMclStage];
    mcl_long_rows<kList>(E, longer, 1, ctl, [&](int row, int s, int e) {
        const int n = e - s;
        const bool staged = n <= kMclStage;
        int c0 = 0;
        for (int q = threadIdx.x; q < n; q += kMclThreads) {
            const unsigned kq = mcl_key(E.val[s + q], prm);
            if (staged) skey[q] = kq;
            c0 += kq != 0u;
        }
        const int cnt = block_sum(c0, red);                     // (barrier: skey ready)
        const bool cut = prm.k >= 0 && cnt > prm.k;
        unsigned prefix = 0u, pmask = 0u;
        int above = 0;
        if (cut) {
            for (int sh = 24; sh >= 0; sh -= 8) {
                hist[threadIdx.x] = 0;
                __syncthreads();
                for (int q = threadIdx.x; q < n; q += kMclThreads) {
                    const unsigned kq = staged ? skey[q] : mcl_key(E.val[s + q], prm);
                    if (kq != 0u && (kq & pmask) == prefix) atomicAdd(&hist[(kq >> sh) & 255u], 1);
                }
                __syncthreads();
                if (threadIdx.x < 32) {
                    int dig, run_at;
                    radix_digit256(hist, above, prm.k, dig, run_at);
                    if (threadIdx.x == 0) {
                        s_dig = dig;
                        s_above = run_at;
                        s_whole = run_at + hist[dig] == prm.k;
                    }
                }
                __syncthreads();
                prefix |= (unsigned)s_dig << sh;
                pmask |= 255u << sh;
                above = s_above;
                if (s_whole) {                                  // the whole bin is kept
                    --prefix;
                    break;
                }
            }
        }
        if (threadIdx.x == 0) {
            counts[row] = cut ? prm.k : cnt;
            thr[row] = prefix;
        }
        __syncthreads();
    });
}

// ---------------------------------------------------------------------------
// Writing: a warp takes entries [q0, q1) of a row in column order, the kept
// ones going to [pos, pend) as (column, value), `eq` of those equal to the
// threshold key being already taken. Returns the position after the last.
// Four groups of 32 are loaded at a time.
__device__ __forceinline__ int mcl_write(const CsrDev& E, const MclParams& prm, unsigned K, int need,
                                         bool cut, int q0, int q1, int pos, int pend, int& eq,
                                         int* col_out, float* val_out) {
    const int lane = lane_id();
    for (int b = q0; b < q1; b += 128) {
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = b + 32 * u + lane < q1 ? E.val[b + 32 * u + lane] : 0.f;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int q = b + 32 * u + lane;
            if (b + 32 * u >= q1) break;                        // warp-uniform
            const unsigned key = q < q1 ? mcl_key(v[u], prm) : 0u;
            bool keep = key > K;
            if (cut) {
                const unsigned eqb = __ballot_sync(kFull, key == K && key != 0u);
                if (eqb) {
                    keep |= key == K && key != 0u && eq + __popc(eqb & lanemask_lt()) < need;
                    eq += __popc(eqb);
                }
            }
            const unsigned kb = __ballot_sync(kFull, keep);
            if (keep) {
                const int o = pos + __popc(kb & lanemask_lt());
                if (o < pend) {
                    col_out[o] = E.col[q];
                    val_out[o] = v[u];
                }
            }
            pos += __popc(kb);
        }
    }
    return pos;
}

// Inflate and normalise kept values in place: w / sum of w, fp64.
template <int kT>
__device__ __forceinline__ double mcl_weights(const float* val, int a, int b, int t, double r) {
    double sum = 0.0;
    for (int q = a + t; q < b; q += kT) sum += mcl_weight(val[q], r);
    return sum;
}

__global__ void __launch_bounds__(kMclThreads) k_mcl_write(CsrDev E, MclParams prm, const unsigned* thr,
                                                           const int* rpt_out, int* col_out,
                                                           float* val_out, Ctl* ctl) {
    const int lane = lane_id();
    const long long gw = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long row = gw; row < E.rows; row += nw) {
        int s, e;
        row_extent(E, (int)row, s, e, ctl);
        if (e - s > kMclWarpMax) continue;
        const unsigned K = thr[row];
        const int p0 = rpt_out[row], p1 = rpt_out[row + 1];
        int eq = 0;
        int pos = mcl_write(E, prm, K, 0, false, s, e, p0, p1, eq, col_out, val_out);
        // a cut inside a run of equal values: once more, with the first of them
        // that there is room for (the row is in L1 by now: 602 us where every
        // row has such a cut, 597 with a second number per row in the workspace)
        if (pos < p1 && prm.k >= 0 && p1 - p0 == prm.k) {
            __syncwarp();                                       // (other lanes write these places now)
            pos = mcl_write(E, prm, K, p1 - pos, true, s, e, p0, p1, eq, col_out, val_out);
        }
        if (lane == 0 && pos != p1) set_status(ctl, ST_INTERNAL);
        __syncwarp();
        const double sum = warp_sum(mcl_weights<32>(val_out, p0, p1, lane, prm.r));
        for (int q = p0 + lane; q < p1; q += 32)
            val_out[q] = sum > 0.0 ? (float)(mcl_weight(val_out[q], prm.r) / sum) : 0.f;
    }
}

// A long row per block, a contiguous share of it per warp: every warp counts
// the entries above and at the threshold in its share first.
template <bool kList>
__global__ void __launch_bounds__(kMclThreads) k_mcl_write_long(CsrDev E, MclParams prm, const unsigned* thr,
                                                                const int* longer, const int* rpt_out,
                                                                int* col_out, float* val_out, Ctl* ctl) {
    constexpr int kWarps = kMclThreads / 32;
    __shared__ int s_gt[kWarps], s_eq[kWarps];
    __shared__ double redd[33];
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    mcl_long_rows<kList>(E, longer, 2, ctl, [&](int row, int s, int e) {
        const unsigned K = thr[row];
        const int p0 = rpt_out[row], p1 = rpt_out[row + 1];
        const bool cut = prm.k >= 0 && p1 - p0 == prm.k;
        const int per = ((e - s + kWarps - 1) / kWarps + 31) & ~31;
        const int q0 = s + warp * per < e ? s + warp * per : e;
        const int q1 = q0 + per < e ? q0 + per : e;
        int gt = 0, at = 0;
        for (int q = q0 + lane; q < q1; q += 32) {
            const unsigned key = mcl_key(E.val[q], prm);
            gt += key > K;
            at += key == K && key != 0u;
        }
        gt = __reduce_add_sync(kFull, gt);
        at = __reduce_add_sync(kFull, at);
        if (lane == 0) {
            s_gt[warp] = gt;
            s_eq[warp] = at;
        }
        __syncthreads();
        int pos = p0, eq = 0, need = p1 - p0;
        for (int w = 0; w < kWarps; ++w) {
            need -= s_gt[w];
            if (w < warp) {
                pos += s_gt[w];
                eq += s_eq[w];
            }
        }
        if (cut) pos += eq < need ? eq : need;
        pos = mcl_write(E, prm, K, need, cut, q0, q1, pos, p1, eq, col_out, val_out);
        if (warp == kWarps - 1 && lane == 0 && pos != p1) set_status(ctl, ST_INTERNAL);
        __syncthreads();
        const double sum = block_sum(mcl_weights<kMclThreads>(val_out, p0, p1, threadIdx.x, prm.r), redd);
        for (int q = p0 + (int)threadIdx.x; q < p1; q += kMclThreads)
            val_out[q] = sum > 0.0 ? (float)(mcl_weight(val_out[q], prm.r) / sum) : 0.f;
        // (s_gt is written again after the barriers of block_sum, the last of
        // which follows every read of the row's number)
    });
}

void launch_mcl_step(const spgemm_plan* p, const CsrDev& E, float theta, int k, double r,
                     int order, const WsPtrs& w, int* rpt_out, int* col_out, float* val_out,
                     cudaStream_t s) {
    if (E.rows == 0) {
        launch_row_ptr(p, w.map, 0, w, rpt_out, s);
        return;
    }
    const MclParams prm{theta, k, r, order};
    const int grid = p->num_sms * 8, grid_long = p->num_sms * 6;
    // the scan takes the counts in place: a thread reads its rows' counts
    // before it writes their row pointers, and no other thread reads them then
    int* counts = rpt_out;
    unsigned* thr = (unsigned*)w.map;
    int* longer = w.row_list;
    cudaMemsetAsync(w.ctl->work, 0, sizeof(w.ctl->work), s);
    auto go = [&](auto select_long, auto write_long) {
        SPG_LAUNCH(p, K_MCL, s, k_mcl_select<<<grid, kMclThreads, 0, s>>>(E, prm, counts, thr, longer, w.ctl));
        SPG_LAUNCH(p, K_MCL, s, select_long<<<grid_long, kMclThreads, 0, s>>>(E, prm, counts, thr, longer, w.ctl));
        launch_row_ptr(p, counts, E.rows, w, rpt_out, s);
        SPG_LAUNCH(p, K_MCL, s, k_mcl_write<<<grid, kMclThreads, 0, s>>>(E, prm, thr, rpt_out, col_out, val_out, w.ctl));
        SPG_LAUNCH(p, K_MCL, s, write_long<<<grid_long, kMclThreads, 0, s>>>(E, prm, thr, longer, rpt_out, col_out, val_out, w.ctl));
    };
    if (longer) go(k_mcl_select_long<true>, k_mcl_write_long<true>);
    else go(k_mcl_select_long<false>, k_mcl_write_long<false>);
}

}  // namespace spg
