// Bitmap tiers, allocation and accumulation phase: rows of C whose products
// outgrow the sort tier, for a B of at most kBitsCols columns.
//
// One block per row marks the row's columns in a bitmap over all of B's
// columns (one shared atomicOr per product). The allocation phase counts the
// bits. The accumulation phase turns the bitmap into ranks (a 16-bit prefix
// per 64 or 32 columns), which give every product its place in the row: rank of its
// word plus the bits below its own. So the row comes out sorted, with no
// hashing, probing, compaction or sort, and no panel table of B is needed,
// because a row is done in one pass. Shared memory per row is 5/32 or 6/32
// byte per column of B and an accumulator (and a column) per entry.
#include "internal.h"

namespace spg {

constexpr int kBitsUnroll = 2;    // products per lane in flight in a walk
constexpr int kBitsRun = 4;       // steps of a run (1 / 2 / 3 / 4 -> 1,712 / 1,310 / 1,225 / 1,211 us for the four
                                  // kernels of R-MAT 2^15 squared); none in the value walk of the sparser
                                  // rows, whose segments are shorter (1,616 -> 1,600 us, 1,075 products a row)

// One tile of A entries: non-empty segments, their offsets and multipliers.
template <int kE>
struct BitsTile {
    int off[kE + 1];
    int bs[kE];
    float a[kE];
    unsigned long long scratch[32];
};

template <int kT>
constexpr int bits_tile() { return kT < 512 ? kT : 512; }

// Exclusive block scan with one barrier (the caller's scratch of kT / 32 words
// must not be written again before another barrier).
template <int kT, typename T>
__device__ __forceinline__ T bits_scan(T v, T* scratch, T* total) {
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    constexpr int kWarps = kT / 32;
    T incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T n = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += n;
    }
    if (lane == 31) scratch[warp] = incl;
    __syncthreads();
    T w = lane < kWarps ? scratch[lane] : T(0);
#pragma unroll
    for (int o = 1; o < kWarps; o <<= 1) {
        const T n = __shfl_up_sync(kFull, w, o);
        if (lane >= o) w += n;
    }
    *total = __shfl_sync(kFull, w, kWarps - 1);
    const T before = __shfl_sync(kFull, w, warp > 0 ? warp - 1 : 0);
    return incl - v + (warp > 0 ? before : T(0));
}

// Fill the tile from A entries [j0, j1), at most kE of them; returns the
// number of segments and their products (64 bits; a tile of 2^30 or more
// products has no offsets and is walked by bits_walk one segment at a time).
// Ends with a block barrier.
template <int kT, int kE>
__device__ __forceinline__ int bits_fill(BitsTile<kE>& tile, const CsrDev& A, const CsrDev& B, int j0,
                                         int j1, bool vals, Ctl* ctl, long long& products) {
    const int j = j0 + (int)threadIdx.x;
    int bs = 0, len = 0;
    float a = 0.f;
    if ((kE == kT || threadIdx.x < kE) && j < j1) {
        a_entry(A, B, j, bs, len, ctl);
        if (vals) a = A.val[j];
    }
    const unsigned long long v = len > 0 ? ((1ull << 48) | (unsigned long long)len) : 0ull;
    unsigned long long tot;
    const unsigned long long ex = bits_scan<kT>(v, tile.scratch, &tot);
    const int n = (int)(tot >> 48);
    products = (long long)(tot & ((1ull << 48) - 1ull));
    const bool offsets = products < (1ll << 30);
    if (len > 0) {
        const int q = (int)(ex >> 48);
        tile.off[q] = offsets ? (int)(ex & ((1ull << 48) - 1ull)) : len;
        tile.bs[q] = bs;
        tile.a[q] = a;
    }
    if (threadIdx.x == 0 && offsets) tile.off[n] = (int)products;
    __syncthreads();
    return n;
}

template <int kT, int kE, int kRun = kBitsRun, class Load, class Apply>
__device__ __forceinline__ void bits_walk(const BitsTile<kE>& tile, int n, long long products,
                                          Load&& load, Apply&& apply) {
    if (products < (1ll << 30)) {
        expand_walk<int, kT / 32, float, kBitsUnroll, false, kRun>(tile.off, tile.bs, tile.a, n,
                                                             (int)products, load, apply);
        return;
    }
    for (int q = 0; q < n; ++q)
        for (long long t = threadIdx.x; t < tile.off[q]; t += kT)
            apply(load(tile.bs[q] + (int)t), tile.a[q]);
}

// Marks the row's columns in bm (clear, nw words). On return the tile holds
// the row's last tile, n segments and `products` products.
template <int kT, int kE>
__device__ __forceinline__ void bits_mark(BitsTile<kE>& tile, const CsrDev& A, const CsrDev& B, int rs,
                                          int re, bool vals, unsigned* bm, Ctl* ctl, int& n,
                                          long long& products) {
    for (int j0 = rs; j0 < re; j0 += kE) {
        n = bits_fill<kT, kE>(tile, A, B, j0, re, vals, ctl, products);
        bits_walk<kT, kE>(
            tile, n, products, [&](int t) { return B.col[t]; },
            [&](int c, float) {
                if ((unsigned)c < (unsigned)B.cols) atomicOr(&bm[c >> 5], 1u << (c & 31));
                else set_status(ctl, ST_INVALID);
            });
        __syncthreads();
    }
}

template <int kT>
__device__ __forceinline__ void bits_clear(unsigned* bm, int nw4) {
    uint4* b4 = reinterpret_cast<uint4*>(bm);
    for (int q = threadIdx.x; q < nw4; q += kT) b4[q] = make_uint4(0u, 0u, 0u, 0u);
}

template <int kT>
__global__ void __launch_bounds__(kT, 1024 / kT) k_sym_bits(CsrDev A, CsrDev B, const int* map,
                                                            Ctl* ctl, int* row_nnz, int bin_lo,
                                                            int bin_hi, int tier, int nw4) {
    constexpr int kE = bits_tile<kT>();
    extern __shared__ __align__(16) unsigned bm[];
    __shared__ BitsTile<kE> tile;
    __shared__ int s_idx;
    __shared__ int red[33];
    const int begin = ctl->bin_off[bin_lo], end = ctl->bin_off[bin_hi];
    if (begin >= end) return;
    for (;;) {
        if (threadIdx.x == 0) s_idx = begin + atomicAdd(&ctl->work[tier], 1);
        bits_clear<kT>(bm, nw4);
        __syncthreads();
        const int idx = s_idx;
        if (idx >= end) break;
        const int row = map[idx];
        int rs, re, n;
        long long products;
        row_extent(A, row, rs, re, ctl);
        bits_mark<kT, kE>(tile, A, B, rs, re, false, bm, ctl, n, products);
        const uint4* b4 = reinterpret_cast<const uint4*>(bm);
        int cnt = 0;
        for (int q = threadIdx.x; q < nw4; q += kT) {
            const uint4 w = b4[q];
            cnt += __popc(w.x) + __popc(w.y) + __popc(w.z) + __popc(w.w);
        }
        cnt = block_sum(cnt, red);                 // (ends with a barrier)
        if (threadIdx.x == 0) row_nnz[row] = cnt;
    }
}

// Words of the rank table: a rank per 64 columns halves the pass over the
// words, a rank per 32 makes the look-up of every product cheaper.
template <bool kCols>
struct BitsWord {
    using type = unsigned long long;
};
template <>
struct BitsWord<false> {
    using type = unsigned;
};
__device__ __forceinline__ int popc_of(unsigned w) { return __popc(w); }
__device__ __forceinline__ int popc_of(unsigned long long w) { return __popcll(w); }

// kCols: the value walk also leaves every product's column at its place, one
// more shared word per entry and store per product. Without it (rows of many
// entries, for which that word is dear) thread t lists the columns of its own
// words in the value array before the walk; on rows that set few bits a word
// that loop was half of the kernel (2,556 -> 1,585 us on 131,072 rows of
// 1,075 products over 131,072 columns).
template <typename Acc, int kT, bool kCols>
__global__ void __launch_bounds__(kT, 1024 / kT) k_num_bits(CsrDev A, CsrDev B, const int* map,
                                                            Ctl* ctl, const int* rptC, int row_begin,
                                                            int* colC, float* valC, int bin_lo,
                                                            int bin_hi, int tier, int nw4, int cap) {
    constexpr int kE = bits_tile<kT>();
    constexpr int kWord = sizeof(Acc) / 4;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    Acc* vals = reinterpret_cast<Acc*>(sm_raw);                 // cap accumulators
    int* stage = reinterpret_cast<int*>(sm_raw);                // !kCols: a column in each one's first word
    int* cols = reinterpret_cast<int*>(vals + cap);             // kCols: cap columns
    using Word = typename BitsWord<kCols>::type;
    constexpr int kBits = 8 * sizeof(Word);
    constexpr int kLog = kCols ? 6 : 5;
    Word* bm = reinterpret_cast<Word*>(cols + (kCols ? cap : 0));
    unsigned short* rk = reinterpret_cast<unsigned short*>(bm + 128 / kBits * nw4);   // a word's rank
    __shared__ BitsTile<kE> tile;
    __shared__ int s_idx;
    __shared__ int scratch[32];
    const int t = threadIdx.x;
    const int begin = ctl->bin_off[bin_lo], end = ctl->bin_off[bin_hi];
    if (begin >= end) return;
    // thread t owns words [w0, w1); an odd count spreads the threads' words
    // over the banks
    const int nw = 128 / kBits * nw4, wpt = ((nw + kT - 1) / kT) | 1;
    const int w0 = t * wpt < nw ? t * wpt : nw;
    const int w1 = w0 + wpt < nw ? w0 + wpt : nw;
    for (;;) {
        if (t == 0) s_idx = begin + atomicAdd(&ctl->work[tier], 1);
        bits_clear<kT>(reinterpret_cast<unsigned*>(bm), nw4);
        __syncthreads();
        const int idx = s_idx;
        if (idx >= end) break;
        const int r = map[idx];
        const int row = row_begin + r;
        const int out = rptC[r];
        const int nnz_row = rptC[r + 1] - out;
        if (kCols)
            for (int i = t; i < nnz_row && i < cap; i += kT) vals[i] = Acc(0);
        int rs, re, n = 0;
        long long products = 0;
        row_extent(A, row, rs, re, ctl);
        bits_mark<kT, kE>(tile, A, B, rs, re, true, reinterpret_cast<unsigned*>(bm), ctl, n, products);
        int cnt = 0;
        for (int w = w0; w < w1; ++w) cnt += popc_of(bm[w]);
        int tot;
        int pos = bits_scan<kT>(cnt, scratch, &tot);
        if (t == 0 && (tot != nnz_row || tot > cap)) set_status(ctl, ST_INTERNAL);
        const int nn = min(min(tot, nnz_row), cap);
        for (int w = w0; w < w1; ++w) {
            Word bits = bm[w];
            rk[w] = (unsigned short)pos;
            if (kCols) {
                pos += popc_of(bits);
            } else {
                while (bits) {
                    if (pos < cap) stage[pos * kWord] = w * kBits + __ffs((unsigned)bits) - 1;
                    bits &= bits - 1;
                    ++pos;
                }
            }
        }
        __syncthreads();
        if (!kCols) {
            for (int i = t; i < nn; i += kT) {
                colC[out + i] = stage[i * kWord];
                vals[i] = Acc(0);
            }
            __syncthreads();
        }
        auto load = [&](int q) { return make_int2(B.col[q], __float_as_int(B.val[q])); };
        auto apply = [&](int2 cv, float a) {
            const unsigned c = (unsigned)cv.x;
            if (c < (unsigned)B.cols) {
                const int rr = rk[c >> kLog] + popc_of(bm[c >> kLog] & ((Word(1) << (c & (kBits - 1))) - Word(1)));
                if (rr < nn) {
                    if (kCols) cols[rr] = (int)c;
                    atomicAdd(&vals[rr], (Acc)a * (Acc)__int_as_float(cv.y));
                }
            }
        };
        if (re - rs <= kE) {                       // the tile of the first walk is the whole row
            bits_walk<kT, kE, kCols ? 0 : kBitsRun>(tile, n, products, load, apply);
            __syncthreads();
        } else {
            for (int j0 = rs; j0 < re; j0 += kE) {
                n = bits_fill<kT, kE>(tile, A, B, j0, re, true, ctl, products);
                bits_walk<kT, kE, kCols ? 0 : kBitsRun>(tile, n, products, load, apply);
                __syncthreads();
            }
        }
        for (int i = t; i < nn; i += kT) {
            if (kCols) colC[out + i] = cols[i];
            valC[out + i] = (float)vals[i];
        }
        // (the next row writes vals and cols after a barrier)
    }
}

// ---------------------------------------------------------------------------

static int bits_nw4(const CsrDev& B) { return (B.cols + 127) / 128; }

static size_t bits_num_smem(const CsrDev& B, size_t acc, bool list, int cap) {
    return (acc + (list ? 4 : 0)) * (size_t)cap + (size_t)bits_nw4(B) * (list ? 20 : 24);
}

bool bits_tier(const CsrDev& B) {
    return B.cols <= kBitsCols && B.cols > kNarrowCols;
}

// Entries a row may have in an accumulation kernel without a column list, one
// block on an SM.
int bits_cap(const spgemm_plan* p, const CsrDev& B, size_t acc) {
    const size_t fixed = (size_t)bits_nw4(B) * 24 + kBitsStatic;
    if (p->smem_optin <= fixed) return 0;
    const size_t cap = (p->smem_optin - fixed) / acc;
    return (int)(cap < 65535 ? cap : 65535) & ~3;
}

// Smallest block that, with as many as shared memory holds, puts 768 threads
// on an SM: small blocks spend less on their barriers and scans.
static int bits_threads(size_t smem, int& blocks) {
    for (int t = 128;; t *= 2) {
        blocks = (int)(kBitsSmem / (smem + 1024 + (t < 512 ? 12 * t : 6144) + 768));
        if (blocks < 1) blocks = 1;
        if (t == 1024 || blocks * t >= 768) {
            if (blocks * t > 2048) blocks = 2048 / t;
            return t;
        }
    }
}

void launch_sym_bits(const spgemm_plan* p, const CsrDev& A, const CsrDev& B, const WsPtrs& w,
                     int* row_nnz, int bin_lo, int bin_hi, int tier, cudaStream_t s) {
    const int nw4 = bits_nw4(B);
    const size_t smem = (size_t)nw4 * 16;
    int blocks;
    const int t = bits_threads(smem, blocks);
#define SPG_BITS(kT)                                                                          \
    SPG_LAUNCH(p, K_SYM_BLOCK, s, k_sym_bits<kT><<<p->num_sms * blocks, kT, smem, s>>>(       \
                                      A, B, w.map, w.ctl, row_nnz, bin_lo, bin_hi, tier, nw4))
    if (t == 128) SPG_BITS(128);
    else if (t == 256) SPG_BITS(256);
    else if (t == 512) SPG_BITS(512);
    else SPG_BITS(1024);
#undef SPG_BITS
}

template <typename Acc, bool kCols>
static void num_bits(const spgemm_plan* p, int kid, const CsrDev& A, const CsrDev& B, const WsPtrs& w,
                     const int* rptC, int row_begin, int* colC, float* valC, int bin_lo, int bin_hi,
                     int tier, int cap, cudaStream_t s) {
    const int nw4 = bits_nw4(B);
    const size_t smem = bits_num_smem(B, sizeof(Acc), kCols, cap);
    int blocks;
    const int t = bits_threads(smem, blocks);
#define SPG_BITS(kT)                                                                              \
    SPG_LAUNCH(p, kid, s, (k_num_bits<Acc, kT, kCols><<<p->num_sms * blocks, kT, smem, s>>>(      \
                              A, B, w.map, w.ctl, rptC, row_begin, colC, valC, bin_lo, bin_hi,    \
                              tier, nw4, cap)))
    if (t == 128) SPG_BITS(128);
    else if (t == 256) SPG_BITS(256);
    else if (t == 512) SPG_BITS(512);
    else SPG_BITS(1024);
#undef SPG_BITS
}

void launch_num_bits(const spgemm_plan* p, bool f64, const CsrDev& A, const CsrDev& B, const WsPtrs& w,
                     const int* rptC, int row_begin, int* colC, float* valC, int bin_lo, int bin_hi,
                     int tier, int cap, cudaStream_t s) {
    // list columns in the walk where rows set few bits a word: up to 2 per 64
    // columns (R-MAT 2^15 squared, rows of up to 16 per 64: 467 us without the
    // list, 489 with it; 131,072 columns and rows of 0.5: 2,556 and 1,585 us)
    const bool list = cap <= 4 * bits_nw4(B) && bits_num_smem(B, f64 ? 8 : 4, true, cap) <= p->smem_optin - kBitsStatic;
    const int kid = f64 ? K_NUM_BLOCK64 : K_NUM_BLOCK32;
    auto go = [&](auto kernel) {
        kernel(p, kid, A, B, w, rptC, row_begin, colC, valC, bin_lo, bin_hi, tier, cap, s);
    };
    if (f64) list ? go(num_bits<double, true>) : go(num_bits<double, false>);
    else list ? go(num_bits<float, true>) : go(num_bits<float, false>);
}

template <int kT>
static void bits_attributes(const spgemm_plan* p) {
    allow_max_dynamic_smem((const void*)k_sym_bits<kT>, p);
    allow_max_dynamic_smem((const void*)k_num_bits<float, kT, true>, p);
    allow_max_dynamic_smem((const void*)k_num_bits<double, kT, true>, p);
    allow_max_dynamic_smem((const void*)k_num_bits<float, kT, false>, p);
    allow_max_dynamic_smem((const void*)k_num_bits<double, kT, false>, p);
}

void occupancy_bits(spgemm_plan* p) {
    bits_attributes<128>(p);
    bits_attributes<256>(p);
    bits_attributes<512>(p);
    bits_attributes<1024>(p);
}

}  // namespace spg
