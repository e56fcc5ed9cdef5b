// Scans of other interaction orders: Eq. 1 applied to two, four, five and six SNPs.
//
// Pairs: every pair i < j gets the 3^2-cell x {control, case} table and its FP64 K2; the k
// lowest are returned in the total order (K2 ascending, then i, j).  The counts are exact
// integers straight from the pair tables and marginals built for the 8-cell triplet forms:
// for class c, cells (a, b) with a, b in {0, 1} are the pair table,
//   (a, 2) = n_i(a) - n_ab0 - n_ab1 over b,  (2, b) = n_j(b) - sum over a,
//   (2, 2) = N_c - the other eight.
// The score is summed in cell order 0..8 (cell = 3 gX + gY), term (lf[r+1] - lf[r0]) - lf[r1],
// from the same FP64 log-factorial table as the triplet rescoring, so it equals the oracle's
// bit for bit.  The thresholded form (launch_pair_filter) bounds every pair from below without a
// table and scores only those in FP64 whose bound does not exceed the threshold: 4096 SNPs x 4096
// samples, k = 64, 1852 -> 292 us (pair tables read once, 268 MB).  The direct form scores every pair
// and sorts every 2048 of them that reach the threshold; it answers where more pairs tie at the k-th
// score than the list of candidates holds (2500 of the 4096 SNPs without a variant: 1896 -> 1421 us;
// all of them, where there is nothing to leave out: 1909 -> 2039 us).
//
// Four SNPs, the direct form: every set i < j < k < l gets its 3^4 = 81-cell table by AND + POPC over the bit
// planes (plane 2 by NOR, pad bits land in cell 80 and are subtracted), built as a product
// tree (3 + 9 + 27 + 81 ANDs per word), both classes' counts packed in one register per cell;
// the FP64 K2 is summed in cell order 0..80 (cell = 27 g_i + 9 g_j + 3 g_k + g_l) like the
// pairs.  The sets are enumerated in colexicographic order from a linear index.
//
// Orders four to six, the counted form (launch_set_scan): every set is first scored in FP32 from its
// exact table, and only the sets within that score's error of the k-th best are counted again and
// scored in FP64.  A thread counts the 2^K cells with genotypes 0 and 1 of its set (AND + POPC) and
// gets the other 3^K - 2^K from the same counts of all smaller sets, by
//     #(.., 2, ..) = #(.., any, ..) - #(.., 0, ..) - #(.., 1, ..),
// both classes in one register and one three-input subtraction per cell: 4 SNPs of 120 with 2000
// samples 13.9 -> 2.41 ms, 5 of 48 with 1500 59.2 -> 1.37 ms.  The direct forms
// (81, 243 or 729 cells counted, every set scored in FP64) serve what the counted form refuses: a few
// sets, tables of the smaller sets past kSubsetBytes, or, with five and six SNPs, more sets tied at the k-th
// score than the list of candidates holds; with four, every set is then counted the same way and
// scored in FP64 (launch_quad_tied).
//
// Selection (pairs and the direct forms): each block scores 2048 consecutive items and keeps its k best (bitonic
// sort in shared memory); further passes merge 2048 survivors per block until one block
// remains.  Ties are ordered by a key that sorts like the SNP indices.
#include <cmath>

#include "epi3_internal.cuh"

namespace epi3 {

namespace {

constexpr int kPairBlock = 2048;      // items sorted per block
constexpr int kPairThreads = 512;     // 4 items per thread
constexpr int kQuadThreads = 256;     // 8 sets per thread (81 packed counters each: registers)

struct Item {
    double s;
    long long key;                    // i * M + j: the tie order (i, j)
};

__device__ __forceinline__ bool item_before(const Item& a, const Item& b) {
    return a.s < b.s || (a.s == b.s && a.key < b.key);
}

// Ascending bitonic sort of n items (a power of two) in shared memory (all threads of the block).
__device__ void sort_items(Item* it, int n = kPairBlock) {
    for (int size = 2; size <= n; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = threadIdx.x; t < n / 2; t += blockDim.x) {
                const int lo = 2 * t - (t & (stride - 1)), hi = lo + stride;
                const bool up = (lo & size) == 0;
                const Item x = it[lo], y = it[hi];
                if (item_before(y, x) == up) {
                    it[lo] = y;
                    it[hi] = x;
                }
            }
            __syncthreads();
        }
}

// -1 / x by the hardware reciprocal (within 1 ulp)
__device__ __forceinline__ float pair_nrcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(-x));
    return y;
}

__device__ __forceinline__ Item pad_item() {
    return Item{__longlong_as_double(0x7ff0000000000000LL), 0x7fffffffffffffffLL};  // +inf, last
}

// Cells r[c][3 gX + gY] of pair p = (i, j); false if a corrupt table makes one negative.
__device__ __forceinline__ bool pair_cells(const PairTables& pt, int M, long long p, int i, int j, int (&r)[2][9]) {
    int neg = 0;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int4 q = __ldg(pt.pt + c * pt.n_pairs + p);        // {n00, n01, n10, n11}
        const int2 mi = __ldg(pt.marg + (size_t)c * M + i), mj = __ldg(pt.marg + (size_t)c * M + j);
        r[c][0] = q.x;
        r[c][1] = q.y;
        r[c][2] = mi.x - q.x - q.y;     // (0, 2)
        r[c][3] = q.z;
        r[c][4] = q.w;
        r[c][5] = mi.y - q.z - q.w;     // (1, 2)
        r[c][6] = mj.x - q.x - q.z;     // (2, 0)
        r[c][7] = mj.y - q.y - q.w;     // (2, 1)
        r[c][8] = pt.n_c[c] - mi.x - mi.y - r[c][6] - r[c][7];   // (2, 2)
#pragma unroll
        for (int cell = 0; cell < 9; ++cell) neg |= r[c][cell];
    }
    return neg >= 0;
}
// FP64 K2 of a pair in cell order.
__device__ __forceinline__ double pair_score(const int (&r)[2][9], const double* __restrict__ lf64) {
    double s = 0.0;
#pragma unroll
    for (int cell = 0; cell < 9; ++cell) {
        const int r0 = r[0][cell], r1 = r[1][cell];
        s = __dadd_rn(s, __dsub_rn(__dsub_rn(lf64[r0 + r1 + 1], lf64[r0]), lf64[r1]));
    }
    return s;
}

// Pass 1 of the direct form: score pairs [b * 2048, (b + 1) * 2048), keep the block's k best of those
// at or below thr in out[b * k ..] (a block without any sorts nothing).
__global__ void __launch_bounds__(kPairThreads)
pair_score_kernel(PairTables pt, const double* __restrict__ lf64, int M, long long n_pairs,
                  float thr, int k, Item* __restrict__ out) {
    __shared__ Item it[kPairBlock];
    const long long p0 = (long long)blockIdx.x * kPairBlock;
    bool any = false;
    for (int t = threadIdx.x; t < kPairBlock; t += kPairThreads) {
        const long long p = p0 + t;
        it[t] = pad_item();
        if (p >= n_pairs) continue;
        int i, j, r[2][9];
        decode_pair(p, &i, &j);
        // exact counts cannot be negative; a corrupt table is ranked last, never looked up
        if (!pair_cells(pt, M, p, i, j, r)) continue;
        const double s = pair_score(r, lf64);
        if (!(s <= (double)thr)) continue;
        it[t] = Item{s, (long long)i * M + j};
        any = true;
    }
    if (__syncthreads_or(any)) sort_items(it);
    for (int t = threadIdx.x; t < k; t += kPairThreads) out[(long long)blockIdx.x * k + t] = it[t];
}

// Merge pass: the k best of each 2048 consecutive survivors.
__global__ void __launch_bounds__(kPairThreads)
pair_merge_kernel(const Item* __restrict__ in, long long n, int k, Item* __restrict__ out) {
    __shared__ Item it[kPairBlock];
    const long long b0 = (long long)blockIdx.x * kPairBlock;
    for (int t = threadIdx.x; t < kPairBlock; t += kPairThreads)
        it[t] = b0 + t < n ? in[b0 + t] : pad_item();
    __syncthreads();
    sort_items(it);
    for (int t = threadIdx.x; t < k; t += kPairThreads) out[(long long)blockIdx.x * k + t] = it[t];
}

// The k best of n items, k from each 2048, in passes over the buffers a and b until one block is left;
// *best: where they are.  Items in `in` (which may be a).
cudaError_t merge_items(const Item* in, long long n, int k, Item* a, Item* b, const Item** best, int* launches,
                        cudaStream_t st) {
    while (n > k) {
        const long long blocks = (n + kPairBlock - 1) / kPairBlock;
        Item* const out = in == a ? b : a;
        pair_merge_kernel<<<(unsigned)blocks, kPairThreads, 0, st>>>(in, n, k, out);
        ++*launches;
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        in = out;
        n = blocks * k;
    }
    *best = in;
    return cudaSuccess;
}

// Control block of the thresholded forms.
struct SetCtrl {
    float thr, last;             // threshold, and the one before
    unsigned n_cand, n_final;    // candidates met (the list holds the first `cap`), rescored ones
    unsigned tied;               // the sample says that more tie at the threshold than the list holds
};
// The answer is in fin[0 .. n_final), to be sorted by one block.
__device__ __forceinline__ bool in_one_block(const SetCtrl* ctrl, unsigned cap) {
    return ctrl->n_cand <= cap && ctrl->n_final <= (unsigned)kPairBlock;
}

// (ctrl: null, or nothing is written unless its answer is in one block)
__global__ void pair_emit_kernel(const Item* __restrict__ best, int k, int M, const SetCtrl* ctrl, unsigned cap,
                                 int32_t* __restrict__ out_pairs, double* __restrict__ out_s) {
    if (ctrl && !in_one_block(ctrl, cap)) return;
    for (int t = threadIdx.x; t < k; t += blockDim.x) {
        const Item e = best[t];
        out_pairs[2 * t] = (int32_t)(e.key / M);
        out_pairs[2 * t + 1] = (int32_t)(e.key % M);
        out_s[t] = e.s;
    }
}

// ---------------------------------------------------------------- four SNPs
__host__ __device__ inline long long choose_ll(long long n, int r) {
    if (n < r) return 0;
    long long v = 1;
    for (int t = 0; t < r; ++t) v = v * (n - t) / (t + 1);
    return v;
}

// Largest x in [lo, hi) with choose(x, r) <= q (choose is increasing in x for x >= r - 1).
__device__ inline int colex_digit(long long q, int r, int lo, int hi) {
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (choose_ll(mid, r) <= q) lo = mid;
        else hi = mid;
    }
    return lo;
}

// The q-th 4-set in colexicographic order: q = C(l,4) + C(k,3) + C(j,2) + i, i < j < k < l.
__device__ inline void decode_quad(long long q, int M, int* x) {
    const int l = colex_digit(q, 4, 3, M);
    q -= choose_ll(l, 4);
    const int k = colex_digit(q, 3, 2, l);
    q -= choose_ll(k, 3);
    const int j = colex_digit(q, 2, 1, k);
    q -= choose_ll(j, 2);
    x[0] = (int)q;
    x[1] = j;
    x[2] = k;
    x[3] = l;
}

__device__ __forceinline__ long long quad_key(const int* x) {
    return ((long long)x[0] << 48) | ((long long)x[1] << 32) | ((long long)x[2] << 16) | x[3];
}

// Pass 1 of the four-SNP scan: score sets [b * 2048, (b + 1) * 2048), keep the k best.
__global__ void __launch_bounds__(kQuadThreads)
quad_score_kernel(Planes pl, const double* __restrict__ lf64, int n0, int n1, long long n_sets,
                  int k, Item* __restrict__ out) {
    __shared__ Item it[kPairBlock];
    const long long q0 = (long long)blockIdx.x * kPairBlock;
    const int M = pl.M;
    for (int t = threadIdx.x; t < kPairBlock; t += kQuadThreads) {
        const long long q = q0 + t;
        if (q >= n_sets) {
            it[t] = pad_item();
            continue;
        }
        int x[4];
        decode_quad(q, M, x);
        // cnt[cell] = count of class 0 + (count of class 1 << 16)
        uint32_t cnt[81];
#pragma unroll
        for (int cell = 0; cell < 81; ++cell) cnt[cell] = 0u;
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            const long long coff = c ? pl.coff[1] : pl.coff[0];
            const int W4 = c ? pl.W4[1] : pl.W4[0];
            const int sh = 16 * c;
#pragma unroll 1
            for (int w4 = 0; w4 < W4; ++w4) {
                uint4 g0[4], g1[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    g0[v] = __ldg(pl.planes + coff + (size_t)w4 * M + x[v]);
                    g1[v] = __ldg(pl.planes + coff + (size_t)(W4 + w4) * M + x[v]);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    uint32_t P[4][3];
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const uint32_t a0 = e == 0 ? g0[v].x : e == 1 ? g0[v].y : e == 2 ? g0[v].z : g0[v].w;
                        const uint32_t a1 = e == 0 ? g1[v].x : e == 1 ? g1[v].y : e == 2 ? g1[v].z : g1[v].w;
                        P[v][0] = a0;
                        P[v][1] = a1;
                        P[v][2] = ~(a0 | a1);        // genotype 2, Sec. IV-A (pad bits read 2)
                    }
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int b = 0; b < 3; ++b) {
                            const uint32_t ab = P[0][a] & P[1][b];
#pragma unroll
                            for (int cc = 0; cc < 3; ++cc) {
                                const uint32_t abc = ab & P[2][cc];
#pragma unroll
                                for (int d = 0; d < 3; ++d)
                                    cnt[27 * a + 9 * b + 3 * cc + d] +=
                                        (uint32_t)__popc(abc & P[3][d]) << sh;
                            }
                        }
                }
            }
        }
        // pad samples read genotype 2 in all four SNPs: cell (2, 2, 2, 2) only
        cnt[80] -= (uint32_t)pl.pad[0] + ((uint32_t)pl.pad[1] << 16);
        double s = 0.0;
#pragma unroll
        for (int cell = 0; cell < 81; ++cell) {
            const int r0 = (int)(cnt[cell] & 0xFFFFu), r1 = (int)(cnt[cell] >> 16);
            const double term = __dsub_rn(__dsub_rn(lf64[r0 + r1 + 1], lf64[r0]), lf64[r1]);
            s = __dadd_rn(s, term);
        }
        (void)n0;
        (void)n1;
        it[t] = Item{s, quad_key(x)};
    }
    __syncthreads();
    sort_items(it);
    for (int t = threadIdx.x; t < k; t += kQuadThreads) out[(long long)blockIdx.x * k + t] = it[t];
}

__global__ void quad_emit_kernel(const Item* __restrict__ best, int k, int32_t* __restrict__ out_snps,
                                 double* __restrict__ out_s) {
    for (int t = threadIdx.x; t < k; t += blockDim.x) {
        const Item e = best[t];
        out_snps[4 * t] = (int32_t)((e.key >> 48) & 0xFFFF);
        out_snps[4 * t + 1] = (int32_t)((e.key >> 32) & 0xFFFF);
        out_snps[4 * t + 2] = (int32_t)((e.key >> 16) & 0xFFFF);
        out_snps[4 * t + 3] = (int32_t)(e.key & 0xFFFF);
        out_s[t] = e.s;
    }
}

// ---------------------------------------------------------------- five and six SNPs
// The same table and score for order K = 5, 6 (3^K = 243, 729 cells), one warp per set: lane l
// owns cells l, l + 32, ..., each cell's genotype digits kept as 2-bit codes (x_0 most
// significant, as in the cell index); per 32-sample word every lane ANDs the K plane words its
// cells select and adds the POPC (both classes packed in one counter, class 1 in the high
// half).  The FP64 K2 is then summed in cell order 0 .. 3^K - 1 by every lane from the lanes'
// terms (warp shuffles in cell order), as the oracle adds them.  Sets are enumerated in
// lexicographic order, so the rank q itself is the tie key.
constexpr int kOrdThreads = 256;      // 8 warps per block, 256 sets each

template <int K>
struct Pow3 {
    static constexpr int v = 3 * Pow3<K - 1>::v;
};
template <>
struct Pow3<0> {
    static constexpr int v = 1;
};

// The q-th K-set x_0 < ... < x_{K-1} of M SNPs in lexicographic order.
template <int K>
__device__ inline void decode_lex(long long q, int M, int* x) {
    int v = 0;
#pragma unroll
    for (int t = 0; t < K; ++t)
        for (;; ++v) {
            const long long c = choose_ll(M - 1 - v, K - 1 - t);   // sets with x_t = v
            if (q < c) {
                x[t] = v++;
                break;
            }
            q -= c;
        }
}

// Genotype codes of the cells a lane owns (2 bits per SNP: the genotype of x_t at bits 2 t).
template <int K>
__device__ __forceinline__ void lane_codes(uint32_t* code) {
    constexpr int kCellsK = Pow3<K>::v, kPer = (kCellsK + 31) / 32;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int m = 0; m < kPer; ++m) {
        int e = lane + 32 * m < kCellsK ? lane + 32 * m : 0;
        uint32_t cd = 0u;
#pragma unroll
        for (int t = K - 1; t >= 0; --t) {
            cd |= (uint32_t)(e % 3) << (2 * t);
            e /= 3;
        }
        code[m] = cd;
    }
}

// FP64 K2 of one set by one warp (every lane returns it).
template <int K>
__device__ double set_score(const Planes& pl, const double* __restrict__ lf64, const int* x,
                            const uint32_t* code) {
    constexpr int kCellsK = Pow3<K>::v, kPer = (kCellsK + 31) / 32;
    const int lane = threadIdx.x & 31;
    const int M = pl.M;
    uint32_t cnt[kPer];
#pragma unroll
    for (int m = 0; m < kPer; ++m) cnt[m] = 0u;
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
        const long long coff = c ? pl.coff[1] : pl.coff[0];
        const int W4 = c ? pl.W4[1] : pl.W4[0];
        const int sh = 16 * c;
#pragma unroll 1
        for (int w4 = 0; w4 < W4; ++w4) {
            uint4 g0[K], g1[K];
#pragma unroll
            for (int v = 0; v < K; ++v) {
                g0[v] = __ldg(pl.planes + coff + (size_t)w4 * M + x[v]);
                g1[v] = __ldg(pl.planes + coff + (size_t)(W4 + w4) * M + x[v]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                uint32_t P[K][3];
#pragma unroll
                for (int v = 0; v < K; ++v) {
                    const uint32_t a0 = e == 0 ? g0[v].x : e == 1 ? g0[v].y : e == 2 ? g0[v].z : g0[v].w;
                    const uint32_t a1 = e == 0 ? g1[v].x : e == 1 ? g1[v].y : e == 2 ? g1[v].z : g1[v].w;
                    P[v][0] = a0;
                    P[v][1] = a1;
                    P[v][2] = ~(a0 | a1);        // genotype 2, Sec. IV-A (pad bits read 2)
                }
#pragma unroll
                for (int m = 0; m < kPer; ++m) {
                    uint32_t acc = 0xFFFFFFFFu;
#pragma unroll
                    for (int v = 0; v < K; ++v) {
                        const uint32_t g = (code[m] >> (2 * v)) & 3u;
                        acc &= g == 0u ? P[v][0] : (g == 1u ? P[v][1] : P[v][2]);
                    }
                    cnt[m] += (uint32_t)__popc(acc) << sh;
                }
            }
        }
    }
    // pad samples read genotype 2 in every SNP: the last cell only
    if (lane == (kCellsK - 1) % 32)
        cnt[(kCellsK - 1) / 32] -= (uint32_t)pl.pad[0] + ((uint32_t)pl.pad[1] << 16);
    double term[kPer];
#pragma unroll
    for (int m = 0; m < kPer; ++m) {
        const int r0 = (int)(cnt[m] & 0xFFFFu), r1 = (int)(cnt[m] >> 16);
        term[m] = lane + 32 * m < kCellsK
                      ? __dsub_rn(__dsub_rn(lf64[r0 + r1 + 1], lf64[r0]), lf64[r1]) : 0.0;
    }
    double sc = 0.0;
#pragma unroll
    for (int m = 0; m < kPer; ++m)
#pragma unroll
        for (int l = 0; l < 32; ++l)
            if (32 * m + l < kCellsK) sc = __dadd_rn(sc, __shfl_sync(0xffffffffu, term[m], l));
    return sc;
}

template <int K>
__global__ void __launch_bounds__(kOrdThreads)
order_score_kernel(Planes pl, const double* __restrict__ lf64, long long n_sets, int k,
                   Item* __restrict__ out) {
    __shared__ Item it[kPairBlock];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t code[(Pow3<K>::v + 31) / 32];
    lane_codes<K>(code);
    const long long q0 = (long long)blockIdx.x * kPairBlock;
    for (int t = warp; t < kPairBlock; t += kOrdThreads / 32) {
        const long long q = q0 + t;
        if (q >= n_sets) {   // uniform over the warp
            if (lane == 0) it[t] = pad_item();
            continue;
        }
        int x[K];
        decode_lex<K>(q, pl.M, x);
        const double sc = set_score<K>(pl, lf64, x, code);
        if (lane == 0) it[t] = Item{sc, q};
    }
    __syncthreads();
    sort_items(it);
    for (int t = threadIdx.x; t < k; t += kOrdThreads) out[(long long)blockIdx.x * k + t] = it[t];
}

template <int K>
__global__ void order_emit_kernel(const Item* __restrict__ best, int k, int M, const SetCtrl* ctrl, unsigned cap,
                                  int32_t* __restrict__ out_snps, double* __restrict__ out_s) {
    if (ctrl && !in_one_block(ctrl, cap)) return;
    const long long n_sets = choose_ll(M, K);
    for (int t = threadIdx.x; t < k; t += blockDim.x) {
        const Item e = best[t];
        if ((unsigned long long)e.key >= (unsigned long long)n_sets) continue;   // no rank: nothing to decode
        int x[K];
        decode_lex<K>(e.key, M, x);
#pragma unroll
        for (int v = 0; v < K; ++v) out_snps[K * t + v] = (int32_t)x[v];
        out_s[t] = e.s;
    }
}

template <int K>
cudaError_t order_scan_k(const Planes& pl, const double* lf64, int k, void* scratch,
                         int32_t* out_snps, double* out_s, int* launches, cudaStream_t st) {
    const long long n_sets = choose_ll(pl.M, K);
    const long long blocks = (n_sets + kPairBlock - 1) / kPairBlock;
    Item* const a = static_cast<Item*>(scratch);
    order_score_kernel<K><<<(unsigned)blocks, kOrdThreads, 0, st>>>(pl, lf64, n_sets, k, a);
    cudaError_t e = cudaGetLastError();
    const Item* best = nullptr;
    if (e == cudaSuccess) e = merge_items(a, blocks * k, k, a, a + blocks * k, &best, launches, st);
    if (e != cudaSuccess) return e;
    order_emit_kernel<K><<<1, 512, 0, st>>>(best, k, pl.M, nullptr, 0u, out_snps, out_s);
    *launches += 2;
    return cudaGetLastError();
}


// ---------------------------------------------------------------- four to six SNPs, counted form
// Sets are numbered in colexicographic order here: {y_1 < ... < y_t} has rank sum of C(y_s, s).  The
// counts of every set of t = 1 .. K - 1 SNPs lie at sub[t] + 2^t rank + (genotypes as bits, the
// smallest SNP's the highest): class 0's count in the low half, class 1's in the high half.
struct SetArgs {
    Planes pl;
    const long long* binom;      // [7][M + 1]: C(x, t)
    const float* lf;             // [N + 2]
    int n_lf;
    uint32_t* sub[6];            // by set size
    uint32_t total;              // class sizes, packed
    long long n_sets;
};
struct SetCand {
    long long q;                 // rank
    float s;
};

__device__ __forceinline__ long long binom_at(const SetArgs& a, int x, int t) {
    return __ldg(a.binom + (size_t)t * (a.pl.M + 1) + x);
}
// The set of rank q, ascending.
template <int T>
__device__ __forceinline__ void decode_colex(const SetArgs& a, long long q, int* x) {
    int hi = a.pl.M;
#pragma unroll
    for (int t = T; t >= 1; --t) {
        int lo = t - 1;          // C(t - 1, t) = 0
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (binom_at(a, mid, t) <= q) lo = mid;
            else hi = mid;
        }
        q -= binom_at(a, lo, t);
        x[t - 1] = lo;
        hi = lo;
    }
}

// Its rank in lexicographic order, the tie key.
template <int K>
__device__ __forceinline__ long long lex_rank(const SetArgs& a, const int* x) {
    long long lex = a.n_sets - 1;
#pragma unroll
    for (int t = 0; t < K; ++t) lex -= binom_at(a, a.pl.M - 1 - x[t], K - t);
    return lex;
}

__global__ void set_tables_kernel(int M, const double* __restrict__ lf64, int n_lf,
                                  long long* __restrict__ binom, float* __restrict__ lf) {
    const int n = blockDim.x * gridDim.x, id = blockIdx.x * blockDim.x + threadIdx.x;
    for (int e = id; e < 7 * (M + 1); e += n) binom[e] = choose_ll(e % (M + 1), e / (M + 1));
    for (int e = id; e < n_lf; e += n) lf[e] = (float)lf64[e];
}

// Counts of the cells of x with genotypes 0 and 1, packed; cnt[bits], x[0] the highest bit.
template <int T>
__device__ __forceinline__ void count_cells(const Planes& pl, const int* x, uint32_t* cnt) {
    const int M = pl.M;
#pragma unroll
    for (int e = 0; e < (1 << T); ++e) cnt[e] = 0u;
#pragma unroll 1
    for (int c = 1; c >= 0; --c) {
        const uint4* const base = pl.planes + (c ? pl.coff[1] : pl.coff[0]);
        const int W4 = c ? pl.W4[1] : pl.W4[0];
#pragma unroll 1
        for (int w4 = 0; w4 < W4; ++w4) {
            uint4 g[T][2];
#pragma unroll
            for (int v = 0; v < T; ++v) {
                g[v][0] = __ldg(base + (size_t)w4 * M + x[v]);
                g[v][1] = __ldg(base + (size_t)(W4 + w4) * M + x[v]);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                uint32_t p[1 << T];
                p[0] = 0xFFFFFFFFu;
#pragma unroll
                for (int v = 0; v < T; ++v) {
                    const uint32_t a0 = e == 0 ? g[v][0].x : e == 1 ? g[v][0].y : e == 2 ? g[v][0].z : g[v][0].w;
                    const uint32_t a1 = e == 0 ? g[v][1].x : e == 1 ? g[v][1].y : e == 2 ? g[v][1].z : g[v][1].w;
#pragma unroll
                    for (int b = (1 << v) - 1; b >= 0; --b) {
                        p[2 * b + 1] = p[b] & a1;
                        p[2 * b] = p[b] & a0;
                    }
                }
#pragma unroll
                for (int b = 0; b < (1 << T); ++b) cnt[b] += (uint32_t)__popc(p[b]);
            }
        }
        if (c == 1)
#pragma unroll
            for (int e = 0; e < (1 << T); ++e) cnt[e] <<= 16;
    }
}

template <int T>
__global__ void __launch_bounds__(128) set_count_kernel(const SetArgs a, long long n_sets) {
    for (long long q = (long long)blockIdx.x * 128 + threadIdx.x; q < n_sets; q += (long long)gridDim.x * 128) {
        int x[T];
        decode_colex<T>(a, q, x);
        uint32_t cnt[1 << T];
        count_cells<T>(a.pl, x, cnt);
        uint32_t* const o = a.sub[T] + (q << T);
#pragma unroll
        for (int e = 0; e < (1 << T); ++e) o[e] = cnt[e];
    }
}

// #(positions of the set in `mask` have the genotypes of `bits`, the others any), packed, for the 2^n
// lowest of those positions' bits (out): the table of that subset, or this set's own counts.
// Bit K - 1 - p of mask and bits stands for position p.
template <int K, int NLOW>
__device__ __forceinline__ void subset_counts(const SetArgs& a, const int* x, const uint32_t* own,
                                              int mask, int bits, uint32_t* out) {
    // mask, bits and NLOW are compile-time constants after unrolling
    if (mask == (1 << K) - 1) {
#pragma unroll
        for (int e = 0; e < (1 << NLOW); ++e) out[e] = own[bits + e];
        return;
    }
    if (mask == 0) {
        out[0] = a.total;
        return;
    }
    long long rank = 0;
    int t = 0, idx = 0;
#pragma unroll
    for (int p = 0; p < K; ++p)
        if (mask & (1 << (K - 1 - p))) {
            ++t;
            rank += binom_at(a, x[p], t);
            idx = 2 * idx + ((bits >> (K - 1 - p)) & 1);
        }
    const uint32_t* const src = a.sub[t] + (rank << t) + idx;
    if (NLOW == 0) out[0] = __ldg(src);
    if (NLOW == 1) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(src));
        out[0] = v.x;
        out[1] = v.y;
    }
    if (NLOW >= 2) {
#pragma unroll
        for (int e = 0; e < (1 << NLOW); e += 4) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(src + e));
            out[e] = v.x;
            out[e + 1] = v.y;
            out[e + 2] = v.z;
            out[e + 3] = v.w;
        }
    }
}

// The 27 cells over the last three positions (index 9 g + 3 h + i) with the positions before them as
// mask / bits say, positions in mask2 with genotype 2 (each #any - #0 - #1).
template <int K>
__device__ __forceinline__ void inner_cells(const SetArgs& a, const int* x, const uint32_t* own,
                                            int mask, int bits, uint32_t* g) {
    // {0, 1, any}^3 first: any at digit 2
    uint32_t v[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) {   // which of the last three positions are fixed
        constexpr int kStep[3] = {9, 3, 1};
        const int n = (m & 1) + ((m >> 1) & 1) + (m >> 2);
        if (n == 0) subset_counts<K, 0>(a, x, own, mask | m, bits, v);
        else if (n == 1) subset_counts<K, 1>(a, x, own, mask | m, bits, v);
        else if (n == 2) subset_counts<K, 2>(a, x, own, mask | m, bits, v);
        else subset_counts<K, 3>(a, x, own, mask | m, bits, v);
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (e < (1 << n)) {
                int cell = 0, left = n;
#pragma unroll
                for (int p = 0; p < 3; ++p) {
                    if (m & (4 >> p)) cell += ((e >> --left) & 1) * kStep[p];
                    else cell += 2 * kStep[p];
                }
                g[cell] = v[e];
            }
    }
#pragma unroll
    for (int st = 1; st < 27; st *= 3)
#pragma unroll
        for (int e = 0; e < 27; ++e)
            if ((e / st) % 3 == 2) g[e] = g[e] - g[e - st] - g[e - 2 * st];
}

// Inner cells with the outer positions' genotypes O (base-3 digits of the first K - 4 positions) and
// position K - 4 fixed to mid (0, 1) or any (2).
template <int K>
__device__ __forceinline__ void outer_cells(const SetArgs& a, const int* x, const uint32_t* own, int outer,
                                            int mid, uint32_t* g) {
    // every outer position with genotype 2 expands into any - 0 - 1
    int mask = 0, bits = 0, n2 = 0, pos2[2] = {0, 0};
#pragma unroll
    for (int p = 0; p < K - 4; ++p) {
        const int d = p == K - 5 ? outer % 3 : outer / 3, bit = 1 << (K - 1 - p);
        if (d == 2) pos2[n2++] = bit;
        else {
            mask |= bit;
            bits |= d ? bit : 0;
        }
    }
    if (mid < 2) {
        mask |= 8;
        bits |= mid ? 8 : 0;
    }
    inner_cells<K>(a, x, own, mask, bits, g);
    uint32_t t[27];
#pragma unroll
    for (int c = 1; c < 9; ++c) {
        const int c0 = c % 3, c1 = c / 3;   // per position with genotype 2: any, 0, 1
        if (n2 < 2 && c1 > 0) continue;
        if (n2 < 1) continue;
        int mk = mask, bt = bits;
        if (c0) {
            mk |= pos2[0];
            bt |= c0 == 2 ? pos2[0] : 0;
        }
        if (c1) {
            mk |= pos2[1];
            bt |= c1 == 2 ? pos2[1] : 0;
        }
        inner_cells<K>(a, x, own, mk, bt, t);
        const bool minus = ((c0 != 0) != (c1 != 0));
#pragma unroll
        for (int e = 0; e < 27; ++e) g[e] = minus ? g[e] - t[e] : g[e] + t[e];
    }
}

// add(27 cells) for the whole table of a set, in cell order; own: its own counts (count_cells).
template <int K, class Add>
__device__ __forceinline__ void all_cells(const SetArgs& a, const int* x, const uint32_t* own, Add add) {
#pragma unroll 1
    for (int outer = 0; outer < (K == 4 ? 1 : K == 5 ? 3 : 9); ++outer) {
        // position K - 4: genotypes 0 and 1, then 2 as what is left of any
        uint32_t any[27], g[27];
        auto step = [&](int o) {
            outer_cells<K>(a, x, own, o, 2, any);
#pragma unroll
            for (int mid = 0; mid < 2; ++mid) {
                outer_cells<K>(a, x, own, o, mid, g);
                add(g);
#pragma unroll
                for (int e = 0; e < 27; ++e) any[e] -= g[e];
            }
            add(any);
        };
        if (K == 4) step(0);
        else if (K == 5) {
            if (outer == 0) step(0);
            else if (outer == 1) step(1);
            else step(2);
        } else {
            switch (outer) {
                case 0: step(0); break;
                case 1: step(1); break;
                case 2: step(2); break;
                case 3: step(3); break;
                case 4: step(4); break;
                case 5: step(5); break;
                case 6: step(6); break;
                case 7: step(7); break;
                default: step(8); break;
            }
        }
    }
}
// Adds the 27 cells' K2 terms in FP32.
__device__ __forceinline__ float add_terms(const float* lf, const uint32_t* g, float s) {
#pragma unroll
    for (int e = 0; e < 27; ++e) {
        const uint32_t r0 = g[e] & 0xFFFFu, r1 = g[e] >> 16;
        s += (lf[r0 + r1 + 1] - lf[r0]) - lf[r1];
    }
    return s;
}
// The same in FP64, every operation that of the direct forms.
__device__ __forceinline__ double add_terms64(const double* __restrict__ lf64, const uint32_t* g, double s) {
#pragma unroll 3
    for (int e = 0; e < 27; ++e) {
        const uint32_t r0 = g[e] & 0xFFFFu, r1 = g[e] >> 16;
        s = __dadd_rn(s, __dsub_rn(__dsub_rn(lf64[r0 + r1 + 1], lf64[r0]), lf64[r1]));
    }
    return s;
}

// FP32 scores of all sets (or of every stride-th one into `sample`); those at or below the threshold
// go to the candidate list.  Bound by POPC (2^K a word and set); the lookups of the score come from
// shared memory where the table fits (kSmemLf).
constexpr int kSetThreads = 128;
constexpr int kSetLfMax = 12288;         // log-factorials in shared memory, at most
template <int K, bool kSmemLf>
__global__ void __launch_bounds__(kSetThreads)
set_scan_kernel(const SetArgs a, long long stride, long long n, float* __restrict__ sample,
                SetCtrl* ctrl, SetCand* __restrict__ cand, unsigned cap) {
    extern __shared__ float s_lf[];
    if (kSmemLf) {
        for (int e = threadIdx.x; e < a.n_lf; e += kSetThreads) s_lf[e] = a.lf[e];
        __syncthreads();
    }
    const float* const lf = kSmemLf ? s_lf : a.lf;
    if (!sample && ctrl->n_cand > cap) return;   // full: the sample says so, or this pass so far
    const float thr = sample ? 0.f : ctrl->thr;
    for (long long t = (long long)blockIdx.x * kSetThreads + threadIdx.x; t < n;
         t += (long long)gridDim.x * kSetThreads) {
        const long long q = t * stride;
        int x[K];
        decode_colex<K>(a, q, x);
        uint32_t own[1 << K];
        count_cells<K>(a.pl, x, own);
        float s = 0.f;
        all_cells<K>(a, x, own, [&](const uint32_t* g) { s = add_terms(lf, g, s); });
        s = fmaxf(s, 0.f);
        if (sample) {
            sample[t] = s;
        } else if (s <= thr) {
            const unsigned pos = atomicAdd(&ctrl->n_cand, 1u);
            if (pos < cap) cand[pos] = SetCand{q, s};
        }
    }
}

// The k-th smallest score (scores are not negative: their bit patterns sort like them) of n floats
// `step` floats apart; ctrl->thr becomes that + 2 delta, rounded up: no set of the answer scores
// higher.  One block.  Of the list (n_dev) its first `cap` candidates; of a sample of every `stride`-th
// item also whether the items that tie at the k-th score alone would overflow the list, which is then
// marked full before the scan begins.
__global__ void __launch_bounds__(1024)
set_threshold_kernel(const float* __restrict__ v, int step, long long n, const unsigned* __restrict__ n_dev,
                     int k, float delta, long long stride, unsigned cap, SetCtrl* ctrl) {
    __shared__ unsigned hist[256];
    __shared__ unsigned s_prefix, s_rank, s_ties;
    if (n_dev) {
        if (ctrl->tied) return;
        n = min(n, (long long)*n_dev);
    }
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) {
        s_prefix = 0u;
        s_rank = (unsigned)k;
    }
    unsigned mask = 0u;
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int b = tid; b < 256; b += 1024) hist[b] = 0u;
        __syncthreads();
        const unsigned prefix = s_prefix, rank = s_rank;
        for (long long e = tid; e < n; e += 1024) {
            const unsigned u = __float_as_uint(v[e * step]);
            if ((u & mask) == prefix) atomicAdd(&hist[(u >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (tid < 32) {   // the bin that holds the rank: eight bins a lane
            unsigned c[8], sum = 0u;
#pragma unroll
            for (int b = 0; b < 8; ++b) sum += c[b] = hist[8 * lane + b];
            unsigned incl = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned o = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += o;
            }
            unsigned before = incl - sum;
            if (before < rank && rank <= incl) {
                int b = 0;
                while (before + c[b] < rank) before += c[b++];
                s_rank = rank - before;
                s_ties = c[b];
                s_prefix = prefix | ((unsigned)(8 * lane + b) << shift);
            }
        }
        mask |= 255u << shift;
        __syncthreads();
    }
    if (tid == 0) {
        if (n_dev) ctrl->last = ctrl->thr;
        else {
            const bool tied = (double)s_ties * (double)stride > (double)cap;
            ctrl->tied = tied ? 1u : 0u;
            ctrl->n_cand = tied ? cap + 1u : 0u;
        }
        ctrl->thr = __fadd_ru(__uint_as_float(s_prefix), 2.f * delta);
        ctrl->n_final = 0u;
    }
}

// FP64 scores of the candidates inside the threshold, one warp each (none if the list overflowed).
template <int K>
__global__ void __launch_bounds__(kOrdThreads)
set_rescore_kernel(const SetArgs a, const double* __restrict__ lf64, SetCtrl* ctrl,
                   const SetCand* __restrict__ cand, unsigned cap, Item* __restrict__ fin) {
    uint32_t code[(Pow3<K>::v + 31) / 32];
    lane_codes<K>(code);
    const unsigned n = ctrl->n_cand <= cap ? ctrl->n_cand : 0u;
    const float thr = ctrl->thr;
    for (unsigned e = blockIdx.x * (kOrdThreads / 32) + (threadIdx.x >> 5); e < n;
         e += gridDim.x * (kOrdThreads / 32)) {
        const SetCand cd = cand[e];
        if (!(cd.s <= thr)) continue;
        int x[K];
        decode_colex<K>(a, cd.q, x);
        const double sc = set_score<K>(a.pl, lf64, x, code);
        if ((threadIdx.x & 31) == 0) {
            const unsigned pos = atomicAdd(&ctrl->n_final, 1u);
            fin[pos] = Item{sc, lex_rank<K>(a, x)};   // at most one per candidate
        }
    }
}

// The k best of at most kPairBlock rescored sets, sorted (more are merged, pair_merge_kernel).
__global__ void __launch_bounds__(kPairThreads)
set_final_kernel(const SetCtrl* ctrl, unsigned cap, const Item* __restrict__ fin, int k, Item* __restrict__ out) {
    __shared__ Item it[kPairBlock];
    if (!in_one_block(ctrl, cap)) return;
    const int n = (int)ctrl->n_final;
    int n2 = 64;
    while (n2 < n || n2 < k) n2 <<= 1;
    for (int t = threadIdx.x; t < n2; t += kPairThreads) it[t] = t < n ? fin[t] : pad_item();
    __syncthreads();
    sort_items(it, n2);
    for (int t = threadIdx.x; t < k; t += kPairThreads) out[t] = it[t];
}

// Where more sets lie at the threshold than the list holds: every set scored in FP64 from its counted
// table, a block's k best of 2048 consecutive ranks at or below thr into out[b * k ..], merged like the
// direct form's.  Four SNPs only: there the passes before it are a sixth of the direct form's time
// (60 SNPs x 1000 samples), with five and six a thirtieth.
constexpr int kTiedThreads = 512;     // four sets each: with 128 threads 50 SNPs, fewer blocks than SMs, took 521 us for 421
template <int K>
__global__ void __launch_bounds__(kTiedThreads)
set_tied_kernel(const SetArgs a, const double* __restrict__ lf64, float thr, int k, Item* __restrict__ out) {
    __shared__ Item it[kPairBlock];
    bool any = false;
    for (int t = threadIdx.x; t < kPairBlock; t += kTiedThreads) {
        const long long q = (long long)blockIdx.x * kPairBlock + t;
        it[t] = pad_item();
        if (q >= a.n_sets) continue;
        int x[K];
        decode_colex<K>(a, q, x);
        uint32_t own[1 << K];
        count_cells<K>(a.pl, x, own);
        double s = 0.0;
        all_cells<K>(a, x, own, [&](const uint32_t* g) { s = add_terms64(lf64, g, s); });
        if (!(s <= (double)thr)) continue;
        it[t] = Item{s, lex_rank<K>(a, x)};
        any = true;
    }
    if (__syncthreads_or(any)) sort_items(it);
    for (int t = threadIdx.x; t < k; t += kTiedThreads) out[(long long)blockIdx.x * k + t] = it[t];
}

// ---------------------------------------------------------------- pairs, thresholded form
// FP64 scores, rounded up to FP32, of every stride-th pair.
__global__ void __launch_bounds__(256)
pair_sample_kernel(PairTables pt, const double* __restrict__ lf64, int M, long long stride, long long n,
                   float* __restrict__ sample) {
    for (long long t = (long long)blockIdx.x * 256 + threadIdx.x; t < n; t += (long long)gridDim.x * 256) {
        const long long p = t * stride;
        int i, j, r[2][9];
        decode_pair(p, &i, &j);
        sample[t] = pair_cells(pt, M, p, i, j, r) ? __double2float_ru(pair_score(r, lf64))
                                                  : __int_as_float(0x7f800000);
    }
}
// Pairs that may lie at or below the threshold: a table-free bound first (that of the compacted
// triplet scan with 9 cells, cmp_bound_terms: K2 >= c (sum of q) + (ln of the product of q) / 2 -
// off), the FP64 score for the few it lets through.  Reads each pair table once (32 bytes a pair, the
// floor); the direct form sorts every 2048 pairs it scores.  CTA row y: second SNP j = y + 1, ...
__global__ void __launch_bounds__(256)
pair_filter_kernel(PairTables pt, const double* __restrict__ lf64, int M, float bound_c, float bound_off,
                   int minor, SetCtrl* ctrl, SetCand* __restrict__ cand, unsigned cap) {
    // the list is full: the sample says so, or this pass so far (a load past L1 for every block cost 110
    // us of 280)
    if (ctrl->n_cand > cap) return;
    const float thr = ctrl->thr, cut = __fadd_ru(thr, bound_off);
    for (int j = 1 + blockIdx.y; j < M; j += gridDim.y) {
        const int i = blockIdx.x * 256 + threadIdx.x;
        if (i >= j) continue;
        const long long p = pair_index(i, j);
        int r[2][9];
        if (!pair_cells(pt, M, p, i, j, r)) continue;
        float sum = 0.f, prod = 1.f;
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const float us = (float)(r[0][e] + r[1][e] + 2), um = (float)((minor ? r[1][e] : r[0][e]) + 1);
            const float q = __fmaf_rn(__fmul_rn(um, pair_nrcp(us)), um, um);
            sum = __fadd_rn(sum, q);
            prod = __fmul_rn(prod, q);
        }
        if (__fmaf_rn(bound_c, sum, 0.34657359f * lg2_hw(prod)) > cut) continue;
        const float s = __double2float_ru(pair_score(r, lf64));
        if (s <= thr) {
            const unsigned pos = atomicAdd(&ctrl->n_cand, 1u);
            if (pos < cap) cand[pos] = SetCand{p, s};
        }
    }
}
__global__ void __launch_bounds__(256)
pair_rescore_kernel(PairTables pt, const double* __restrict__ lf64, int M, SetCtrl* ctrl,
                    const SetCand* __restrict__ cand, unsigned cap, Item* __restrict__ fin) {
    const unsigned n = ctrl->n_cand <= cap ? ctrl->n_cand : 0u;
    const float thr = ctrl->thr;
    for (unsigned e = blockIdx.x * 256 + threadIdx.x; e < n; e += gridDim.x * 256) {
        const SetCand cd = cand[e];
        if (!(cd.s <= thr)) continue;
        int i, j, r[2][9];
        decode_pair(cd.q, &i, &j);
        pair_cells(pt, M, cd.q, i, j, r);
        const unsigned pos = atomicAdd(&ctrl->n_final, 1u);
        fin[pos] = Item{pair_score(r, lf64), (long long)i * M + j};   // at most one per candidate
    }
}

constexpr unsigned kSetCand = 1u << 18;          // candidate list
constexpr size_t kSubsetBytes = (size_t)16 << 30;   // counts of the smaller sets, at most
// items of one of the two buffers that merge the rescored candidates
constexpr size_t kMergeItems = (size_t)(kSetCand / kPairBlock) * EPI3_MAX_TOPK;

// Entries of the list that a scan of n items uses.  A candidate of a pair or four-SNP scan costs some
// ten times an item of the form that answers when the list overflows (230 300 tied sets of 50 SNPs x 500
// samples: 1975 us through the list, 388 by the direct form), so an eighth of the items at most; with
// five and six SNPs it costs the same.
unsigned list_cap(long long n, int order, unsigned most) {
    long long cap = kSetCand;
    if (order <= 4 && n / 8 < cap) cap = n / 8 < kPairBlock ? kPairBlock : n / 8;
    return cap < most ? (unsigned)cap : most;
}

struct SetLayout {
    size_t binom, lf, ctrl, cand, fin, best, merge, sample, sub[6], total;
    long long n_sample;
};
SetLayout set_layout(int M, int N, int order) {
    SetLayout L{};
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += (bytes + 255) & ~(size_t)255;
        return at;
    };
    const long long n = choose_ll(M, order);
    L.n_sample = n / 256 < 16384 ? (n < 16384 ? n : 16384) : n / 256 < 262144 ? n / 256 : 262144;
    L.binom = take(sizeof(long long) * 7 * ((size_t)M + 1));
    L.lf = take(sizeof(float) * ((size_t)N + 2));
    L.ctrl = take(sizeof(SetCtrl));
    L.cand = take(sizeof(SetCand) * kSetCand);
    L.fin = take(sizeof(Item) * kSetCand);
    L.best = take(sizeof(Item) * EPI3_MAX_TOPK);
    L.merge = take(sizeof(Item) * 2 * kMergeItems);
    L.sample = take(sizeof(float) * (size_t)L.n_sample);
    for (int t = 1; t < order; ++t) L.sub[t] = take((sizeof(uint32_t) << t) * (size_t)choose_ll(M, t));
    L.total = o;
    return L;
}

template <int T>
cudaError_t count_subsets(const SetArgs& a, int grid, cudaStream_t st) {
    const long long n = choose_ll(a.pl.M, T);
    const long long blocks = (n + 127) / 128;
    set_count_kernel<T><<<(unsigned)(blocks < grid ? blocks : grid), 128, 0, st>>>(a, n);
    return cudaGetLastError();
}

// Passes over the items until the list of candidates holds all of them, or cannot: *done false.  A
// pass (`scan`) fills the list, `rescore` scores the candidates inside the list's own threshold in FP64
// into fin, `emit` writes the answer.  One wait a pass.
template <class Scan, class Rescore, class Emit>
cudaError_t threshold_passes(int k, float delta, unsigned cap, char* base, size_t ctrl_at, size_t cand_at, size_t fin_at,
                             size_t best_at, size_t merge_at, SetCtrl* h_ctrl, ThresholdInfo* info, cudaStream_t st,
                             Scan scan, Rescore rescore, Emit emit) {
    SetCtrl* const ctrl = reinterpret_cast<SetCtrl*>(base + ctrl_at);
    SetCand* const cand = reinterpret_cast<SetCand*>(base + cand_at);
    Item* const fin = reinterpret_cast<Item*>(base + fin_at);
    Item* const best = reinterpret_cast<Item*>(base + best_at);
    Item* const merge = reinterpret_cast<Item*>(base + merge_at);
    info->done = false;
    for (int attempt = 0;; ++attempt) {
        scan(ctrl, cand);
        // the threshold from the candidates themselves (any k of them bound the k-th)
        set_threshold_kernel<<<1, 1024, 0, st>>>(&cand->s, sizeof(SetCand) / sizeof(float), cap, &ctrl->n_cand, k,
                                                 delta, 1, cap, ctrl);
        rescore(ctrl, cand, fin);
        set_final_kernel<<<1, kPairThreads, 0, st>>>(ctrl, cap, fin, k, best);
        emit(best, ctrl);
        info->launches += 5;
        cudaError_t e = cudaMemcpyAsync(h_ctrl, ctrl, sizeof(SetCtrl), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        info->thr = h_ctrl->thr;
        info->n_cand = h_ctrl->n_cand;
        info->n_final = h_ctrl->n_final;
        if (h_ctrl->n_cand <= cap) {
            info->done = true;
            if (h_ctrl->n_final <= (unsigned)kPairBlock) return cudaSuccess;
            const Item* top = nullptr;   // thousands at the k-th score
            e = merge_items(fin, h_ctrl->n_final, k, merge, merge + kMergeItems, &top, &info->launches, st);
            if (e != cudaSuccess) return e;
            emit(top, nullptr);
            ++info->launches;
            return cudaGetLastError();
        }
        // the list overflowed: once more with the threshold of what it holds, if that is lower
        if (h_ctrl->tied || !(h_ctrl->thr < h_ctrl->last) || attempt == 2) return cudaSuccess;
        e = cudaMemsetAsync(&ctrl->n_cand, 0, sizeof(unsigned), st);
        if (e != cudaSuccess) return e;
    }
}

template <int K>
cudaError_t set_scan_k(const SetArgs& a, const SetLayout& L, const double* lf64, int sms, int k, float delta,
                       unsigned cap, char* base, SetCtrl* h_ctrl, int32_t* out_snps, double* out_s,
                       ThresholdInfo* info, cudaStream_t st) {
    const bool smem = a.n_lf <= kSetLfMax;
    const size_t bytes = smem ? sizeof(float) * (size_t)a.n_lf : 0;
    float* const sample = reinterpret_cast<float*>(base + L.sample);
    const int grid = 16 * sms;
    cudaError_t e = cudaSuccess;
    e = count_subsets<1>(a, grid, st);
    if (e == cudaSuccess) e = count_subsets<2>(a, grid, st);
    if (e == cudaSuccess) e = count_subsets<3>(a, grid, st);
    if (e == cudaSuccess && K > 4) e = count_subsets<4>(a, grid, st);
    if (e == cudaSuccess && K > 5) e = count_subsets<5>(a, grid, st);
    if (e != cudaSuccess) return e;
    auto scan = [&](long long stride, long long n, float* smp, SetCtrl* ctrl, SetCand* cand) {
        const long long blocks = (n + kSetThreads - 1) / kSetThreads;
        const unsigned g = (unsigned)(blocks < grid ? blocks : grid);
        if (smem) set_scan_kernel<K, true><<<g, kSetThreads, bytes, st>>>(a, stride, n, smp, ctrl, cand, cap);
        else set_scan_kernel<K, false><<<g, kSetThreads, 0, st>>>(a, stride, n, smp, ctrl, cand, cap);
    };
    SetCtrl* const ctrl = reinterpret_cast<SetCtrl*>(base + L.ctrl);
    const long long stride = a.n_sets / L.n_sample;
    scan(stride, L.n_sample, sample, ctrl, nullptr);
    set_threshold_kernel<<<1, 1024, 0, st>>>(sample, 1, L.n_sample, nullptr, k, delta, stride, cap, ctrl);
    info->launches += K + 1;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return threshold_passes(
        k, delta, cap, base, L.ctrl, L.cand, L.fin, L.best, L.merge, h_ctrl, info, st,
        [&](SetCtrl* c, SetCand* cand) { scan(1, a.n_sets, nullptr, c, cand); },
        [&](SetCtrl* c, const SetCand* cand, Item* fin) {
            set_rescore_kernel<K><<<4 * sms, kOrdThreads, 0, st>>>(a, lf64, c, cand, cap, fin);
        },
        [&](const Item* top, const SetCtrl* c) {
            order_emit_kernel<K><<<1, 512, 0, st>>>(top, k, a.pl.M, c, cap, out_snps, out_s);
        });
}

}  // namespace

// Scratch bytes of the counted form, 0 if it does not serve the size.
size_t set_scan_scratch(int M, int N, int order) {
    if (order < 4 || order > 6 || M < order) return 0;
    // A few sets take the direct form: up to one a thread (four SNPs) or one a warp of its first block
    // it needs two launches instead of eleven and more (4 SNPs of 10 with 2000 samples, 210 sets: 153 us,
    // counted 178; of 11, 330 sets: 195 and 176; 6 of 7: 402 and 661; 5 of 7, 21 sets: 384 and 275).
    if (choose_ll(M, order) <= (order == 4 ? kQuadThreads : kOrdThreads / 32)) return 0;
    double sub = 0.0, c = 1.0;
    for (int t = 1; t < order; ++t) {
        c = c * (M - t + 1) / t;
        sub += c * (4 << t);
    }
    if (sub > (double)kSubsetBytes) return 0;
    return set_layout(M, N, order).total;
}

// The kernels' view of the counted form's scratch.
static SetArgs set_args(const Planes& pl, int n0, int n1, int order, const SetLayout& L, char* base) {
    SetArgs a{};
    a.pl = pl;
    a.binom = reinterpret_cast<const long long*>(base + L.binom);
    a.lf = reinterpret_cast<const float*>(base + L.lf);
    a.n_lf = n0 + n1 + 2;
    for (int t = 1; t < order; ++t) a.sub[t] = reinterpret_cast<uint32_t*>(base + L.sub[t]);
    a.total = (uint32_t)n0 + ((uint32_t)n1 << 16);
    a.n_sets = choose_ll(pl.M, order);
    return a;
}

cudaError_t launch_set_scan(const Planes& pl, const double* lf64, int n0, int n1, int order, int k, int sms,
                            unsigned cap, void* scratch, void* h_ctrl, int32_t* out_snps, double* out_s,
                            ThresholdInfo* info, cudaStream_t st) {
    const int N = n0 + n1;
    const SetLayout L = set_layout(pl.M, N, order);
    char* const base = static_cast<char*>(scratch);
    const SetArgs a = set_args(pl, n0, n1, order, L, base);
    cap = list_cap(a.n_sets, order, cap);
    // |FP32 score - K2|: the table's entries and the two subtractions round by 2^-24 of lf(r + 1) at
    // most, and the cells' lf(r + 1) sum to at most lf(N + 3^K); each addition rounds by 2^-24 of the
    // score.  Both with a margin, plus the subtraction's own rounding of small terms.
    const double cells = order == 4 ? 81.0 : order == 5 ? 243.0 : 729.0;
    const double top = std::lgamma((double)N + cells + 1.0);
    const double score = (double)N * std::log(2.0) + std::fmin((double)N, cells) * std::log((double)N + 2.0);
    const float delta = (float)(std::ldexp(1.0, -24) * (6.0 * top + cells * score) * 1.1 + 0.01);
    set_tables_kernel<<<sms, 256, 0, st>>>(pl.M, lf64, N + 2, reinterpret_cast<long long*>(base + L.binom),
                                           reinterpret_cast<float*>(base + L.lf));
    info->launches = 1;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    SetCtrl* const hc = static_cast<SetCtrl*>(h_ctrl);
    if (order == 4) return set_scan_k<4>(a, L, lf64, sms, k, delta, cap, base, hc, out_snps, out_s, info, st);
    if (order == 5) return set_scan_k<5>(a, L, lf64, sms, k, delta, cap, base, hc, out_snps, out_s, info, st);
    return set_scan_k<6>(a, L, lf64, sms, k, delta, cap, base, hc, out_snps, out_s, info, st);
}

cudaError_t launch_quad_tied(const Planes& pl, const double* lf64, int n0, int n1, float thr, int k, void* tables,
                             void* scratch, int32_t* out_snps, double* out_s, int* launches, cudaStream_t st) {
    const SetArgs a = set_args(pl, n0, n1, 4, set_layout(pl.M, n0 + n1, 4), static_cast<char*>(tables));
    const long long blocks = (a.n_sets + kPairBlock - 1) / kPairBlock;
    Item* const items = static_cast<Item*>(scratch);
    set_tied_kernel<4><<<(unsigned)blocks, kTiedThreads, 0, st>>>(a, lf64, thr, k, items);
    cudaError_t e = cudaGetLastError();
    const Item* best = nullptr;
    if (e == cudaSuccess) e = merge_items(items, blocks * k, k, items, items + blocks * k, &best, launches, st);
    if (e != cudaSuccess) return e;
    order_emit_kernel<4><<<1, 512, 0, st>>>(best, k, a.pl.M, nullptr, 0u, out_snps, out_s);
    *launches += 2;
    return cudaGetLastError();
}

long long order_count(int M, int order) { return choose_ll(M, order); }

size_t order_scan_scratch(int M, int order, int k) {
    const long long blocks = (choose_ll(M, order) + kPairBlock - 1) / kPairBlock;
    return (size_t)2 * (size_t)blocks * (size_t)k * sizeof(Item);
}

cudaError_t launch_order_scan(const Planes& pl, const double* lf64, int order, int k, void* scratch,
                              int32_t* out_snps, double* out_s, int* launches, cudaStream_t st) {
    if (order == 5) return order_scan_k<5>(pl, lf64, k, scratch, out_snps, out_s, launches, st);
    if (order == 6) return order_scan_k<6>(pl, lf64, k, scratch, out_snps, out_s, launches, st);
    return cudaErrorInvalidValue;
}

long long quad_count(int M) { return choose_ll(M, 4); }

size_t quad_scan_scratch(int M, int k) {
    const long long blocks = (choose_ll(M, 4) + kPairBlock - 1) / kPairBlock;
    return (size_t)2 * (size_t)blocks * (size_t)k * sizeof(Item);
}

cudaError_t launch_quad_scan(const Planes& pl, const double* lf64, int n0, int n1, int k,
                             void* scratch, int32_t* out_snps, double* out_s, int* launches, cudaStream_t st) {
    const long long n_sets = choose_ll(pl.M, 4);
    const long long blocks = (n_sets + kPairBlock - 1) / kPairBlock;
    Item* const a = static_cast<Item*>(scratch);
    quad_score_kernel<<<(unsigned)blocks, kQuadThreads, 0, st>>>(pl, lf64, n0, n1, n_sets, k, a);
    cudaError_t e = cudaGetLastError();
    const Item* best = nullptr;
    if (e == cudaSuccess) e = merge_items(a, blocks * k, k, a, a + blocks * k, &best, launches, st);
    if (e != cudaSuccess) return e;
    quad_emit_kernel<<<1, 512, 0, st>>>(best, k, out_snps, out_s);
    *launches += 2;
    return cudaGetLastError();
}

namespace {
struct PairLayout {
    size_t ctrl, cand, fin, best, merge, sample, total;
    long long n_sample;
};
PairLayout pair_layout(long long n) {
    PairLayout L{};
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += (bytes + 255) & ~(size_t)255;
        return at;
    };
    // evenly spaced pairs for the first threshold: enough that about k n / n_sample candidates are few
    L.n_sample = n < 32768 ? n : 32768;
    L.ctrl = take(sizeof(SetCtrl));
    L.cand = take(sizeof(SetCand) * kSetCand);
    L.fin = take(sizeof(Item) * kSetCand);
    L.best = take(sizeof(Item) * EPI3_MAX_TOPK);
    L.merge = take(sizeof(Item) * 2 * kMergeItems);
    L.sample = take(sizeof(float) * (size_t)L.n_sample);
    L.total = o;
    return L;
}
}  // namespace

size_t pair_filter_scratch(long long n_pairs) { return pair_layout(n_pairs).total; }

cudaError_t launch_pair_filter(const PairTables& pt, const double* lf64, int M, int k, const CmpBoundTerms& bound,
                               int sms, unsigned cap, void* scratch, void* h_ctrl, int32_t* out_pairs, double* out_s,
                               ThresholdInfo* info, cudaStream_t st) {
    const PairLayout L = pair_layout(pt.n_pairs);
    char* const base = static_cast<char*>(scratch);
    float* const sample = reinterpret_cast<float*>(base + L.sample);
    cap = list_cap(pt.n_pairs, 2, cap);
    const long long stride = pt.n_pairs / L.n_sample;
    pair_sample_kernel<<<(unsigned)((L.n_sample + 255) / 256), 256, 0, st>>>(pt, lf64, M, stride, L.n_sample, sample);
    set_threshold_kernel<<<1, 1024, 0, st>>>(sample, 1, L.n_sample, nullptr, k, 0.f, stride, cap,
                                             reinterpret_cast<SetCtrl*>(base + L.ctrl));
    info->launches = 2;
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const dim3 grid((M + 255) / 256, M < 8192 ? M : 8192);
    return threshold_passes(
        k, 0.f, cap, base, L.ctrl, L.cand, L.fin, L.best, L.merge, static_cast<SetCtrl*>(h_ctrl), info, st,
        [&](SetCtrl* c, SetCand* cand) {
            pair_filter_kernel<<<grid, 256, 0, st>>>(pt, lf64, M, bound.c, bound.off2, bound.minor, c, cand, cap);
        },
        [&](SetCtrl* c, const SetCand* cand, Item* fin) {
            pair_rescore_kernel<<<sms, 256, 0, st>>>(pt, lf64, M, c, cand, cap, fin);
        },
        [&](const Item* top, const SetCtrl* c) {
            pair_emit_kernel<<<1, 512, 0, st>>>(top, k, M, c, cap, out_pairs, out_s);
        });
}

size_t pair_scan_scratch(long long n_pairs, int k) {
    const long long blocks = (n_pairs + kPairBlock - 1) / kPairBlock;
    return (size_t)2 * (size_t)blocks * (size_t)k * sizeof(Item);
}

cudaError_t launch_pair_scan(const PairTables& pt, const double* lf64, int M, float thr, int k,
                             void* scratch, int32_t* out_pairs, double* out_s, int* launches, cudaStream_t st) {
    const long long n_pairs = pt.n_pairs;
    const long long blocks = (n_pairs + kPairBlock - 1) / kPairBlock;
    Item* const a = static_cast<Item*>(scratch);
    pair_score_kernel<<<(unsigned)blocks, kPairThreads, 0, st>>>(pt, lf64, M, n_pairs, thr, k, a);
    cudaError_t e = cudaGetLastError();
    const Item* best = nullptr;
    if (e == cudaSuccess) e = merge_items(a, blocks * k, k, a, a + blocks * k, &best, launches, st);
    if (e != cudaSuccess) return e;
    pair_emit_kernel<<<1, 512, 0, st>>>(best, k, M, nullptr, 0u, out_pairs, out_s);
    *launches += 2;
    return cudaGetLastError();
}

}  // namespace epi3
