// Tensor-core counting scan on sample-compacted operands (path EPI3_PATH_MMA4C).
//
// For a fixed first SNP i, class c and genotype a of SNP i, let S be the samples of class c
// with g_i = a.  The cells (a, b, z) with b, z in {0,1} of every triplet (i, j, k) are
//     n(a, b, z) = sum over s in S of [g_j(s) = b] [g_k(s) = z],
// a plain GEMM of two one-hot matrices over the samples of S: rows (j, b) x columns (k, z).  Two
// genotypes a of SNP i are counted this way, the two least frequent over all samples; the most
// frequent one is derived with the other 19 cells (the same genotype in both classes), so the
// GEMMs run over the smallest share of the samples.  The samples of each of the four sets
// (c, a) are gathered once per first SNP ("compaction": the samples' genotype bits, transposed and
// expanded to FP4 E2M1 0/1 values in the 128B-swizzled shared-memory image), and the scan
// multiplies compacted chunks straight from L2: both MMA operands come from shared memory,
// filled by bulk copies, with no operand formed on chip and 4 MACs per sample-triplet whose
// first-SNP genotype is counted.  SNP i's genotypes are relabelled (counted ones 0 and 1, the
// derived one 2) in the pair-table and marginal inputs; the epilogue derives the 19 other cells and
// bounds the table's score from below; the few triplets whose bound does not exceed the candidate
// threshold get their exact integer table and FP32 score: K2 and the candidate band exactly as in
// the other scans (Eq. 1; the paper counts with POPCNT, Sec. IV, and points at tensor-core
// formulations in Sec. II).
//
// Every set carries one bias sample (a 1 in every row) after its samples, so every accumulator
// ends at count + 1, the argument of the epilogue's count + 1 arithmetic.
//
// Tile = (i, 64 second SNPs j, 32 third SNPs k): MMA M = 128 rows (j, b), N = 64 columns (k, z),
// kind::mxf4 (K = 64 FP4 samples per instruction, four per 256-sample step, every block scale
// 2^0), FP32 accumulation in tensor memory: one 64-column region per set, regions taken from a
// ring of seven so that the next tile's first sets run while the epilogue reads this one.
// Shared memory: a ring of three slots of two K-steps each (A 32 KB in one copy, B 2 x 8 KB),
// with one full barrier, one empty barrier and one tcgen05.commit per slot (a set's odd last
// step takes half a slot): every commit costs the tensor pipe a bubble, so fewer, larger slots
// beat one slot per step.
//
// Warp roles (16 warps): 0 = operand loader + tensor-memory allocator, 1 = MMA issuer, 2-3 = stagers
// (the per-tile constants of the derived cells), 4-15 = epilogue.  The epilogue warps meet only every
// few tiles; mbarriers pass accumulators and staged constants to and from each.  Every mbarrier wait
// is bounded; on timeout the kernel records kStTimeout, waits for its own copies and MMAs, frees
// tensor memory and returns.
//
// Measured (GB300, scan kernel without the compaction): 2048 SNPs x 4096 samples 46.0 -> 18.6 ms,
// 2048 x 16384 50.2 -> 29.5 ms.  At 4096 samples a tile takes 7600 cycles, of which the bound's
// operations take the FP32 pipe 3070; at 16 384 it takes 12 100, of which the tensor pipe's operand
// reads and the ring's hand-offs alone take 10 300.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "epi3_internal.cuh"
#include "tc_common.cuh"

namespace epi3 {

namespace {

constexpr int kCmpChunk = 16384;         // one compacted chunk: 128 rows (m, z) x 256 samples

// 32 x 32 bit transpose across a warp: bit t of lane r's x becomes bit r of lane t's.
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 16; k >= 1; k >>= 1) {
        const uint32_t m = k == 16 ? 0x0000FFFFu : k == 8 ? 0x00FF00FFu : k == 4 ? 0x0F0F0F0Fu
                         : k == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, k);
        x = lane & k ? (x & ~m) | ((y >> k) & m) : (x & m) | ((y << k) & ~m);
    }
    return x;
}

// ------------------------------------------------------------------ compaction
// The compaction gathers samples: what one sample contributes to a 64-SNP block is 16 bytes, the
// genotype-0 and genotype-1 bits of the block's SNPs (rows[c][b][s], built once per data set), and
// 32 gathered samples turn into a K-step unit of all 128 operand rows by four bit transposes across
// a warp (80 instructions for 128 words).  Extracting the selected bits of every row's plane words
// instead cost 40 instructions a source word and set, for 0.19 output words.
//
// Warp: one 32-sample word of class c, one block: planes -> rows.
__global__ void __launch_bounds__(256)
sample_rows_kernel(Planes pl, int nblk, uint4* __restrict__ rows) {
    const int lane = threadIdx.x & 31;
    const int words0 = 4 * pl.W4[0], words = words0 + 4 * pl.W4[1];
    const long long n = (long long)words * nblk;
    const int M = pl.M;
    for (long long t = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); t < n; t += (long long)gridDim.x * 8) {
        const int b = (int)(t / words), ww = (int)(t % words);
        const int c = ww >= words0 ? 1 : 0, w = c ? ww - words0 : ww;
        const int W4 = c ? pl.W4[1] : pl.W4[0];
        const uint32_t* const p =
            reinterpret_cast<const uint32_t*>(pl.planes + (c ? pl.coff[1] : pl.coff[0])) + (w & 3);
        uint32_t x[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {   // genotype e / 2, SNP half e % 2
            const int m = 64 * b + 32 * (e & 1) + lane;
            x[e] = m < M ? __ldg(p + ((size_t)((e >> 1) * W4 + (w >> 2)) * M + m) * 4) : 0u;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = warp_transpose(x[e]);
        rows[((size_t)b * words + ww) * 32 + lane] = make_uint4(x[0], x[1], x[2], x[3]);
    }
}

// CTA (f, c): the class-c samples of each counted genotype of first SNP i0 + f, ascending, into
// list + f N + (class 1: N0): slot 0's, then slot 1's.
__global__ void __launch_bounds__(256)
sample_list_kernel(Planes pl, const CmpFirst* __restrict__ firsts, int i0, int n0, int n,
                   uint32_t* __restrict__ list) {
    __shared__ uint32_t s_warp[8];
    const int f = blockIdx.x, c = blockIdx.y, i = i0 + f, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int W4 = c ? pl.W4[1] : pl.W4[0], W = 4 * W4, Nc = c ? n - n0 : n0, M = pl.M;
    const int drop = firsts[f].drop;
    uint32_t* const l0 = list + (size_t)f * n + (c ? n0 : 0);
    uint32_t* const l1 = l0 + firsts[f].cnt[2 * c];
    const uint32_t* const p = reinterpret_cast<const uint32_t*>(pl.planes + (c ? pl.coff[1] : pl.coff[0]));
    uint32_t at0 = 0, at1 = 0;
    for (int w0 = 0; w0 < W; w0 += 256) {
        const int w = w0 + tid;
        uint32_t m0 = 0u, m1 = 0u;
        if (w < W) {
            const uint32_t g0 = __ldg(p + ((size_t)(w >> 2) * M + i) * 4 + (w & 3));
            const uint32_t g1 = __ldg(p + ((size_t)(W4 + (w >> 2)) * M + i) * 4 + (w & 3));
            // genotype 2 by NOR, without the pad positions past the class's last sample
            const int nv = Nc - 32 * w;
            const uint32_t valid = nv >= 32 ? 0xFFFFFFFFu : (nv <= 0 ? 0u : (1u << nv) - 1u);
            const uint32_t g2 = ~(g0 | g1) & valid;
            m0 = drop == 0 ? g1 : g0;       // the two counted genotypes, ascending (cmp_geno)
            m1 = drop == 2 ? g1 : g2;
        }
        const uint32_t own = (uint32_t)__popc(m0) | ((uint32_t)__popc(m1) << 16);   // at most 8192 each
        uint32_t incl = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        if (lane == 31) s_warp[wid] = incl;
        __syncthreads();
        uint32_t before = incl - own, all = 0;
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            const uint32_t o = s_warp[v];
            before += v < wid ? o : 0u;
            all += o;
        }
        uint32_t* o0 = l0 + at0 + (before & 0xFFFFu);
        uint32_t* o1 = l1 + at1 + (before >> 16);
        for (; m0; m0 &= m0 - 1) *o0++ = (uint32_t)(32 * w + __ffs(m0) - 1);
        for (; m1; m1 &= m1 - 1) *o1++ = (uint32_t)(32 * w + __ffs(m1) - 1);
        at0 += all & 0xFFFFu;
        at1 += all >> 16;
        __syncthreads();
    }
}

// CTA (b, f, c): block b's chunks of the two sets of class c of first SNP f.  Rows of a chunk come in
// 16-row groups: row 16 G + 8 z + r holds SNP m = 64 b + 8 G + r with genotype z (8 SNPs of genotype
// 0, then the same 8 of genotype 1), so that a 16x256b tensor-memory load hands a thread both genotype
// rows of one SNP (see the epilogue).  Warp u makes unit u (32 samples) of every K-step: the samples
// in list order, then the bias sample (a 1 in every row), then zeros.  The 16 KB image is put together
// in shared memory and leaves in one bulk copy, two images in flight.  Bound by the chunks' writes
// (2048 x 16384: 14.2 GB).
constexpr int kCompactThreads = 256;
__global__ void __launch_bounds__(kCompactThreads)
compact_kernel(const uint4* __restrict__ rows, int words0, int words, const CmpFirst* __restrict__ firsts,
               const uint32_t* __restrict__ list, int n0, int n, uint8_t* __restrict__ cmp) {
    __shared__ __align__(128) uint8_t s_img[2][kCmpChunk];
    const int b = blockIdx.x, f = blockIdx.y, c = blockIdx.z;
    const CmpFirst* const fp = firsts + f;
    const int b_lo = fp->b_lo;
    if (b < b_lo) return;  // whole CTA: no block before the first SNP's successors
    const int tid = threadIdx.x, lane = tid & 31, u = tid >> 5;
    const uint4* const src = rows + ((size_t)b * words + (c ? words0 : 0)) * 32;
    const int ks[2] = {fp->ks[2 * c], fp->ks[2 * c + 1]}, cnt[2] = {fp->cnt[2 * c], fp->cnt[2 * c + 1]};
    const uint32_t* const l0 = list + (size_t)f * n + (c ? n0 : 0);
    const int steps = ks[0] + ks[1];
    auto gather = [&](int q) {   // this lane's sample of K-step q (both sets' steps in a row)
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (q >= steps) return v;
        const int s = q >= ks[0] ? 1 : 0, p = 256 * (s ? q - ks[0] : q) + 32 * u + lane, m = s ? cnt[1] : cnt[0];
        if (p < m) v = __ldg(src + __ldg(l0 + (s ? cnt[0] : 0) + p));
        else if (p == m) v = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
        return v;
    };
    uint4 next = gather(0);
    for (int q = 0; q < steps; ++q) {
        const uint4 v = next;
        next = gather(q + 1);
        const uint32_t x[4] = {warp_transpose(v.x), warp_transpose(v.y), warp_transpose(v.z), warp_transpose(v.w)};
        uint8_t* const img = s_img[q & 1];
        // the copy two K-steps ago has read this image
        if (tid == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        __syncthreads();
#pragma unroll
        for (int e = 0; e < 4; ++e) {   // genotype e / 2, SNP 32 (e % 2) + lane
            const uint32_t w = x[e];
            const int m = 32 * (e & 1) + lane, row = 16 * (m >> 3) + 8 * (e >> 1) + (m & 7);
            *reinterpret_cast<uint4*>(img + sw128_off((uint32_t)row, (uint32_t)u)) =
                make_uint4(byte_to_e2m1(w), byte_to_e2m1(w >> 8), byte_to_e2m1(w >> 16), byte_to_e2m1(w >> 24));
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            const int s = q >= ks[0] ? 1 : 0;
            const long long chunk = fp->base[2 * c + s] + (long long)(b - b_lo) * ks[s] + (s ? q - ks[0] : q);
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                         ::"l"(cmp + (size_t)chunk * kCmpChunk), "r"(smem_u32(img)), "r"(kCmpChunk) : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
    }
    if (tid == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// ------------------------------------------------------------------ the scan kernel
constexpr int kTJ = 64;                  // second SNPs per tile: A rows (j, b)
constexpr int kTK = 32;                  // third SNPs per tile: B rows (k, z), MMA N = 64
constexpr int kN = 2 * kTK;
constexpr int kSlotSteps = 2;            // K-steps per shared-memory slot: one commit frees both
constexpr int kSlots = 3;                // shared-memory ring
constexpr int kStepA = kCmpChunk;        // one K-step of A: 128 rows x 128 B
constexpr int kStepB = kCmpChunk / 2;    // one K-step of B: 64 rows x 128 B
constexpr int kSlotA = kSlotSteps * kStepA;
constexpr int kSlotB = kSlotSteps * kStepB;
constexpr int kCmpRegions = 7;           // 64-column accumulator regions (columns 0..447)
constexpr uint32_t kCmpSfCol = 480;      // block scales: A at 480..495, B at 496..511
// 16 warps: 0 loader, 1 MMA issuer, 2 and 3 stagers, 4..15 epilogue, 128 registers a thread.  The
// three epilogue warps of a tensor-memory lane quadrant (all on one SM quarter) split its eight
// items (2 lane groups x 4 column groups) 3 / 3 / 2.
constexpr int kCmpEpiWarp0 = 4, kCmpEpiWarps = 12, kCmpEpiThreads = kCmpEpiWarps * 32;
constexpr int kCmpEpiParts = kCmpEpiWarps / 4, kCmpEpiItems = (8 + kCmpEpiParts - 1) / kCmpEpiParts;
constexpr int kCmpThreads = (kCmpEpiWarp0 + kCmpEpiWarps) * 32;
static_assert(kTJ == 4 * 2 * 8 && kTK == 4 * 8, "epilogue item split");
static_assert(kCmpRegions * kN <= (int)kCmpSfCol, "tensor memory budget");
constexpr int kMaxSyncTiles = 16;        // tiles between the epilogue warps' rendezvous, at most

// One tile's epilogue inputs, staged by the stager warp (two buffers).  Every value comes for two
// tables, the samples of both classes (s, each u = count + 2) and those of the smaller class
// (m, u = count + 1), with the offsets that make a difference of u values a u value.
//   row[j][phase][..]  {s, s, m, m} per constant (f32x2 operands for two triplets of one j):
//                      phase a = 0, 1: (a, 0, .), (a, 1, .), (a, 2, .) summed over z;
//                      phase 2: (2, 0, .), (2, 1, .), (2, 2, .)
//   col[k / 2][phase]  {k, k + 1} per constant: phase a: s(a, ., 0), s(a, ., 1), m(a, ., 0),
//                      m(a, ., 1); phase 2 the same for a = 2
//   thr[j]             prune a triplet whose bound exceeds this (-inf: no triplet in this row)
//   i, f, jb, kb       the tile; flags: kStageRun the first tile of a run, kStageLast this CTA's last
struct CmpStage {
    float4 row[kTJ][3][3];
    float2 col[kTK / 2][3][4];
    float thr[kTJ];
    int f, jb, kb, flags;
};
constexpr int kStageRun = 1, kStageLast = 2;

// Instruction descriptor of kind::mxf4: A/B E2M1, UE8M0 scales, K-major, N = 64, M = 128.
constexpr uint32_t kIdescCmp = (1u << 7) | (1u << 10) | ((uint32_t)(kN >> 3) << 17) | (1u << 23) |
                               ((128u >> 4) << 24);

// One K-step: four MMAs of 64 samples (32 bytes of K each) into d, issued warp-wide by the lane
// that elect.sync picks (see tc_common.cuh), once for all four; acc: add to d from the first on.
__device__ __forceinline__ void mma_step_elect(uint32_t d, uint64_t a, uint64_t b, uint32_t acc,
                                               uint32_t sfa, uint32_t sfb) {
    asm volatile(
        "{\n .reg .pred p, e;\n .reg .b64 a1, a2, a3, b1, b2, b3;\n"
        " add.s64 a1, %1, 2;\n add.s64 a2, %1, 4;\n add.s64 a3, %1, 6;\n"
        " add.s64 b1, %2, 2;\n add.s64 b2, %2, 4;\n add.s64 b3, %2, 6;\n"
        " setp.ne.b32 p, %3, 0;\n elect.sync _|e, 0xffffffff;\n"
        " @e tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %6, [%4], [%5], p;\n"
        " @e tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], a1, b1, %6, [%4], [%5], 1;\n"
        " @e tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], a2, b2, %6, [%4], [%5], 1;\n"
        " @e tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], a3, b3, %6, [%4], [%5], 1;\n}\n"
        ::"r"(d), "l"(a), "l"(b), "r"(acc), "r"(sfa), "r"(sfb), "r"(kIdescCmp) : "memory");
}
// A slot's copies: its barrier told the bytes, the A chunks in one copy, the B halves of one or two
// chunks (b1: the second, if two).
__device__ __forceinline__ void load_slot_elect(uint32_t bar, uint32_t da, const uint8_t* a, uint32_t abytes,
                                                uint32_t db, const uint8_t* b, uint32_t two) {
    asm volatile(
        "{\n .reg .pred e, t;\n .reg .b32 n, d1;\n .reg .b64 b1;\n"
        " add.u32 n, %3, %7;\n setp.ne.u32 t, %6, 0;\n @t add.u32 n, n, %7;\n"
        " add.u32 d1, %4, %7;\n add.s64 b1, %5, %8;\n"
        " elect.sync _|e, 0xffffffff;\n and.pred t, t, e;\n"
        " @e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], n;\n"
        " @e cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%1], [%2], %3, [%0];\n"
        " @e cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%4], [%5], %7, [%0];\n"
        " @t cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [d1], [b1], %7, [%0];\n}\n"
        ::"r"(bar), "r"(da), "l"(a), "r"(abytes), "r"(db), "l"(b), "r"(two), "n"(kCmpChunk / 2), "n"(kCmpChunk)
        : "memory");
}

// 16 lanes x 16 FP32 columns from taddr: thread t gets lane t / 4 (v[0..1]) and lane t / 4 + 8
// (v[2..3]) at columns 2 (t % 4) + {0, 1}, then the same at columns + 8 (v[4..7]).
__device__ __forceinline__ void tc_ld16x2(uint32_t taddr, float* v) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]),
          "=f"(v[7])
        : "r"(taddr));
}
// A shared-memory load that stays where it is written: the compiler moves plain ones to their use,
// where their latency shows (2048 x 4096: 7740 -> 7310 cycles a tile with the next phase's constants
// loaded before a phase's work).
__device__ __forceinline__ void lds128(float4& v, const float4* p) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(smem_u32(p)));
}
// 16 bytes from global to shared memory, asynchronously.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
// Wait for every such load; the registers of two or four pass through, so that no use moves above it.
__device__ __forceinline__ void tc_wait_ld4(float (&v)[4][8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0][0]), "+f"(v[0][1]), "+f"(v[0][2]), "+f"(v[0][3]), "+f"(v[0][4]),
                   "+f"(v[0][5]), "+f"(v[0][6]), "+f"(v[0][7]), "+f"(v[1][0]), "+f"(v[1][1]),
                   "+f"(v[1][2]), "+f"(v[1][3]), "+f"(v[1][4]), "+f"(v[1][5]), "+f"(v[1][6]),
                   "+f"(v[1][7]), "+f"(v[2][0]), "+f"(v[2][1]), "+f"(v[2][2]), "+f"(v[2][3]),
                   "+f"(v[2][4]), "+f"(v[2][5]), "+f"(v[2][6]), "+f"(v[2][7]), "+f"(v[3][0]),
                   "+f"(v[3][1]), "+f"(v[3][2]), "+f"(v[3][3]), "+f"(v[3][4]), "+f"(v[3][5]),
                   "+f"(v[3][6]), "+f"(v[3][7]));
}

__device__ __forceinline__ void tc_wait_ld2(float (&v)[2][8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0][0]), "+f"(v[0][1]), "+f"(v[0][2]), "+f"(v[0][3]), "+f"(v[0][4]),
                   "+f"(v[0][5]), "+f"(v[0][6]), "+f"(v[0][7]), "+f"(v[1][0]), "+f"(v[1][1]),
                   "+f"(v[1][2]), "+f"(v[1][3]), "+f"(v[1][4]), "+f"(v[1][5]), "+f"(v[1][6]),
                   "+f"(v[1][7]));
}

// The tiles of a CTA, in order.  A run is a (j block, k block) of a group of consecutive first
// SNPs; CTA c takes runs c, c + gridDim.x, ... and in each run the group's first SNPs one after
// another, so that what depends on (j, k) only is set up once per run.
struct CmpCursor {
    int r;                       // run
    int g_end;                   // one past the group's runs
    int jb_run0;                 // first run of j block jb
    int g, f0, n, f;             // group, its first SNPs (relative to the range), the current one
    int jb, kb;

    __device__ __forceinline__ bool seek(const CmpArgs& a) {
        if (r >= a.n_runs) return false;
        const int nk = (a.cd.pl.M + kTK - 1) / kTK;
        if (r >= g_end) {
            do ++g;
            while (a.groups[g].run_end <= r);
            const CmpGroup& G = a.groups[g];
            g_end = G.run_end;
            f0 = G.f0;
            n = G.n;
            jb = G.b_lo;
            jb_run0 = G.run_end - G.runs;
        }
        while (r - jb_run0 >= nk - 2 * jb) {
            jb_run0 += nk - 2 * jb;
            ++jb;
        }
        kb = 2 * jb + (r - jb_run0);
        f = f0;
        return true;
    }
    __device__ __forceinline__ bool first(const CmpArgs& a) {
        r = blockIdx.x;
        g = -1;
        g_end = 0;
        return seek(a);
    }
    __device__ __forceinline__ bool next(const CmpArgs& a) {
        if (++f < f0 + n) return true;
        r += gridDim.x;
        return seek(a);
    }
};

// A warp's triplets that the bound did not prune, waiting for their exact score: the counted cells
// (count + 1, [8 c + 4 a + 2 b + z]) and the SNPs.  They arrive a few at a time, scattered over
// lanes; queued, a warp scores up to 16 at once.
constexpr int kQueue = 16;
struct CmpQueue {
    float n8[16][kQueue];
    int i[kQueue], j[kQueue], k[kQueue];
    // per lane, set at the first tile of a run: its triplets with k > j in range (bits 2 it + m) and
    // its first (Y, Z) block for the tile's k in lane groups h = 0, 1
    unsigned vmask[32], yz[2][32];
    int n;                       // entries, fewer than kQueue between tiles
    int pad_[3];
};

// One queued triplet's exact tables, its FP32 score (k2_f32's operations in its order) and, if that
// is inside the threshold, its place in the candidate buffer.  One genotype of the first SNP at a
// time (nine cells of both classes: the whole table would cost the epilogue its registers): its
// counted cells, or for the derived genotype the (Y, Z) pair table minus the counted ones, then the
// cells with a 2 from the integer pair tables and marginals, as in derive27.
template <bool kInstr>
__device__ __forceinline__ void cmp_score(const CmpArgs& a, EpiShared& es, const CmpQueue& qu, int at,
                                          unsigned long long* sums) {
    const CohortDev& cd = a.cd;
    const PairTables& pt = cd.pt;
    const int M = cd.pl.M;
    int i = qu.i[at], j = qu.j[at], k = qu.k[at];
    const int drop = __ldg(&a.firsts[i - a.i0].drop);
    float ah = 0.f, al = 0.f;
    unsigned long long hash = 0;
    bool ok = true;
#pragma unroll 1
    for (int g = 0; g < 3; ++g) {
        int r[2][9], t[9];
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            // opaque: keeps the compiler from holding every table entry across the loops
            asm volatile("" : "+r"(i), "+r"(j), "+r"(k));
            const int4* const tab = pt.pt + c * pt.n_pairs;
            const int2* const mg = pt.marg + (size_t)c * M;
            const int4 xy = __ldg(tab + pair_index(i, j)), xz = __ldg(tab + pair_index(i, k));
            const int2 mx = __ldg(mg + i), my = __ldg(mg + j), mz = __ldg(mg + k);
            int n[4];    // (g, b, z), index 2 b + z
            const float* const q0 = &qu.n8[8 * c][at];
            if (g == drop) {
                const int4 yz = __ldg(tab + pair_index(j, k));
                const int y[4] = {yz.x, yz.y, yz.z, yz.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) n[e] = y[e] - ((int)q0[kQueue * e] - 1) - ((int)q0[kQueue * (4 + e)] - 1);
            } else {
                const float* const q = q0 + kQueue * 4 * (g > drop ? g - 1 : g);
#pragma unroll
                for (int e = 0; e < 4; ++e) n[e] = (int)q[kQueue * e] - 1;
            }
            const int xy0 = g == 0 ? xy.x : g == 1 ? xy.z : my.x - xy.x - xy.z;     // (g, Y = 0), (g, Y = 1)
            const int xy1 = g == 0 ? xy.y : g == 1 ? xy.w : my.y - xy.y - xy.w;
            const int xz0 = g == 0 ? xz.x : g == 1 ? xz.z : mz.x - xz.x - xz.z;
            const int xz1 = g == 0 ? xz.y : g == 1 ? xz.w : mz.y - xz.y - xz.w;
            const int mg_ = g == 0 ? mx.x : g == 1 ? mx.y : (c ? pt.n_c[1] : pt.n_c[0]) - mx.x - mx.y;
            t[0] = n[0];
            t[1] = n[1];
            t[2] = xy0 - n[0] - n[1];
            t[3] = n[2];
            t[4] = n[3];
            t[5] = xy1 - n[2] - n[3];
            t[6] = xz0 - n[0] - n[2];
            t[7] = xz1 - n[1] - n[3];
            t[8] = (mg_ - xy0 - xy1) - t[6] - t[7];
#pragma unroll
            for (int e = 0; e < 9; ++e) {
                ok = ok && (unsigned)t[e] <= (unsigned)(c ? pt.n_c[1] : pt.n_c[0]);
                if (c == 0) r[0][e] = t[e];
                else r[1][e] = t[e];
            }
        }
        if (!ok) break;
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const float2 s = __ldg(cd.k2.lf2 + r[0][e] + r[1][e] + 1), u = __ldg(cd.k2.lf2 + r[0][e]),
                         w = __ldg(cd.k2.lf2 + r[1][e]);
            ah += __fsub_rn(__fsub_rn(s.x, u.x), w.x);
            al += __fsub_rn(__fsub_rn(s.y, u.y), w.y);
            if (kInstr) hash = table_fold(hash, r[0][e], r[1][e]);
        }
    }
    if (!ok) {
        atomicOr(&cd.ctrl->status, kStBadCount);
        return;
    }
    const float sc = __fadd_rn(ah, al);
    if (cd.dbg) cd.dbg[((size_t)i * M + j) * M + k] = sc;
    if (kInstr && cd.tsum) {
        sums[0] += table_mix(hash, i, j, k);
        ++sums[1];
    }
    const float thr_g = __uint_as_float(*(volatile unsigned*)&cd.ctrl->thr);
    if (sc <= fminf(*(volatile float*)&es.tloc, thr_g)) {
        const int idx = atomicAdd(&es.cnt, 1);
        if (idx < kCandCap) es.buf[idx] = Cand{sc, i, j, k};
        else cand_global(cd, Cand{sc, i, j, k});
    }
}

// A warp's surviving triplets of an item (mask: bit m, triplet (i, j, k0 + m)) go to its queue, their
// counted cells read from tensor memory again (t: the item's four sets); before it would overflow, the
// queue is scored.  Called by a whole warp; with no survivors at all (mask 0 in every lane) it scores
// what is left.
struct CmpItems {
    uint32_t t[4];
    int i, j, k0;
    unsigned mask;
};
template <bool kInstr>
__device__ __forceinline__ void cmp_survivors(const CmpArgs& a, EpiShared& es, CmpQueue& qu, const CmpItems x,
                                           unsigned long long* sums) {
    const CohortDev& cd = a.cd;
    const int lane = threadIdx.x & 31, i = x.i, j = x.j, M = cd.pl.M;
    const long long pij = j > i && j < M ? pair_index(i, j) : -1;
    const bool row = pij >= 0 && pij >= cd.pair_begin && pij < cd.pair_end;
    int n = qu.n;
    const bool flush = !__any_sync(0xffffffffu, x.mask != 0u);
#pragma unroll 1
    for (int m = flush ? 1 : 0; m < 2; ++m) {
        const int k = x.k0 + m;
        bool want = row && ((x.mask >> m) & 1u) && k > j && k < M;
        unsigned who = __ballot_sync(0xffffffffu, want);
#pragma unroll 1
        while (who || flush) {
            const int at = n + __popc(who & ((1u << lane) - 1u));
            const bool take = want && at < kQueue;
            if (who) {
                float v[4][8];
#pragma unroll
                for (int q = 0; q < 4; ++q) tc_ld16x2(x.t[q], v[q]);
                tc_wait_ld4(v);
                if (take) {
#pragma unroll
                    for (int e = 0; e < 16; ++e) {   // register 4 z + 2 b + m of set (c, a)
                        const int r = 4 * (e & 1) + 2 * ((e >> 1) & 1);
                        qu.n8[e][at] = m ? v[e >> 2][r + 1] : v[e >> 2][r];
                    }
                    qu.i[at] = i;
                    qu.j[at] = j;
                    qu.k[at] = k;
                }
                n = min(n + __popc(who), kQueue);
                want = want && !take;
                who = __ballot_sync(0xffffffffu, want);
            }
            if (n == kQueue || flush) {
                __syncwarp();
                if (lane < n) cmp_score<kInstr>(a, es, qu, lane, sums);
                __syncwarp();
                n = 0;
                if (flush) break;
            }
        }
    }
    __syncwarp();
    if (lane == 0) qu.n = n;
    __syncwarp();
}

// The bound of one lane's two triplets of an item (L = LaneOps2), or of one of them (LaneOps1): the sum
// of um^2 / us and of lg2 us over the cells, us and um the cell's u in tables s and m (cmp_bound_terms).
// Two cells a, b share a denominator that is also their factor of the product:
//     um_a^2 / us_a + um_b^2 / us_b = (um_a^2 us_b + um_b^2 us_a) / (us_a us_b),
// six FP32 operations, and two such pairs share a reciprocal (a reciprocal holds its pipe for 8 cycles
// a warp, a product the FP32 pipe for 2).  The nine cells of a phase go through each operation
// together: one after the other, every operation would wait for the one before it.  (The us of nine
// cells sum to at most N + 54: at the 131072 samples a handle takes their product is at most 3.0e37.)
template <class L>
struct CmpBound {
    typedef typename L::T T;
    T sum[2], lgs;
    __device__ __forceinline__ void init() { sum[0] = sum[1] = lgs = L::dup(0.f); }
    __device__ __forceinline__ void phase(const T (&us)[9], const T (&um)[9]) {
        T w[5], r[5], n[9];
#pragma unroll
        for (int e = 0; e < 4; ++e) w[e] = L::mul(us[2 * e], us[2 * e + 1]);
        w[4] = us[8];
        const T p0 = L::mul(w[0], w[1]), p1 = L::mul(w[2], w[3]);
        const T q0 = L::rcp(p0), q1 = L::rcp(p1);
        r[4] = L::rcp(w[4]);
        const T all = L::mul(L::mul(p0, p1), w[4]);
#pragma unroll
        for (int e = 0; e < 9; ++e) n[e] = L::mul(um[e], um[e]);
#pragma unroll
        for (int e = 0; e < 4; ++e) n[2 * e] = L::mul(n[2 * e], us[2 * e + 1]);
#pragma unroll
        for (int e = 0; e < 4; ++e) n[2 * e] = L::fma(n[2 * e + 1], us[2 * e], n[2 * e]);
        r[0] = L::mul(q0, w[1]);
        r[1] = L::mul(q0, w[0]);
        r[2] = L::mul(q1, w[3]);
        r[3] = L::mul(q1, w[2]);
#pragma unroll
        for (int e = 0; e < 5; ++e) sum[e & 1] = L::fma(n[2 * e], r[e], sum[e & 1]);
        lgs = L::add(lgs, L::lg(all));
    }
};

// Shared memory from the 1024-byte aligned base on: operand ring, staged rows, survivor queues,
// candidate buffer, barriers.
constexpr int kBarBytes = 256;
constexpr size_t kOffB = (size_t)kSlots * kSlotA;
constexpr size_t kOffStage = kOffB + (size_t)kSlots * kSlotB;
constexpr size_t kOffQueue = kOffStage + 2 * sizeof(CmpStage);
constexpr size_t kOffYz = kOffQueue + kCmpEpiWarps * sizeof(CmpQueue);   // float4 [warp][4][32]
constexpr size_t kOffEpi = kOffYz + (size_t)kCmpEpiWarps * 4 * 32 * sizeof(float4);
constexpr size_t kOffBars = (kOffEpi + sizeof(EpiShared) + 15) & ~(size_t)15;
constexpr size_t kCmpSmem = kOffBars + kBarBytes;
static_assert(1024 + kCmpSmem <= 232448, "shared memory of one CTA");
static_assert(kOffStage % 16 == 0 && kOffQueue % 16 == 0 && kOffYz % 16 == 0 && kOffEpi % 16 == 0,
              "alignment");

// kInstr: the instrumented instantiation (table checksums; with a.prof, per role the cycles spent
// waiting, summed over CTAs: [0] loader on free slots, [1] MMA issuer on loaded slots, [2] MMA
// issuer on free accumulator regions, [4] epilogue thread 0 on finished tiles, [5] kernel cycles,
// [7] MMA issuer issuing MMAs and commits).
// kPaired: the epilogue takes the bound of a lane's two triplets together in f32x2 instructions
// (half the instructions of the one-at-a-time form).
template <bool kInstr, bool kPaired>
__global__ void __launch_bounds__(kCmpThreads, 1) scan_cmp_kernel(const __grid_constant__ CmpArgs a) {
    const long long t_start = kInstr ? clock64() : 0;
    unsigned long long* const prof = kInstr ? a.prof : nullptr;
    unsigned long long w_acc = 0, w_acc2 = 0, w_acc3 = 0;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint8_t* sA = base;                                 // [kSlots][kSlotSteps][16 KB] rows (j, b)
    uint8_t* sB = base + kOffB;                         // [kSlots][kSlotSteps][8 KB] rows (k, z)
    CmpStage* const stage = reinterpret_cast<CmpStage*>(base + kOffStage);   // [2]
    CmpQueue* const queues = reinterpret_cast<CmpQueue*>(base + kOffQueue);  // one per epilogue warp
    EpiShared& es = *reinterpret_cast<EpiShared*>(base + kOffEpi);
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + kOffBars);
    // bars: fullS[kSlots], emptyS[kSlots], accF[2], rowF[2], rowE[2], regE[kCmpRegions], drain
    constexpr int kNBars = 2 * kSlots + 6 + kCmpRegions + 1;
    static_assert(kNBars * 8 + 12 <= kBarBytes, "barrier area");
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kNBars);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const uint32_t fullS0 = smem_u32(bars), emptyS0 = smem_u32(bars + kSlots),
                   accF0 = smem_u32(bars + 2 * kSlots), rowF0 = accF0 + 16, rowE0 = rowF0 + 16,
                   regE0 = rowE0 + 16, drain0 = regE0 + 8 * kCmpRegions;
    const CohortDev& cd = a.cd;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kSlots; ++s) {
            mbar_init(fullS0 + 8 * s, 1);
            mbar_init(emptyS0 + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accF0 + 8 * b, 1);
            mbar_init(rowF0 + 8 * b, 2);
            mbar_init(rowE0 + 8 * b, kCmpEpiWarps);
        }
        for (int r = 0; r < kCmpRegions; ++r) mbar_init(regE0 + 8 * r, kCmpEpiWarps);
        mbar_init(drain0, 1);
        *abort_flag = 0;
        es.cnt = 0;
        for (int w = 0; w < kCmpEpiWarps; ++w) queues[w].n = 0;
        es.tloc = __int_as_float(0x7f800000);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (warp < 4) {  // block scale factors 2^0 (UE8M0 127) in every byte of the scale columns
        uint32_t one[32];
#pragma unroll
        for (int t = 0; t < 32; ++t) one[t] = 0x7F7F7F7Fu;
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
            "%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
            ::"r"(tmem + ((uint32_t)(32 * warp) << 16) + kCmpSfCol), "r"(one[0]), "r"(one[1]),
              "r"(one[2]), "r"(one[3]), "r"(one[4]), "r"(one[5]), "r"(one[6]), "r"(one[7]),
              "r"(one[8]), "r"(one[9]), "r"(one[10]), "r"(one[11]), "r"(one[12]), "r"(one[13]),
              "r"(one[14]), "r"(one[15]), "r"(one[16]), "r"(one[17]), "r"(one[18]), "r"(one[19]),
              "r"(one[20]), "r"(one[21]), "r"(one[22]), "r"(one[23]), "r"(one[24]), "r"(one[25]),
              "r"(one[26]), "r"(one[27]), "r"(one[28]), "r"(one[29]), "r"(one[30]), "r"(one[31])
            : "memory");
        tc_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    // role: 1 loader (on a free slot), 2 MMA issuer (region), 3 MMA issuer (operands),
    // 4 epilogue (accumulators), 5 the timeout test hook, 6 stager (free buffer), 7 epilogue
    // (staged rows)
    auto fail_at = [&](unsigned role, long long tl, int q, int ks, unsigned extra = 0u) {
        *abort_flag = 1;
        if (atomicCAS(&cd.ctrl->wait_role, 0u, role) == 0u) {
            cd.ctrl->wait_tile = (unsigned)tl;
            cd.ctrl->wait_set = (unsigned)q;
            cd.ctrl->wait_step = (unsigned)ks;
            cd.ctrl->pad_[0] = extra;
        }
        atomicOr(&cd.ctrl->status, kStTimeout);
    };

    // The loader (warp 0), the MMA issuer (warp 1) and the stagers run as whole warps with
    // warp-uniform control flow; one elected lane issues each copy, MMA and commit.  Values read
    // from memory are broadcast by shuffles so that every operand is provably uniform; a tile's
    // sizes are fetched one tile ahead (lanes 0..3, one set each).
    if (warp < kCmpEpiWarp0) {
    if (warp == 0) {
        // ------------------------------------------------ operand loader
        static_assert(kSlotSteps == 2, "load_slot_elect");
        const uint32_t sA0 = smem_u32(sA), sB0 = smem_u32(sB);
        Ring rs{0, 0u};
        uint32_t used = 0, fph = 0;
        bool stop = false;
        CmpCursor cu;
        bool have = cu.first(a);
        int ks_n = 0, blo_n = 0;
        long long base_n = 0;
        auto fetch = [&](int f) {
            ks_n = a.firsts[f].ks[lane & 3];
            base_n = a.firsts[f].base[lane & 3];
            blo_n = a.firsts[f].b_lo;
        };
        if (have) fetch(cu.f);
        for (long long tl = 0; have && !stop; ++tl) {
            const int ks_l = ks_n, b_lo = warp_uniform(blo_n);
            const long long base_l = base_n;
            const int jb = warp_uniform(cu.jb), kb = warp_uniform(cu.kb);
            have = cu.next(a);
            if (have) fetch(cu.f);
            for (int q = 0; q < kCmpSets && !stop; ++q) {
                const int KS = __shfl_sync(0xffffffffu, ks_l, q);
                const long long base_q = __shfl_sync(0xffffffffu, base_l, q);
                const uint8_t* pa = a.cmp + (size_t)(base_q + (long long)(jb - b_lo) * KS) * kCmpChunk;
                const uint8_t* pb = a.cmp + (size_t)(base_q + (long long)((kb >> 1) - b_lo) * KS) * kCmpChunk +
                                    (size_t)(kb & 1) * kStepB;
                for (int ks = 0; ks < KS; ks += kSlotSteps) {
                    // a slot takes up to kSlotSteps consecutive steps of one set: their A
                    // chunks are adjacent (one copy), their B halves are not
                    const int n = min(kSlotSteps, KS - ks);
                    const int s = rs.s;
                    const bool got = mbar_wait_t(emptyS0 + 8 * s, rs.ph ^ 1u, abort_flag,
                                                 (prof && lane == 0) ? &w_acc : nullptr);
                    if (!__all_sync(0xffffffffu, got)) {
                        if (lane == 0) fail_at(1, tl, q, ks, (unsigned)s | (rs.ph << 8));
                        stop = true;
                        break;
                    }
                    load_slot_elect(fullS0 + 8 * s, sA0 + (uint32_t)(s * kSlotA), pa, (uint32_t)(n * kStepA),
                                    sB0 + (uint32_t)(s * kSlotB), pb, n > 1 ? 1u : 0u);
                    pa += (size_t)kSlotSteps * kCmpChunk;
                    pb += (size_t)kSlotSteps * kCmpChunk;
                    used |= 1u << s;
                    fph ^= 1u << s;
                    ring_next(rs, kSlots);
                }
            }
        }
        // drain: the copies issued must land before the CTA exits
        for (int b = 0; b < kSlots; ++b) {
            if (!((used >> b) & 1u)) continue;
            volatile int no_abort = 0;
            mbar_wait(fullS0 + 8 * b, ((fph >> b) & 1u) ^ 1u, &no_abort);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        bool ok = true;
        if (cd.inject_timeout) {  // test hook: a wait that can only run out (about 1 s)
            const bool got = mbar_wait(drain0, 0, abort_flag);
            if (!__all_sync(0xffffffffu, got) && lane == 0) fail_at(5, 0, 0, 0);
            ok = false;
        }
        Ring rR{0, 0u}, rs{0, 0u};
        const uint64_t da0 = sw128_desc(smem_u32(sA)), db0 = sw128_desc(smem_u32(sB));
        CmpCursor cu;
        bool have = cu.first(a);
        int ks_n = have ? a.firsts[cu.f].ks[lane & 3] : 0;
        for (long long tl = 0; have && ok; ++tl) {
            const int ks_l = ks_n;
            have = cu.next(a);
            if (have) ks_n = a.firsts[cu.f].ks[lane & 3];
            for (int q = 0; q < kCmpSets && ok; ++q) {
                const bool freed = mbar_wait_t(regE0 + 8 * rR.s, rR.ph ^ 1u, abort_flag,
                                               (prof && lane == 0) ? &w_acc2 : nullptr);
                if (!__all_sync(0xffffffffu, freed)) {
                    if (lane == 0) fail_at(2, tl, q, 0);
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(rR.s * kN);
                ring_next(rR, kCmpRegions);
                const int KS = __shfl_sync(0xffffffffu, ks_l, q);
                for (int ks = 0; ks < KS; ks += kSlotSteps) {
                    const int n = min(kSlotSteps, KS - ks);
                    const int s = rs.s;
                    const bool got = mbar_wait_t(fullS0 + 8 * s, rs.ph, abort_flag,
                                                 (prof && lane == 0) ? &w_acc : nullptr);
                    if (!__all_sync(0xffffffffu, got)) {
                        if (lane == 0) fail_at(3, tl, q, ks, (unsigned)s | (rs.ph << 8));
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const long long t_issue = prof ? clock64() : 0;
                    const uint64_t da = da0 + (uint32_t)(s * (kSlotA >> 4)), db = db0 + (uint32_t)(s * (kSlotB >> 4));
                    mma_step_elect(d, da, db, (uint32_t)ks, tmem + kCmpSfCol, tmem + kCmpSfCol + 16);
                    if (n > 1)
                        mma_step_elect(d, da + (kStepA >> 4), db + (kStepB >> 4), 1u, tmem + kCmpSfCol,
                                       tmem + kCmpSfCol + 16);
                    tc_commit_elect(emptyS0 + 8 * s);  // the slot is free once these MMAs complete
                    if (prof) w_acc3 += (unsigned long long)(clock64() - t_issue);
                    ring_next(rs, kSlots);
                }
            }
            if (ok) tc_commit_elect(accF0 + 8 * (int)(tl & 1));
        }
        // every MMA issued must complete before tensor memory is released
        tc_commit_elect(drain0);
        volatile int no_abort = 0;
        mbar_wait(drain0, 0, &no_abort);
        __syncwarp();
    } else {
        // ------------------------------------------------ stagers (warps 2 and 3)
        // The (i, j) and (i, k) parts of a tile's derived cells, with SNP i's genotypes
        // relabelled, ready as the epilogue's operands: the epilogue warps used to form them per
        // thread from pair-table rows they each loaded from L2.  One j per lane (32 of the tile's
        // 64 to each stager) and one k per lane of the first; the next tile's table entries are
        // fetched while this one's buffer is not free yet.
        const int M = cd.pl.M, half = warp - 2;
        const PairTables& pt = cd.pt;
        const int cm = a.minor;
        const float kInf = __int_as_float(0x7f800000);
        const bool prune_on = !cd.dbg && !(kInstr && cd.tsum);
        CmpCursor cu;
        bool have = cu.first(a);
        int4 nxy[2], nxz[2];
        int2 nmx[2], nmy[2], nmz[2];
        int ndrop = 0;
        auto fetch = [&]() {
            const int i = a.i0 + cu.f, j = kTJ * cu.jb + 32 * half + lane, k = kTK * cu.kb + lane;
            const int jc = j < M && j > i ? j : i + 1, kc = k < M && k > i ? k : i + 1;   // i + 1 < M
            ndrop = a.firsts[cu.f].drop;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int4* const tab = pt.pt + c * pt.n_pairs;
                const int2* const mg = pt.marg + (size_t)c * M;
                nmx[c] = __ldg(mg + i);
                nmy[c] = __ldg(mg + jc);
                nxy[c] = __ldg(tab + pair_index(i, jc));
                if (half == 0) {
                    nmz[c] = __ldg(mg + kc);
                    nxz[c] = __ldg(tab + pair_index(i, kc));
                }
            }
        };
        if (have) fetch();
        for (long long tl = 0; have; ++tl) {
            const int f = cu.f, i = a.i0 + f, jb = cu.jb, kb = cu.kb, drop = ndrop;
            const int fresh = f == cu.f0 ? kStageRun : 0;
            const int j = kTJ * jb + 32 * half + lane;
            const bool in = j < M && j > i;
            const long long pij = in ? pair_index(i, j) : -1;
            int w[2][9];   // [class]: [0..3] xy, [4..5] (a, 2), [6..7] (2, b), [8] (2, 2)
            int wz[2][6];  // [class]: [0..3] xz, [4..5] (2, z)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int2 mx = relabel_marg(nmx[c], pt.n_c[c], drop);
                const int4 p = relabel_xy(nxy[c], nmy[c], drop);
                w[c][0] = p.x;
                w[c][1] = p.y;
                w[c][2] = p.z;
                w[c][3] = p.w;
                w[c][4] = mx.x - p.x - p.y;
                w[c][5] = mx.y - p.z - p.w;
                w[c][6] = nmy[c].x - p.x - p.z;
                w[c][7] = nmy[c].y - p.y - p.w;
                w[c][8] = pt.n_c[c] - mx.x - mx.y - w[c][6] - w[c][7];
                if (half == 0) {
                    const int4 z = relabel_xy(nxz[c], nmz[c], drop);
                    wz[c][0] = z.x;
                    wz[c][1] = z.y;
                    wz[c][2] = z.z;
                    wz[c][3] = z.w;
                    wz[c][4] = nmz[c].x - z.x - z.z;
                    wz[c][5] = nmz[c].y - z.y - z.w;
                }
            }
            have = cu.next(a);
            if (have) fetch();
            const int buf = (int)(tl & 1);
            if (!__all_sync(0xffffffffu, mbar_wait(rowE0 + 8 * buf, (unsigned)((tl >> 1) & 1) ^ 1u,
                                                   abort_flag))) {
                if (lane == 0) fail_at(6, tl, 0, 0);
                break;
            }
            CmpStage& S = stage[buf];
            // a bound above this proves the exact score above the threshold (cmp_bound_terms)
            const float thr = fminf(__uint_as_float(*(volatile unsigned*)&cd.ctrl->thr), *(volatile float*)&es.tloc);
            const float cut = prune_on && thr < kInf ? __fadd_ru(thr, a.bound_off) : kInf;
            constexpr int kOrder[9] = {0, 1, 4, 2, 3, 5, 6, 7, 8};   // phase-major
            float4* const dst = &S.row[32 * half + lane][0][0];
#pragma unroll
            for (int e = 0; e < 9; ++e) {
                const int o = kOrder[e];
                const float s = (float)(w[0][o] + w[1][o] + 6), m = (float)((cm ? w[1][o] : w[0][o]) + 3);
                dst[e] = make_float4(s, s, m, m);
            }
            S.thr[32 * half + lane] = pij >= cd.pair_begin && pij < cd.pair_end ? cut : -kInf;
            if (half == 0) {
                float* const dz = reinterpret_cast<float*>(&S.col[lane >> 1][0][0]) + (lane & 1);
#pragma unroll
                for (int ph = 0; ph < 3; ++ph)
#pragma unroll
                    for (int z = 0; z < 2; ++z) {
                        const int o = 2 * ph + z;
                        dz[2 * (4 * ph + z)] = (float)(wz[0][o] + wz[1][o] + 6);
                        dz[2 * (4 * ph + 2 + z)] = (float)((cm ? wz[1][o] : wz[0][o]) + 3);
                    }
                if (lane == 0) {
                    S.f = f;
                    S.jb = jb;
                    S.kb = kb;
                    S.flags = fresh | (have ? 0 : kStageLast);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(rowF0 + 8 * buf);
        }
        __syncwarp();
    }
    } else {
        // ------------------------------------------------ epilogue
        // Per set (c, a), tensor-memory lane 16 G + 8 b + r holds the counts + 1 of second SNP
        // jl = 8 G + r with genotype b, in column 16 H + 8 z + s for third SNP kl = 8 H + s with
        // genotype z (the chunks' row order).  A 16x256b.x2 load at lane group G, column group H
        // gives thread t the cells (b, z) of jl = 8 G + t / 4 and kl = 8 H + 2 (t % 4) + e,
        // e = 0, 1, in registers 4 z + 2 b + e: all 8 cells of a set for two triplets, the two in
        // neighbouring registers, as the f32x2 instructions take them.  Items of a quadrant: lane
        // groups G = 2 quad + h (h = 0, 1) x column groups H = 0..3; each warp takes two column
        // groups of one h.
        // The bound per triplet: 105 FP32 operations for the 27 cells, 84 additions and subtractions
        // for the 19 derived cells in two tables, 192 lane operations with the last three (3070 cycles
        // a tile at 128 a clock), and 12 reciprocals and logs (1540 at 16 a clock).  The form before,
        // phi(us) - phi(u0) - phi(u1) per cell, took 81 logs, and each thread formed the constants that
        // the stagers now form once a tile.
        const int tid = threadIdx.x - kCmpEpiWarp0 * 32;     // 0 .. 383
        const int quad = warp & 3, part = (warp - kCmpEpiWarp0) >> 2;
        const int jl0 = 16 * quad + (lane >> 2), tcol = 2 * (lane & 3);
        const int M = cd.pl.M;
        const int cm = a.minor;
        const float cq = a.bound_c;
        CmpQueue& qu = queues[warp - kCmpEpiWarp0];
        unsigned long long sums[2] = {0, 0};
        const uint32_t tbase = tmem + ((uint32_t)(32 * quad) << 16);
        int reg0 = 0;            // region of the tile's first set
        bool bad = false, last = (int)blockIdx.x >= a.n_runs;
        int since = 0, interval = 1;
        const int prune_at = min(max(2 * cd.top_k, 32), kPruneAt + 1);
        // An item's (Y, Z) entries come into this lane's slots while the item before is worked on
        // (asynchronous copies: plain loads shared a scoreboard with the shared-memory loads of the
        // constants, and every item waited for L2).
        const float4* const ys = reinterpret_cast<const float4*>(base + kOffYz) +
                                 (size_t)(warp - kCmpEpiWarp0) * 128 + lane;   // [4], 32 apart
        auto fetch = [&](int item) {
            const float4* const src =
                a.yz + 16 * ((size_t)qu.yz[item >> 2][lane] + (item & 3)) + (lane & 3);
#pragma unroll
            for (int e = 0; e < 4; ++e) cp_async16(smem_u32(ys + 32 * e), src + 4 * e);
            cp_async_commit();
        };
        for (unsigned tl = 0; !last; ++tl) {
            // region of set q of this tile
            auto region = [&](int q) { return reg0 + q < kCmpRegions ? reg0 + q : reg0 + q - kCmpRegions; };
            const int buf = (int)(tl & 1);
            if (!bad) {
                const bool got = mbar_wait(rowF0 + 8 * buf, (tl >> 1) & 1u, abort_flag);
                if (!__all_sync(0xffffffffu, got)) {
                    if (lane == 0) fail_at(7, tl, 0, 0);
                    bad = true;
                }
            }
            if (!bad) {
                const CmpStage& S = stage[buf];
                last = (S.flags & kStageLast) != 0;
                if (S.flags & kStageRun) {  // a new run: its (j, k) parts
                    unsigned vmask = 0;
#pragma unroll
                    for (int it = 0; it < kCmpEpiItems; ++it) {
                        const int item = part + kCmpEpiParts * it;
                        const int j = kTJ * S.jb + jl0 + 8 * (item >> 2), k = kTK * S.kb + 8 * (item & 3) + tcol;
                        if (item < 8)
                            vmask |= ((k > j && k < M ? 1u : 0u) | (k + 1 > j && k + 1 < M ? 2u : 0u)) << (2 * it);
                    }
                    qu.vmask[lane] = vmask;
                    // blocks of k <= j or k >= M are other pairs' or padding: masked
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        qu.yz[h][lane] = (unsigned)yz_block(min(kTJ * S.jb + jl0 + 8 * h, M - 1), kTK * S.kb, M);
                    cp_async_wait();   // the last run's prefetch
                    fetch(part);
                }
                const bool got = mbar_wait_t(accF0 + 8 * buf, (tl >> 1) & 1u, abort_flag,
                                             (prof && tid == 0) ? &w_acc : nullptr);
                if (!__all_sync(0xffffffffu, got)) {
                    if (lane == 0) fail_at(4, tl, 0, 0);
                    bad = true;
                }
            }
            if (!bad) {
                tc_fence_after();
                const CmpStage& S = stage[buf];
                const unsigned vmask_all = qu.vmask[lane];
#pragma unroll 1
                for (int it = 0; it < kCmpEpiItems; ++it) {
                    const int item = part + kCmpEpiParts * it, jl = jl0 + 8 * (item >> 2);
                    const unsigned vmask = (vmask_all >> (2 * it)) & 3u;
                    if (item >= 8) break;
                    const int next = item + kCmpEpiParts < 8 ? item + kCmpEpiParts : part;
                    if (!__any_sync(0xffffffffu, vmask)) {   // k <= j throughout
                        cp_async_wait();
                        fetch(next);
                        continue;
                    }
                    const float cut = S.thr[jl];
                    const float4* const row = &S.row[jl][0][0];
                    const float4* const col =
                        reinterpret_cast<const float4*>(&S.col[4 * (item & 3) + (lane & 3)][0][0]);
                    const uint32_t tb = tbase + (uint32_t)(16 * (item & 3)) + ((uint32_t)(item & 4) << 18);
                    unsigned sv = 0;
#pragma unroll
                    for (int pass = 0; pass < (kPaired ? 1 : 2); ++pass) {
                        typedef typename std::conditional<kPaired, LaneOps2, LaneOps1>::type L;
                        typedef typename L::T T;
                        CmpBound<L> B;
                        B.init();
                        float v[2][8];    // one counted genotype's cells: the larger class, the smaller
                        auto load = [&](int ph) {
                            tc_ld16x2(tb + (uint32_t)(region(2 * (cm ^ 1) + ph) * kN), v[0]);
                            tc_ld16x2(tb + (uint32_t)(region(2 * cm + ph) * kN), v[1]);
                        };
                        float4 cs, cmn, r0, r1, r2;   // a phase's constants
                        auto constants = [&](int ph) {
                            lds128(cs, col + 2 * ph);
                            lds128(cmn, col + 2 * ph + 1);
                            lds128(r0, row + 3 * ph);
                            lds128(r1, row + 3 * ph + 1);
                            lds128(r2, row + 3 * ph + 2);
                        };
                        constants(0);
                        T ds[4], dm[4];   // cells (2, b, z): the (Y, Z) table minus the counted genotypes
#pragma unroll
                        for (int ph = 0; ph < 3; ++ph) {
                            if (ph < 2) load(ph);
                            T us[4], um[4];   // cells (b, z) of this first-SNP genotype, index 2 b + z
                            float4 y4[4];
                            if (ph == 2) {
                                if (pass == 0) cp_async_wait();
#pragma unroll
                                for (int e = 0; e < 4; ++e) y4[e] = ys[32 * e];
                            }
                            if (ph < 2) tc_wait_ld2(v);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                if (ph < 2) {
                                    const int w = 4 * (e & 1) + 2 * (e >> 1);
                                    const T c0 = L::pick(make_float2(v[0][w], v[0][w + 1]), pass);
                                    const T c1 = L::pick(make_float2(v[1][w], v[1][w + 1]), pass);
                                    us[e] = L::add(c0, c1);
                                    um[e] = c1;
                                    ds[e] = ph ? L::add(ds[e], us[e]) : us[e];
                                    dm[e] = ph ? L::add(dm[e], um[e]) : um[e];
                                } else {
                                    const float4 ys = y4[e >> 1], ym = y4[2 + (e >> 1)];
                                    us[e] = L::sub(L::pick(e & 1 ? make_float2(ys.z, ys.w) : make_float2(ys.x, ys.y), pass), ds[e]);
                                    um[e] = L::sub(L::pick(e & 1 ? make_float2(ym.z, ym.w) : make_float2(ym.x, ym.y), pass), dm[e]);
                                }
                            }
                            const T cst[9] = {us[0], us[1], us[2], us[3], L::two(r0.x, r0.y), L::two(r1.x, r1.y),
                                              L::pick(make_float2(cs.x, cs.y), pass),
                                              L::pick(make_float2(cs.z, cs.w), pass), L::two(r2.x, r2.y)};
                            const T cmt[9] = {um[0], um[1], um[2], um[3], L::two(r0.z, r0.w), L::two(r1.z, r1.w),
                                              L::pick(make_float2(cmn.x, cmn.y), pass),
                                              L::pick(make_float2(cmn.z, cmn.w), pass), L::two(r2.z, r2.w)};
                            T s9[9], m9[9];   // (., b, z), (., 0, 2), (., 1, 2), (., 2, 0), (., 2, 1), (., 2, 2)
#pragma unroll
                            for (int e = 0; e < 9; ++e) {
                                s9[e] = cst[e];
                                m9[e] = cmt[e];
                            }
                            constexpr int kSub[8] = {0, 2, 0, 1, 1, 3, 2, 3};   // first and second minuend's partner
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                s9[4 + e] = L::sub(s9[4 + e], us[kSub[e]]);
                                m9[4 + e] = L::sub(m9[4 + e], um[kSub[e]]);
                            }
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                s9[4 + e] = L::sub(s9[4 + e], us[kSub[4 + e]]);
                                m9[4 + e] = L::sub(m9[4 + e], um[kSub[4 + e]]);
                            }
                            s9[8] = L::sub(L::sub(s9[8], s9[6]), s9[7]);
                            m9[8] = L::sub(L::sub(m9[8], m9[6]), m9[7]);
                            if (ph == 2 && (kPaired || pass == 1)) fetch(next);
                            if (ph < 2) constants(ph + 1);
                            B.phase(s9, m9);
                        }
                        // ln 2 / 2 (sum of lg2 us) - c (sum of um^2 / us) against the cut
                        const T b = L::fma(L::dup(-cq), L::add(B.sum[0], B.sum[1]), L::mul(L::dup(0.34657359f), B.lgs));
                        if constexpr (kPaired) sv = (b.x > cut ? 0u : 1u) | (b.y > cut ? 0u : 2u);
                        else sv |= (b > cut ? 0u : 1u) << pass;
                    }
                    sv &= vmask;
                    if (__any_sync(0xffffffffu, sv != 0u)) {
                        CmpItems x;
#pragma unroll
                        for (int q = 0; q < kCmpSets; ++q) x.t[q] = tb + (uint32_t)(region(q) * kN);
                        x.i = a.i0 + S.f;
                        x.j = kTJ * S.jb + jl;
                        x.k0 = kTK * S.kb + 8 * (item & 3) + tcol;
                        x.mask = sv;
                        cmp_survivors<kInstr>(a, es, qu, x, kInstr ? sums : nullptr);
                    }
                }
                // accumulators and staged rows read: back to the MMA issuer and the stager
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
#pragma unroll
                    for (int q = 0; q < kCmpSets; ++q) mbar_arrive(regE0 + 8 * region(q));
                    mbar_arrive(rowE0 + 8 * buf);
                }
            }
            reg0 = region(kCmpSets);
            if (++since < interval && !last) continue;
            // rendezvous of the epilogue warps: agree on a stop, and cut the candidate buffer to
            // this CTA's best once it holds twice as many (which lowers the threshold).  It comes
            // less often while few candidates arrive: the schedule is the same for every warp,
            // since it depends on a count read between two barriers.
            if (epi_sync_or<kCmpEpiThreads>(bad || *abort_flag)) break;
            const int cnt = min(*(volatile int*)&es.cnt, kCandCap);
            epi_sync<kCmpEpiThreads>();
            interval = cnt >= prune_at ? 1 : min(kMaxSyncTiles, 2 * interval);
            since = 0;
            if (cnt >= prune_at) {
                const int kept = epi_prune<kCmpEpiThreads>(cd, es, cnt, tid, false);
                if (tid == 0) es.cnt = kept;
                epi_sync<kCmpEpiThreads>();
            }
        }
        {   // what is left in this warp's queue
            CmpItems x{};
            cmp_survivors<kInstr>(a, es, qu, x, kInstr ? sums : nullptr);
        }
        epi_sync<kCmpEpiThreads>();
        epi_prune<kCmpEpiThreads>(cd, es, min(es.cnt, kCandCap), tid, true);
        if (kInstr && cd.tsum) table_sum_flush(cd.tsum, sums[0], sums[1]);
    }
    if (prof) {
        if (warp == 0 && lane == 0) atomicAdd(prof + 0, w_acc);
        if (warp == 1 && lane == 0) {
            atomicAdd(prof + 1, w_acc);
            atomicAdd(prof + 2, w_acc2);
            atomicAdd(prof + 7, w_acc3);
        }
        if (threadIdx.x == kCmpEpiWarp0 * 32) {
            atomicAdd(prof + 4, w_acc);
            atomicAdd(prof + 5, (unsigned long long)(clock64() - t_start));
        }
    }
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                     : "memory");
    }
}

}  // namespace

size_t scan_cmp_smem() { return 1024 + kCmpSmem; }   // the base is aligned to 1024 bytes
int scan_cmp_threads() { return kCmpThreads; }

int cmp_tiles_of(int M, int b_lo, int jb_end) {
    const int nb = std::min((M + 63) / 64, jb_end), nk = (M + kTK - 1) / kTK;
    int t = 0;
    for (int jb = b_lo; jb < nb; ++jb) t += nk - 2 * jb;
    return t;
}

size_t sample_rows_bytes(const Planes& pl) {
    return (size_t)((pl.M + 63) / 64) * 128 * (size_t)(pl.W4[0] + pl.W4[1]) * sizeof(uint4);
}

cudaError_t launch_sample_rows(const Planes& pl, uint4* rows, cudaStream_t st) {
    const int nblk = (pl.M + 63) / 64;
    const long long warps = 4LL * (pl.W4[0] + pl.W4[1]) * nblk, blocks = (warps + 7) / 8;
    sample_rows_kernel<<<(unsigned)std::min<long long>(blocks, 65535), 256, 0, st>>>(pl, nblk, rows);
    return cudaGetLastError();
}

cudaError_t launch_compact(const Planes& pl, const uint4* rows, const CmpFirst* firsts, int i0, int n_first,
                           int n0, int n, uint32_t* list, uint8_t* cmp, cudaStream_t st) {
    if (n_first == 0) return cudaSuccess;
    sample_list_kernel<<<dim3(n_first, 2), 256, 0, st>>>(pl, firsts, i0, n0, n, list);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const dim3 grid((pl.M + 63) / 64, n_first, 2);
    compact_kernel<<<grid, kCompactThreads, 0, st>>>(rows, 4 * pl.W4[0], 4 * (pl.W4[0] + pl.W4[1]), firsts, list,
                                                     n0, n, cmp);
    return cudaGetLastError();
}

template <bool kInstr, bool kPaired>
static cudaError_t launch_cmp_variant(const CmpArgs& a, int grid, cudaStream_t st) {
    const size_t smem = scan_cmp_smem();
    // once per device: allow the dynamic shared memory
    static std::atomic<unsigned long long> ready{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(ready.load(std::memory_order_acquire) & bit)) {
        e = cudaFuncSetAttribute(scan_cmp_kernel<kInstr, kPaired>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem);
        if (e != cudaSuccess) return e;
        ready.fetch_or(bit, std::memory_order_release);
    }
    if (a.n_runs == 0) return cudaSuccess;
    scan_cmp_kernel<kInstr, kPaired><<<grid, kCmpThreads, smem, st>>>(a);
    return cudaGetLastError();
}

// The instrumented instantiation serves table checksums and wait profiles only, so the product
// kernel carries no hook.
cudaError_t launch_scan_cmp(const CmpArgs& a, int grid, cudaStream_t st, bool instrumented, bool paired) {
    if (paired)
        return instrumented ? launch_cmp_variant<true, true>(a, grid, st)
                            : launch_cmp_variant<false, true>(a, grid, st);
    return instrumented ? launch_cmp_variant<true, false>(a, grid, st)
                        : launch_cmp_variant<false, false>(a, grid, st);
}

}  // namespace epi3
