// Dual-trit-plane layer for up to 64 activation rows per launch on packed formats 3 and 2, on the fifth-generation tensor cores
// (tcgen05.mma, operand A and accumulators in tensor memory):
//     Y[m] = alpha1 (.) (T1 X[m]) + alpha2 (.) (T2 X[m]),   m < M <= 64.
//
// A CTA owns up to 128 weight rows (8 tiles per superblock, contiguous in the blob); a row is a lane of every MMA.  Per scale group
// of 128 columns two fp32 accumulators, one per plane, of 128 x NPAD: 16 MMAs of 128 x NPAD x 16.  27 warps in five roles meet on
// mbarriers alone:
//   * 16 warps decode: a shift and a mask of a code word make two trits (times 2) of operand A, 16 instructions per 16 trits, stored
//     straight to tensor memory (tcgen05.st 16x256b, whose fragment is a k-step of four lanes x four columns, what a code word holds).
//     Each of the four warpgroups takes a quarter of a superblock's half-groups (64 columns, both planes); the stages of trits hold three
//     and a half groups at 16 rows, two at 64.
//   * one warp issues the MMAs; one poll by four of its lanes covers all that a group waits for.
//   * 8 warps read the accumulators (tcgen05.ld), two sets of them in turn: y += alpha1 d1 + alpha2 d2 in fp32, half of the
//     columns each.
//   * one warp copies the codes (bulk copies, a superblock at a time, four barriers so that the first quarter can start alone), one the
//     activations (TMA, 128-byte swizzle, rows past M as zeros), fp16 as given.
// Format 2 differs in the copies and in where a word lies: two tensor maps for the code bytes and two for the scale quads (full slices, the last
// slice) bring the same 512 columns of 128 rows by TMA, as lines of 128 bytes [atom][row pair] whose swizzle spreads the eight row
// pairs that a warp reads over the banks (14336 x 4096 with a workspace at 16, 32, 64 rows: 16.1, 17.9, 21.0 us; before 23.0, 41.1, 74.3).
// Matrices with few rows split K over a cluster of up to 8 CTAs; every rank copies its partial sums (bulk copies between the
// shared memories, counted on the receiver's mbarrier) to the rank that owns the columns, which adds them in rank order: no
// atomics, no workspace, reproducible.
//
// What bounds it, from clock stamps in a copy of the kernel: at 64 rows the tensor pipe for two thirds of the time (37 cycles per MMA with A
// from tensor memory, 600 a group, of about 900; the rest is not accounted for: a decoding warpgroup has one of the four stages of
// trits there and cannot work ahead), at 16 rows the issue slots of the SM (670 cycles a group, 330 of them MMAs; by the counters 528
// instructions per group and scheduler, start and end of the launch among them, three of four slots of the SMs that have a CTA; 260 of
// them are the shifts, masks and stores of decoding, the others, loads, sums, polls and the issuing warp, have not been told apart);
// 3.5 us of a launch are start (first codes and activations 2 us after the wait) and end.  Measured in a chain at level 0, microseconds (14336 x 4096, 4096 x 14336, 4096 x 4096,
// 1024 x 4096), in brackets the kernel before it (trits by byte permutes and FMAs, activations by cp.async, decoding, sums and fetch in
// the same warps): 64 rows 20.0, 20.0, 10.2, 7.4 (50.0, 43.3, 17.1, 11.3), 48 rows 18.3, 18.4, 9.1, 6.5 (40.5, 36.8, 14.4, 10.1), 32
// rows 16.8, 16.6, 8.2, 5.8 (35.9, 32.8, 12.9, 9.0), 16 rows 15.1, 15.0, 7.4, 5.2 (30.7, 28.2, 11.4, 7.9).
// What it took: activations by TMA (with cp.async four fetching warps needed 2500 cycles to issue a group of 64 rows: 37.7 us on 14336
// x 4096), one issuing warp with few instructions, partial sums by bulk copies (loads from the ranks' shared memory took 4500 cycles
// with eight ranks, st.async of 8 bytes 5000 at 64 rows), one compact loop for the output.  Without effect or slower:
// multiplications for the shifts, the next words loaded ahead, four sets of accumulators, one commit per group, rolled loops, seven
// tiles per CTA on 128 SMs.
//
// Precision, the rounding of y taken out (512 x 4096 and the groups that cancel the result; in brackets the kernel before it with as
// many CTAs per row block): normal x 0.82e-7 and 0.73e-7 at 16 and 32 rows as the library chooses (warp MMAs 0.82e-7, 0.84e-7), one
// CTA per row block 1.09e-7 (1.44e-7), four 0.80e-7 at 16, 0.94e-7 at 64 rows (0.94e-7, 1.17e-7); x of mean 4 0.80e-7, 1.12e-7,
// 0.79e-7 (0.80e-7, 1.45e-7, 0.91e-7); x over 24 powers of two 1.98e-7, 2.12e-7, 1.99e-7 (1.98e-7, 2.32e-7, 2.07e-7).
//
// Launched as a dependent of the kernel before it on the stream: set-up before griddepcontrol.wait, and on format 3 a prefetch of the
// first codes into L2, the point of coherence; the next launch is released after it.  At overlap levels 1 and 2 the codes themselves are
// read before it, as many as the ring holds, and the next launch is released at once.  Waits on mbarriers are bounded: a wait
// that gives up marks the launch failed (status word, NaN rows); the CTA still meets its cluster and frees its tensor memory.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>
#include <atomic>
#include "ptqtp_internal.h"

namespace ptqtp {

namespace {

constexpr int kBlockTiles8 = 8;                        // tiles per CTA and superblock at most: 128 weight rows
constexpr int kStage8 = kBlockTiles8 * kTile3;         // 34816 bytes
constexpr int kQuarter2 = 8192;                        // format 2: code bytes of a quarter (16 row pairs) of a stage; the scale quads follow the four quarters
constexpr int kCodeStages8 = 3;
constexpr int kDone8 = 4;                               // MMAs of a group done: barriers, taken in turn
constexpr int kXStages8 = 4;                           // scale groups of activations
// warps: decoders (a warpgroup per quarter of a superblock's half-groups), sums, MMA issue, code copies, activations
constexpr int kDecoders8 = 16, kSummers8 = 8;
constexpr int kWarpSum8 = kDecoders8, kWarpMma8 = kWarpSum8 + kSummers8, kWarpCopy8 = kWarpMma8 + 1, kWarpX8 = kWarpCopy8 + 1;
constexpr int kThreads8 = 32 * (kWarpX8 + 1);

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst_smem, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst_smem), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
// A box of the tensor map (64 columns x its rows), first column x, to this CTA's shared memory; rows past the tensor read as zeros.
__device__ __forceinline__ void tma_load(uint32_t dst_smem, const CUtensorMap* map, int x, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst_smem), "l"(map), "r"(x), "r"(0), "r"(bar) : "memory");
}
// Format 2: a box of code bytes (128 bytes, 16 row pairs, the four atoms of 64 columns) or of scale quads (32 bytes, 16 row pairs).
__device__ __forceinline__ void tma_load_codes(uint32_t dst_smem, const CUtensorMap* map, int x, int pair, int slice, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(dst_smem), "l"(map), "r"(x), "r"(pair), "r"(0), "r"(slice), "r"(bar) : "memory");
}
__device__ __forceinline__ void tma_load_scales(uint32_t dst_smem, const CUtensorMap* map, int x, int pair, int slice, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(dst_smem), "l"(map), "r"(x), "r"(pair), "r"(slice), "r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Wait of a converged warp for a phase of an mbarrier (lanes may name different ones); gives up after `limit` polls or when
// another warp of the CTA has given up.
__device__ __forceinline__ bool wait_on8(uint32_t bar, uint32_t parity, int limit, volatile int* failed) {
    for (int i = 0; i < limit; ++i) {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        if ((i & 31) == 31 && __any_sync(0xffffffffu, *failed != 0)) break;
    }
    *failed = 1;
    return false;
}
__device__ __forceinline__ bool wait8(uint32_t bar, uint32_t parity, int limit, volatile int* failed) {
    return __all_sync(0xffffffffu, mbar_try_wait(bar, parity)) || wait_on8(bar, parity, limit, failed);
}
// One arrival for the whole warp; the warp barrier orders every lane's earlier operations before it.
__device__ __forceinline__ void warp_arrive(uint32_t bar) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// The MMAs of a scale group, issued by one elected lane of a converged warp: eight k-steps for each plane, four of them (64 columns) from
// either stage of trits.  d, d2: accumulators of the planes; a0, a1: the stages (plane 1 is 32 columns on, a k-step 8); b: activations
// (a k-step is 32 bytes, the second half BOX bytes on).  The stages are free, and the group is done, when the barriers say so.
// One piece of assembly: election, operands and issue have no branch around them, and few instructions; beside 16 decoding warps each
// costs this warp about ten cycles.
#define PTQTP_MMA8(D, A, B, ADD) "@e tcgen05.mma.cta_group::1.kind::f16 [" D "], [" A "], " B ", %4, " ADD ";\n\t"
#define PTQTP_COMMIT8(BAR) "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [" BAR "];\n\t"
#define PTQTP_HALF8(A, FIRST)                                                                                                  \
    "add.u32 a1, " A ", 8;\n\tadd.u32 a2, " A ", 16;\n\tadd.u32 a3, " A ", 24;\n\tadd.u32 c0, " A ", 32;\n\t"                    \
    "add.u32 c1, " A ", 40;\n\tadd.u32 c2, " A ", 48;\n\tadd.u32 c3, " A ", 56;\n\t"                                           \
    "add.u64 b1, b0, 2;\n\tadd.u64 b2, b0, 4;\n\tadd.u64 b3, b0, 6;\n\t"                                                       \
    PTQTP_MMA8("%0", A, "b0", FIRST) PTQTP_MMA8("%1", "c0", "b0", FIRST) PTQTP_MMA8("%0", "a1", "b1", "t")                       \
    PTQTP_MMA8("%1", "c1", "b1", "t") PTQTP_MMA8("%0", "a2", "b2", "t") PTQTP_MMA8("%1", "c2", "b2", "t")                        \
    PTQTP_MMA8("%0", "a3", "b3", "t") PTQTP_MMA8("%1", "c3", "b3", "t")
template <int BOX>
__device__ __forceinline__ void mma_group(uint32_t d, uint32_t d2, uint32_t a0, uint32_t a1, uint64_t b, uint32_t idesc, uint32_t free0, uint32_t free1,
                                          uint32_t done) {
    asm volatile(
        "{\n\t.reg .pred e, t, f;\n\t.reg .b32 a1, a2, a3, c0, c1, c2, c3;\n\t.reg .b64 b0, b1, b2, b3;\n\t"
        "elect.sync _|e, 0xffffffff;\n\tsetp.eq.b32 t, 0, 0;\n\tsetp.ne.b32 f, 0, 0;\n\t"
        "mov.b64 b0, %3;\n\t"
        PTQTP_HALF8("%2", "f")
        PTQTP_COMMIT8("%6")
        "add.u64 b0, b0, %9;\n\t"
        PTQTP_HALF8("%5", "t")
        PTQTP_COMMIT8("%7") PTQTP_COMMIT8("%8")
        "}"
        ::"r"(d), "r"(d2), "r"(a0), "l"(b), "r"(idesc), "r"(a1), "r"(free0), "r"(free1), "r"(done), "n"(BOX / 16) : "memory");
}
#undef PTQTP_HALF8
#undef PTQTP_COMMIT8
#undef PTQTP_MMA8
// 16 lanes x 32 columns of tensor memory; thread (g, t): columns 8 i + 2 t + 0 | 1 of lane g in r[4 i], r[4 i + 1], of lane g + 8 in
// r[4 i + 2], r[4 i + 3].
__device__ __forceinline__ void tmem_st_16x256b_x4(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile("tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
                   "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr) : "memory");
}
// The loads above complete here; the registers pass through so that no use of them can be scheduled earlier.
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&a)[8], uint32_t (&b)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                   "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7])
                 :: "memory");
}
// Shared-memory matrix descriptor, K-major, 128-byte swizzle: rows of 128 bytes (64 columns), 1024 bytes between groups of eight rows.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3fffu) | (uint64_t)1 << 16 | (uint64_t)(1024 >> 4) << 32 | (uint64_t)1 << 46 | (uint64_t)2 << 61;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, uint32_t rank) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
    return remote;
}
// A copy into the shared memory of a rank of the cluster; its bytes count on an mbarrier of that rank.
__device__ __forceinline__ void copy_to_rank(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ bool wait_cluster8(uint32_t bar, int limit) {
    bool ok = false;
    for (int i = 0; i <= limit && !ok; ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(bar) : "memory");
        ok = __all_sync(0xffffffffu, done != 0);
    }
    return ok;
}

// Two fp32 operations per instruction (each rounded on its own, as in single ones).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    float2 d;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(v));
    return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Tensor memory: kDSets sets of accumulators (both planes), then kAStages stages of trits (half a scale group, both planes: 64
// columns).
template <int NPAD>
struct Cfg8 {
    static constexpr int kDSets = 2;
    static constexpr int kACol = kDSets * 2 * NPAD;
    static constexpr int kAStages = (512 - kACol) / 64;
    static constexpr int kSums = NPAD / 2;             // each of the two summing warpgroups has half of the columns
    static constexpr int x_box = NPAD * 128, x_buf = 2 * x_box;          // 64 columns of every row, swizzled; a scale group
    static constexpr int x_off = kCodeStages8 * kStage8;                 // a multiple of 1024
    static constexpr int bar_off = x_off + kXStages8 * x_buf;
    static constexpr int bars = 5 * kCodeStages8 + kXStages8 + 2 * kAStages + kDSets + kDone8 + 1;
    static constexpr int red_off = bar_off + (8 * bars + 16 + 127) / 128 * 128;
    static constexpr int red = 128 * NPAD * 4;                           // partial sums from the ranks of a cluster: [rank][column][row]
    static constexpr int total = red_off + red + 1024;                   // (the base is moved to a multiple of 1024)
    static_assert(x_off % 1024 == 0, "the swizzle goes by address bits");
    static_assert(kAStages >= 4, "a decoding warpgroup steps four stages at a time");
    static_assert(total <= 227 * 1024, "shared memory");
};

// The trits of field F of the low or high bytes of a code word's halves (two columns), times 2: a code at the top of a half, inverted, is
// the sign and the top bit of the exponent (00 -> -2, 01 -> -0, 10 -> 2).
template <int F, bool HIGH>
__device__ __forceinline__ uint32_t trits(uint32_t word) {
    return ~(word << ((HIGH ? 6 : 14) - 2 * F)) & 0xc000c000u;
}

struct Args8 {
    CUtensorMap map;                                   // X: k columns x m rows, boxes of 64 x NPAD
    CUtensorMap code_map[2], scale_map[2];             // format 2: full slices, last slice
    int slices;
    const unsigned char* codes;
    __half* Y;
    int n, k, m, nrb, sbs, tiles_base, tiles_rem, csize, early, spin_limit, inject;
    int* status_word;
};

// LEVELS: 2 sums the groups of a superblock by themselves first (up to 32 rows: the registers); the short chains round less.  1 is the same
// for every batch size: a row's bits do not depend on the rows around it.
template <int FMT, int NPAD, int LEVELS>
__global__ void __launch_bounds__(kThreads8, 1)
gemm8_kernel(const __grid_constant__ Args8 a) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    using C = Cfg8<NPAD>;
    const uint32_t bars = smem_u32(smem + C::bar_off);
    const uint32_t code_full = bars, code_free = code_full + 32 * kCodeStages8, x_full = code_free + 8 * kCodeStages8,
                   a_full = x_full + 8 * kXStages8, a_free = a_full + 8 * C::kAStages, d_free = a_free + 8 * C::kAStages, done = d_free + 8 * C::kDSets, r_full = done + 8 * kDone8;
    uint32_t& tmem_slot = *reinterpret_cast<uint32_t*>(smem + C::bar_off + 8 * C::bars);
    volatile int* failed = reinterpret_cast<volatile int*>(smem + C::bar_off + 8 * C::bars + 8);

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int crank = (int)blockIdx.x % a.csize, blk = (int)blockIdx.x / a.csize;
    const int rb0 = blk * a.tiles_base + min(blk, a.tiles_rem), tiles = a.tiles_base + (blk < a.tiles_rem ? 1 : 0);
    const int sb_base = a.sbs / a.csize, sb_rem = a.sbs % a.csize;
    const int sb_lo = crank * sb_base + min(crank, sb_rem), nsb = sb_base + (crank < sb_rem ? 1 : 0);
    const int gg_lo = 4 * sb_lo, ng = max(0, min(4 * nsb, a.k / 128 - gg_lo));       // scale groups of this CTA

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 32) {
        for (int i = 0; i < 4 * kCodeStages8; ++i) mbar_init(code_full + 8 * i, 1);          // one per stage and quarter of the block
        for (int i = 0; i < kCodeStages8; ++i) mbar_init(code_free + 8 * i, kDecoders8 + kSummers8);
        for (int i = 0; i < kXStages8; ++i) mbar_init(x_full + 8 * i, 1);
        for (int i = 0; i < C::kAStages; ++i) { mbar_init(a_full + 8 * i, 4); mbar_init(a_free + 8 * i, 1); }
        for (int i = 0; i < C::kDSets; ++i) mbar_init(d_free + 8 * i, kSummers8);
        for (int i = 0; i < kDone8; ++i) mbar_init(done + 8 * i, 1);
        mbar_init(r_full, 1);
        *failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (a.csize > 1) mbar_expect_tx(r_full, 128u * NPAD * 4u);
    }
    if (warp == kWarpX8 && lane == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(&a.map) : "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    constexpr uint32_t tbase = 0u;                       // all columns are this CTA's
    if (tmem_slot != tbase) *failed = 1;
    const uint32_t xbuf = smem_u32(smem + C::x_off);
    // The MMAs of group g are done: its activations may be overwritten, its accumulators read.  Nobody who waits is four groups late:
    // the MMAs of group g + 4 need something from each of them that comes after.
    auto group_done = [&](int g) { return wait8(done + 8 * (g % kDone8), (uint32_t)(g / kDone8) & 1u, a.spin_limit, failed); };
    if (a.csize > 1) cluster_arrive();                   // awaited before the first store into another rank
    const int rows = min(16 * tiles, a.n - 16 * rb0);
    // One warp of a CTA releases the next launch for all of it.  The copying warp, which has not waited yet, does so only where launches
    // may overlap; otherwise the next kernel starts when everything before this one is complete, as after a plain launch.
    if (warp != kWarpCopy8) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (warp != kWarpCopy8 || a.early) asm volatile("griddepcontrol.launch_dependents;");

    if (warp < kDecoders8) {
        // ---- codes -> trits in tensor memory ----
        const int wg = warp >> 2, q = warp & 3, u = wg >> 1, half = wg & 1, g = lane >> 2, t = lane & 3;
        const uint32_t tlane = tbase + ((uint32_t)(32 * q) << 16) + C::kACol;
        int stage = wg, cs = 0;
        uint32_t aph = 1, cph = 0;
        bool ok = a.inject == 0;
        if (!ok) *failed = 1;
        // The words of k-step kk, for columns 4 t .. 4 t + 3, of both groups that this warpgroup takes of a superblock (h: groups u, 2 + u).
        // Format 3: chunk 4 half + kk, of the two words of a lane entry the one for these columns; the groups lie side by side.
        // Format 2: word t of atom kk of the 64 columns 2 (2 h + u) + half, in lines of 128 bytes [atom][row pair] swizzled by TMA.
        const unsigned char* words = FMT == 3 ? smem + 2 * q * kTile3 + 4 * half * 512 + (4 * g + 2 * u + (t & 1)) * 16 + (t >> 1) * 8
                                              : smem + q * kQuarter2 + g * 128 + (((2 * u + half) ^ g) * 16) + 4 * t;
        const int other = FMT == 3 ? 0 : ((((4 + 2 * u + half) ^ g) - ((2 * u + half) ^ g)) * 16);        // from h = 0 to h = 1
        for (int sl = 0; sl < nsb && ok; ++sl) {
            ok = wait8(code_full + 8 * (4 * cs + q), cph, a.spin_limit, failed);
            if (!ok) break;
            uint2 v[2][4];
#pragma unroll
            for (int tl = 0; tl < 2; ++tl)
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    if constexpr (FMT == 3) {
                        v[tl][kk] = *reinterpret_cast<const uint2*>(words + cs * kStage8 + tl * kTile3 + kk * 512);
                    } else {
                        const unsigned char* w = words + cs * kStage8 + kk * 2048 + tl * 1024;
                        v[tl][kk] = make_uint2(*reinterpret_cast<const uint32_t*>(w), *reinterpret_cast<const uint32_t*>(w + other));
                    }
                }
            warp_arrive(code_free + 8 * cs);
            if (++cs == kCodeStages8) { cs = 0; cph ^= 1u; }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (4 * sl + 2 * h + u >= ng) break;
                ok = wait8(a_free + 8 * stage, aph, a.spin_limit, failed);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int tl = 0; tl < 2; ++tl) {
                    const uint32_t dst = tlane + 64 * stage + ((uint32_t)(16 * tl) << 16);
                    uint32_t w[4], p[16];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        w[i] = __byte_perm(h == 0 ? v[tl][i].x : v[tl][i].y, 0u, 0x3120);
                        p[4 * i] = trits<0, false>(w[i]); p[4 * i + 1] = trits<0, true>(w[i]);
                        p[4 * i + 2] = trits<2, false>(w[i]); p[4 * i + 3] = trits<2, true>(w[i]);
                    }
                    tmem_st_16x256b_x4(dst, p);          // (a tile past the block's: lanes that nobody reads)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        p[4 * i] = trits<1, false>(w[i]); p[4 * i + 1] = trits<1, true>(w[i]);
                        p[4 * i + 2] = trits<3, false>(w[i]); p[4 * i + 3] = trits<3, true>(w[i]);
                    }
                    tmem_st_16x256b_x4(dst + 32, p);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                warp_arrive(a_full + 8 * stage);
                stage += 4;
                if (stage >= C::kAStages) { stage -= C::kAStages; aph ^= 1u; }
            }
        }
    } else if (warp < kWarpMma8) {
        // ---- accumulators -> sums ----
        const int ew = (warp - kWarpSum8) >> 2, q = warp & 3;
        const uint32_t tlane = tbase + ((uint32_t)(32 * q) << 16) + ew * C::kSums;
        const unsigned char* quads = (FMT == 3 ? smem + (2 * q + (lane >> 4)) * kTile3 + kTileCodes3 : smem + 4 * kQuarter2 + q * 512 + (lane >> 4) * 256) +
                                     (lane & 7) * 32 + ((lane >> 3) & 1) * 4;
        uint64_t y[C::kSums / 2], part[LEVELS == 2 ? C::kSums / 2 : 1];
#pragma unroll
        for (int i = 0; i < C::kSums / 2; ++i) y[i] = 0ull;
        int cs = 0, gi = 0;
        uint32_t cph = 0;
        bool ok = true;
#pragma unroll 1
        for (int sl = 0; sl < nsb && ok; ++sl) {
            ok = wait8(code_full + 8 * (4 * cs + q), cph, a.spin_limit, failed);
            if (!ok) break;
            __half2 alpha[4];
#pragma unroll
            for (int G = 0; G < 4; ++G) alpha[G] = *reinterpret_cast<const __half2*>(quads + cs * kStage8 + 8 * G);
            warp_arrive(code_free + 8 * cs);
            if (++cs == kCodeStages8) { cs = 0; cph ^= 1u; }
            if constexpr (LEVELS == 2) {
#pragma unroll
                for (int i = 0; i < C::kSums / 2; ++i) part[i] = 0ull;
            }
#pragma unroll
            for (int G = 0; G < 4; ++G, ++gi) {
                if (gi >= ng) break;
                const int ds = G % C::kDSets;        // (superblocks start with an even group)
                ok = group_done(gi);
                if (!ok) break;
                tc_fence_after();
                const float f1 = 0.5f * __low2float(alpha[G]), f2 = 0.5f * __high2float(alpha[G]);        // (the trits are times 2)
                const uint64_t a1 = pack2(f1, f1), a2 = pack2(f2, f2);
#pragma unroll
                for (int c0 = 0; c0 < C::kSums; c0 += 8) {
                    uint32_t d1[8], d2[8];
                    tmem_ld8(tlane + ds * 2 * NPAD + c0, d1);
                    tmem_ld8(tlane + ds * 2 * NPAD + NPAD + c0, d2);
                    tmem_ld_wait(d1, d2);
                    if (c0 + 8 == C::kSums) {
                        tc_fence_before();
                        warp_arrive(d_free + 8 * ds);
                    }
#pragma unroll
                    for (int i = 0; i < 8; i += 2) {
                        const uint64_t e1 = pack2(__uint_as_float(d1[i]), __uint_as_float(d1[i + 1])), e2 = pack2(__uint_as_float(d2[i]), __uint_as_float(d2[i + 1]));
                        if constexpr (LEVELS == 2) part[(c0 + i) / 2] = fma2(a1, e1, fma2(a2, e2, part[(c0 + i) / 2]));
                        else y[(c0 + i) / 2] = add2(y[(c0 + i) / 2], fma2(a1, e1, fma2(a2, e2, 0ull)));       // (one rounding at the size of the sum)
                    }
                }
            }
            if constexpr (LEVELS == 2) {
#pragma unroll
                for (int i = 0; i < C::kSums / 2; ++i) y[i] = add2(y[i], part[i]);
            }
        }
        if (*failed) {
            for (int i = 0; i < 64; ++i) __nanosleep(1000);          // copies in flight would land on the partial sums
#pragma unroll
            for (int i = 0; i < C::kSums / 2; ++i) y[i] = 0x7fc000007fc00000ull;
        }
        // [column][row] over the first code stage.  The last group's MMAs follow from every decoder's words, so these have been read, but of the
        // scales only those of superblocks whose first group is two groups back (two sets of accumulators): a last superblock of one or
        // two groups may be entered by the other summing warps only now.  Nobody stores before all of them are through.
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kSummers8) : "memory");
        float* dst = reinterpret_cast<float*>(smem) + ew * C::kSums * 128 + 32 * q + 16 * (lane >> 4) + 2 * (lane & 7) + ((lane >> 3) & 1);
#pragma unroll
        for (int i = 0; i < C::kSums; i += 2) {
            const float2 v = unpack2(y[i / 2]);
            dst[i * 128] = v.x;
            dst[i * 128 + 128] = v.y;
        }
        if (a.csize > 1) {
            // rank r of the cluster gets its share of the columns, from every rank: a copy each
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            cluster_wait();
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kSummers8) : "memory");
            if (warp == kWarpSum8 && lane < a.csize) {
                const uint32_t bytes = (uint32_t)(NPAD / a.csize) * 512u;
                copy_to_rank(cluster_addr(smem_u32(smem + C::red_off) + crank * bytes, (uint32_t)lane), smem_u32(smem) + lane * bytes, bytes,
                             cluster_addr(r_full, (uint32_t)lane));
            }
        }
    } else if (warp == kWarpMma8) {
        // ---- the MMAs, in the order of the groups ----
        constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(NPAD >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        // what a group waits for, a barrier per lane: activations, accumulators, the trits of either half; one poll for all
        const uint32_t ring_bar = lane == 0 ? x_full : lane == 1 ? d_free : a_full;
        const int ring = lane == 0 ? kXStages8 : lane == 1 ? C::kDSets : C::kAStages, step = lane < 2 ? 1 : 2;
        int pos = lane == 3 ? 1 : 0, stage = 0, xs = 0, ds = 0;
        uint32_t par = lane == 1 ? 1u : 0u;
        for (int gi = 0; gi < ng; ++gi) {
            if (!wait8(ring_bar + 8 * pos, par, a.spin_limit, failed)) break;
            pos += step;
            if (pos >= ring) { pos -= ring; par ^= 1u; }
            tc_fence_after();
            const uint64_t b = smem_desc(xbuf + xs * C::x_buf);
            const uint32_t d = tbase + ds * 2 * NPAD;
            const int stage1 = stage + 1 == C::kAStages ? 0 : stage + 1;
            mma_group<C::x_box>(d, d + NPAD, tbase + C::kACol + 64 * stage, tbase + C::kACol + 64 * stage1, b, idesc, a_free + 8 * stage,
                                a_free + 8 * stage1, done + 8 * (gi % kDone8));
            stage = stage1 + 1 == C::kAStages ? 0 : stage1 + 1;
            if (++xs == kXStages8) xs = 0;
            if (++ds == C::kDSets) ds = 0;
        }
    } else if (warp == kWarpCopy8) {
        // ---- the ring of code stages: lane q copies quarter q of the block (two tiles) ----
        const uint32_t bytes = lane >= 4 || tiles <= 2 * lane ? 0u : FMT == 3 ? (uint32_t)min(tiles - 2 * lane, 2) * kTile3 : kQuarter2 + 512u;
        const unsigned char* src = FMT == 3 ? a.codes + ((size_t)sb_lo * a.nrb + rb0 + 2 * (lane & 3)) * kTile3 : nullptr;
        if (!a.early) {
            // nothing is read before earlier work of the stream is complete but for a prefetch into L2, the point of coherence
            if (FMT == 3 && bytes && nsb > 0) bulk_prefetch_l2(src, bytes);
            asm volatile("griddepcontrol.wait;" ::: "memory");
        }
        int cs = 0;
        uint32_t cph = 1;
        for (int sl = 0; sl < nsb; ++sl) {
            // past the first round of the ring a stage is freed by warps that wait for the kernel ahead: its time is not for the polls to count
            if (a.early && sl == kCodeStages8) asm volatile("griddepcontrol.wait;" ::: "memory");
            if (!wait8(code_free + 8 * cs, cph, a.spin_limit, failed)) break;
            if (lane < 4) {
                const uint32_t full = code_full + 8 * (4 * cs + lane);
                mbar_expect_tx(full, bytes);
                if constexpr (FMT == 3) {
                    if (bytes) bulk_copy_g2s(smem_u32(smem + cs * kStage8 + 2 * lane * kTile3), src + (size_t)sl * a.nrb * kTile3, bytes, full);
                } else if (bytes) {
                    // 16 row pairs, whether the block has them or not: what lies past its end or past the matrix nobody reads
                    const int slice = (sb_lo + sl) >> 2, part = (sb_lo + sl) & 3, last = slice == a.slices - 1 ? 1 : 0, at = last ? 0 : slice;
                    tma_load_codes(smem_u32(smem + cs * kStage8 + lane * kQuarter2), &a.code_map[last], 128 * part, 8 * rb0 + 16 * lane, at, full);
                    tma_load_scales(smem_u32(smem + cs * kStage8 + 4 * kQuarter2 + lane * 512), &a.scale_map[last], 32 * part, 8 * rb0 + 16 * lane, at, full);
                }
            }
            __syncwarp();
            if (++cs == kCodeStages8) { cs = 0; cph ^= 1u; }
        }
        if (a.early && nsb <= kCodeStages8) asm volatile("griddepcontrol.wait;" ::: "memory");
    } else {
        // ---- activations, a scale group of all rows at a time ----
        int xs = 0;
        for (int gi = 0; gi < ng; ++gi) {
            if (gi >= kXStages8 && !group_done(gi - kXStages8)) break;
            if (lane == 0) {
                mbar_expect_tx(x_full + 8 * xs, C::x_buf);
                for (int b = 0; b < 2; ++b) tma_load(xbuf + xs * C::x_buf + b * C::x_box, &a.map, 128 * (gg_lo + gi) + 64 * b, x_full + 8 * xs);
            }
            __syncwarp();
            if (++xs == kXStages8) xs = 0;
        }
    }
    bool arrived = true;
    if (a.csize > 1) {
        if (warp < kWarpSum8 || warp >= kWarpMma8) cluster_wait();
        arrived = wait_cluster8(r_full, a.spin_limit);
        if (!arrived) *failed = 1;
    } else {
        __syncthreads();
    }
    {
        // this rank's columns: the partial sums of all ranks, in their order; eight rows per thread
        const int per = NPAD / a.csize;
        const float* sums = reinterpret_cast<const float*>(smem + (a.csize > 1 ? C::red_off : 0));
        const bool wide = (a.n & 7) == 0;
#pragma unroll 1
        for (int i = tid; i < per * 16; i += kThreads8) {
            const int col = crank * per + (i >> 4), row = 8 * (i & 15);
            float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
            for (int r = 0; r < a.csize; ++r) {
                const float4* v = reinterpret_cast<const float4*>(sums + (r * per + (i >> 4)) * 128 + row);
                const float4 v0 = v[0], v1 = v[1];
                s0.x += v0.x; s0.y += v0.y; s0.z += v0.z; s0.w += v0.w;
                s1.x += v1.x; s1.y += v1.y; s1.z += v1.z; s1.w += v1.w;
            }
            __half2 h[4] = {__floats2half2_rn(s0.x, s0.y), __floats2half2_rn(s0.z, s0.w), __floats2half2_rn(s1.x, s1.y), __floats2half2_rn(s1.z, s1.w)};
            if (!arrived)
                for (int e = 0; e < 4; ++e) h[e] = __half2half2(__ushort_as_half((unsigned short)0x7fffu));
            if (col >= a.m) continue;
            __half* dst = a.Y + (size_t)col * a.n + 16 * rb0 + row;
            if (wide && row + 8 <= rows) {
                *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(h);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (row + e < rows) dst[e] = e & 1 ? __high2half(h[e >> 1]) : __low2half(h[e >> 1]);
            }
        }
    }
    __syncthreads();
    if (*failed) {
        if (tid == 0) atomicExch(a.status_word, (int)PTQTP_ERR_CUDA);
        // copies and MMAs whose waits gave up may still be in flight: give them time before the memory is given back
        for (int i = 0; i < 64; ++i) __nanosleep(1000);
    }
    if (a.csize > 1) {                                   // no rank leaves while another may still send to it
        cluster_arrive();
        cluster_wait();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tbase) : "memory");
}

// cuTensorMapEncodeTiled, asked of the runtime once (the library does not link against the driver).
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static std::atomic<PFN_cuTensorMapEncodeTiled_v12000> known{nullptr};
    PFN_cuTensorMapEncodeTiled_v12000 f = known.load(std::memory_order_acquire);
    if (!f) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult found = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        f = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        known.store(f, std::memory_order_release);
    }
    return f;
}

template <int FMT, int NPAD, int LEVELS>
ptqtp_status launch_n8(Args8& a, const uint16_t* X, int blocks, cudaStream_t st) {
    ptqtp_status s = configure_once<gemm8_kernel<FMT, NPAD, LEVELS>>();
    if (s != PTQTP_OK) return s;
    const PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();
    const cuuint64_t dims[2] = {(cuuint64_t)a.k, (cuuint64_t)a.m}, strides[1] = {(cuuint64_t)a.k * 2};
    const cuuint32_t box[2] = {64, NPAD}, steps[2] = {1, 1};
    if (!encode || encode(&a.map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<uint16_t*>(X), dims, strides, box, steps,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) return PTQTP_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks * a.csize);
    cfg.blockDim = dim3(kThreads8);
    cfg.dynamicSmemBytes = Cfg8<NPAD>::total;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = a.csize;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, gemm8_kernel<FMT, NPAD, LEVELS>, a);
    if (e != cudaSuccess) { set_last_cuda_error(e); (void)cudaGetLastError(); return PTQTP_ERR_CUDA; }
    return PTQTP_OK;
}

// Clusters of csize CTAs that run at once (one CTA per SM; larger clusters leave SMs of a GPC idle): of 4 and 8 what the runtime said
// on this device for kernels of this footprint, 33 and 15 of 148 SMs.
int clusters8(int csize, int sms) {
    return csize <= 2 ? sms / csize : csize == 4 ? max(1, sms * 33 / 148) : max(1, sms * 15 / 148);
}

// How many CTAs share the columns of a row block, and the microseconds that the launch should take in a chain at level 0.  A wave of
// CTAs takes a fixed time and its longest share of superblocks; a cluster takes a little longer to meet.  Microseconds per scale
// group as measured (16, 32, 48, 64 rows).
struct Plan8 {
    int split;
    double us;
};
Plan8 plan8(int blocks, int sbs, int npad) {
    const double group = npad == 16 ? 0.35 : npad == 32 ? 0.39 : npad == 48 ? 0.46 : 0.53;
    const int sms = sm_count();
    Plan8 best = {1, 0.0};
    for (int c = 1; c <= 8 && (c == 1 || c <= sbs); c *= 2) {
        const int waves = (blocks + clusters8(c, sms) - 1) / clusters8(c, sms);
        const double us = waves * (4.2 + 4.0 * group * ((sbs + c - 1) / c)) + (c > 1 ? 0.7 : 0.0);
        if (c == 1 || us < best.us) best = {c, us};
    }
    return best;
}
int blocks8(const Layout3& L) { return (L.nrb + kBlockTiles8 - 1) / kBlockTiles8; }

}  // namespace

double gemm8_plan_us(const Layout3& L, int m) { return plan8(blocks8(L), L.sbs, (m + 15) / 16 * 16).us; }

// What a launch of up to 32 rows takes in a chain at level 0, closer than the plan, which is high for small matrices: per wave a fixed time and
// the scale groups of the busiest CTA, a cluster's meeting, bytes, rows that no 16-byte store takes.  Within 11 % (4 % on average) of
// 961 calls on format 2 (9 to 16 rows) and 849 on format 3 (17 to 32), 128 to 28672 rows by 256 to 28672 columns.
static double gemm8_us(int blocks, int n, int k, int m, size_t total, bool v2) {
    const int sbs = (k + kSuper3 - 1) / kSuper3, split = plan8(blocks, sbs, (m + 15) / 16 * 16).split;
    const int clusters = clusters8(split, sm_count()), waves = (blocks + clusters - 1) / clusters, groups = min(4 * ((sbs + split - 1) / split), k / kGroup);
    const bool odd = n % 8 != 0;
    return v2 ? waves * (2.55 + 0.33 * groups + (odd ? 0.27 : 0.0)) + 1.25 * (waves - 1) + (split > 1 ? 0.68 : 0.0) + 0.16e-6 * (double)total
              : waves * (3.35 + 0.28 * groups + (odd ? 0.56 : 0.0)) + 1.0 * (waves - 1) + (split > 1 ? 0.65 : 0.0) + 0.09e-6 * (double)total;
}
double gemm8_us(const Layout3& L, int m) { return gemm8_us(blocks8(L), L.n, L.k, m, L.total, false); }
double gemm8_us(const Layout2& L, int m) { return gemm8_us((L.nrp + 63) / 64, L.n, L.k, m, L.total, true); }
int gemm8_ctas(const Layout2& L, int m) {
    const int blocks = (L.nrp + 63) / 64;
    return blocks * plan8(blocks, (L.k + kSuper3 - 1) / kSuper3, (m + 15) / 16 * 16).split;
}

namespace {
void common8(Args8& a, int n, int k, int m, int nrb, int sbs, int split, uint16_t* Y, cudaStream_t st) {
    const int blocks = (nrb + kBlockTiles8 - 1) / kBlockTiles8;
    a.Y = reinterpret_cast<__half*>(Y);
    a.n = n; a.k = k; a.m = m; a.nrb = nrb; a.sbs = sbs;
    a.csize = split;
    a.tiles_base = nrb / blocks;
    a.tiles_rem = nrb % blocks;
    a.spin_limit = wait_poll_limit();
    a.early = overlap_enabled() && !consume_pack(st) ? 1 : 0;
    a.inject = take_injected_wait_failure() ? 1 : 0;
}
}  // namespace

// 1 <= m <= 64 rows of X (16-byte aligned) on format 3.  ksplit: CTAs of a cluster that share the columns of a row block (1, 2, 4 or
// 8; 0 = the split that should be fastest; -1 = as many as bring 128 CTAs, where K has that many superblocks).
ptqtp_status launch_gemm8(const Layout3& L, const void* packed, int m, const uint16_t* X, uint16_t* Y, int ksplit, cudaStream_t st) {
    if (m < 1 || m > 64) return PTQTP_ERR_SHAPE;
    if (ksplit != -1 && ksplit != 0 && ksplit != 1 && ksplit != 2 && ksplit != 4 && ksplit != 8) return PTQTP_ERR_CONFIG;
    const int blocks = blocks8(L), npad = (m + 15) / 16 * 16;
    const bool chosen = ksplit == 0;
    if (chosen) ksplit = plan8(blocks, L.sbs, npad).split;
    if (ksplit == -1) {
        ksplit = 1;
        while (ksplit < 8 && blocks * ksplit < 128 && 2 * ksplit <= L.sbs) ksplit *= 2;
    }
    Args8 a = {};
    a.codes = static_cast<const unsigned char*>(packed) + L.codes_off;
    if (gemv_status_word(&a.status_word) != PTQTP_OK) return PTQTP_ERR_CUDA;
    common8(a, L.n, L.k, m, L.nrb, L.sbs, ksplit, Y, st);
    switch (npad) {
        case 16: return chosen ? launch_n8<3, 16, 2>(a, X, blocks, st) : launch_n8<3, 16, 1>(a, X, blocks, st);
        case 32: return chosen ? launch_n8<3, 32, 2>(a, X, blocks, st) : launch_n8<3, 32, 1>(a, X, blocks, st);
        case 48: return launch_n8<3, 48, 1>(a, X, blocks, st);
        default: return launch_n8<3, 64, 1>(a, X, blocks, st);
    }
}

// The same on format 2.
ptqtp_status launch_gemm8(const Layout2& L, const void* packed, int m, const uint16_t* X, uint16_t* Y, cudaStream_t st) {
    if (m < 1 || m > 64) return PTQTP_ERR_SHAPE;
    const int nrb = (L.nrp + kTileRp3 - 1) / kTileRp3, sbs = (L.k + kSuper3 - 1) / kSuper3, npad = (m + 15) / 16 * 16;
    const int blocks = (nrb + kBlockTiles8 - 1) / kBlockTiles8;
    Args8 a = {};
    a.slices = L.slices;
    const PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();
    if (!encode || gemv_status_word(&a.status_word) != PTQTP_OK) return PTQTP_ERR_CUDA;
    for (int last = L.slices > 1 ? 0 : 1; last < 2; ++last) {
        // a unit: [4 atoms][64-column blocks] of 16 bytes, then a quad of 8 bytes per group
        const cuuint64_t blocks64 = last ? L.last_active : 32, unit = last ? L.last_unit : kUnit2, slices = last ? 1 : L.slices - 1;
        unsigned char* base = static_cast<unsigned char*>(const_cast<void*>(packed)) + L.codes_off + (last ? (size_t)(L.slices - 1) * L.nrp * kUnit2 : 0);
        const cuuint64_t dims[4] = {16 * blocks64, (cuuint64_t)L.nrp, 4, slices}, strides[3] = {unit, 16 * blocks64, unit * L.nrp};
        const cuuint32_t box[4] = {128, 16, 4, 1}, steps[4] = {1, 1, 1, 1};
        const cuuint64_t sdims[3] = {4 * blocks64, (cuuint64_t)L.nrp, slices}, sstrides[2] = {unit, unit * L.nrp};
        const cuuint32_t sbox[3] = {32, 16, 1};
        if (encode(&a.code_map[last], CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, base, dims, strides, box, steps, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
            encode(&a.scale_map[last], CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, base + 64 * blocks64, sdims, sstrides, sbox, steps, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return PTQTP_ERR_CUDA;
    }
    common8(a, L.n, L.k, m, nrb, sbs, plan8(blocks, sbs, npad).split, Y, st);
    switch (npad) {
        case 16: return launch_n8<2, 16, 2>(a, X, blocks, st);
        case 32: return launch_n8<2, 32, 2>(a, X, blocks, st);
        case 48: return launch_n8<2, 48, 1>(a, X, blocks, st);
        default: return launch_n8<2, 64, 1>(a, X, blocks, st);
    }
}

}  // namespace ptqtp
