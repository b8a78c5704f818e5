// Dual-trit-plane layer for 2 to 64 activation rows on packed formats 2 and 3:
//     Y[m] = alpha1 (.) (T1 X[m]) + alpha2 (.) (T2 X[m]),   m < M.
//
// Warp MMAs, every warp on its own: it streams tiles (16 weight rows x 512 columns) through a ring, decodes them in registers
// and multiplies.  Nothing is handed from warp to warp before the end.  The 16 rows of an MMA are 8 row pairs x 2 fields of
// their code bytes (row of the pair, plane); lanes read the entries of one group pair, not the entries a batch-1 fragment
// would take, so that an MMA contracts columns of one scale group only.
//   * fp16 (m16n8k16, fp32 sums; format 3): a shift and a mask of a code word make two trits of operand A, 15 instructions per 16
//     trits.  B is the activations as given, a column of B one batch row: y += alpha d in fp32.
//   * int8 (m16n8k32, exact int32 sums; formats 3 and 2): three masks per code word; B the activations in 15-bit block
//     fixed point per 128 columns (as in gemv5.cu and skinny3.cu), two columns, high and low byte, per batch row.  Codes are
//     trit + 1: the sum of x over the group comes off in the epilogue, y += alpha 2^s (4^-f d - sum x).
//   An MMA chain holds both planes of a row, which meet in the same lane.
// B is in shared memory, for all of a CTA's columns at once, in fragment order.
// Grid: clusters of C CTAs split the superblocks of K, clusters split the rows in tiles of 16; in a CTA kw warps split its
// superblocks.  The partial sums of a tile go to one rank's shared memory (st.async in a cluster), slot by slot, and are added in
// a fixed order at the end: no atomics, no workspace, reproducible.  C and kw depend on the shape alone.
//
// What bounds it, from microbenchmarks on an SM quarter: an MMA takes 8 cycles, a mask or shift 2 on another pipe beside it, a
// single-precision instruction 1 that the MMAs wait for.  A tile is 64 MMAs per 8 rows and 480 masks and shifts in fp16: 240 cycles
// per SM at 8 rows, 256 at 16, and the sums, against 187 of HBM; int8 with 4 rows 32 MMAs and 96 masks: 64.  On top of that 3 us per
// launch: start, activations, last sums.  14336 x 4096, microseconds per call in a chain at level 0: 4 rows 9.5 (one-group fragments of
// gemv5: 17.4), 8 rows 13.9 and 16 rows 19.2 (tcgen05 kernel: 15.5 and 15.3).
// Clusters of 4 and 8 leave 16 and 28 SMs idle (33 and 15 fit); larger C only where an activation slice does not fit.
//
// Precision of the fp16 form, the rounding of y taken out (512 x 4096, 16 rows; in brackets the tcgen05 kernel of the time with one CTA
// per row block, with four): 0.82e-7 of the result on normal x (1.44e-7, 0.94e-7), 0.80e-7 on x of mean 4 (1.44e-7, 0.92e-7),
// 0.82e-7 with a column of 30 to 30000 in every group whose trits are 0 (1.46e-7, 0.93e-7), 2.10e-7 with a column of 1000 in
// every group and any trits (2.41e-7, 2.15e-7), 1.99e-7 on x over 24 powers of two (2.31e-7, 2.06e-7).
//
// The kernel is always launched as a dependent of the kernel before it on the stream: everything that is visible to
// other work happens after griddepcontrol.wait, and the next kernel may start only then; before it the first tiles are
// prefetched into L2.  At overlap levels 1 and 2 (where it pays, see launch_nt7) they are read, and the next kernel may start at once.  Waits on mbarriers
// are bounded: a warp that gives up marks the launch failed (status word) and its rows come out as NaN.
#include <cuda_fp16.h>
#include <atomic>
#include "ptqtp_internal.h"

namespace ptqtp {

namespace {

// Warps of a CTA: as many as the registers leave (the accumulators grow with the batch).
__host__ __device__ constexpr int max_warps7(bool int8, int nt) { return nt <= 2 || (int8 && nt == 3) ? 16 : 8; }
constexpr int kDepth7 = 2;                             // tiles in flight per warp
constexpr size_t kSmem7 = 227 * 1024;
// Format 2: what one copy can bring is a slice unit (one row pair, 2048 columns), so four warps share a ring of tiles of
// 8 row pairs x 2048 columns and take a superblock each.  32 bytes between the row pairs spread them over the banks.
// (16-byte asynchronous copies by the lanes of each warp cost more issue slots than the arithmetic: 14.9 against 8.7 us on
// 14336 x 4096 at four rows.)
constexpr int kPair2 = kUnit2 + 32;
constexpr int kTile2 = 8 * kPair2;
__host__ __device__ constexpr int team7(int fmt) { return fmt == 3 ? 1 : 4; }        // warps that share a ring

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
template <bool CLUSTER>
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    if constexpr (CLUSTER)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
template <bool CLUSTER>
__device__ __forceinline__ bool wait_bounded(uint32_t bar, uint32_t parity, int limit) {
    bool ok = mbar_try_wait<CLUSTER>(bar, parity);
    for (int i = 0; i < limit && !ok; ++i) ok = mbar_try_wait<CLUSTER>(bar, parity);
    return __all_sync(0xffffffffu, ok);
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, uint32_t rank) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
    return remote;
}
// A store into the shared memory of a rank of the cluster; its bytes count on an mbarrier of that rank.
__device__ __forceinline__ void st_async2(uint32_t addr, uint32_t bar, float x, float y) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%2, %3}, [%1];"
                 ::"r"(addr), "r"(bar), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ void st_async1(uint32_t addr, uint32_t bar, float x) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %2, [%1];" ::"r"(addr), "r"(bar), "f"(x) : "memory");
}
__device__ __forceinline__ void mma_u8s8(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_u8s8_first(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(0));
}
__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16_first(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// Offsets in dynamic shared memory: the warps' rings, the activations of a chunk in fragment order, their group
// records (int8), the partial sums pushed here [own tile][source][16][stride], sums kept between chunks, barriers (one per ring slot,
// one for the partial sums).
struct Smem7 {
    uint32_t x, sx, red, keep, bars;
    size_t total;
};
inline int red_stride7(int npad) { return npad + 2; }      // rows two banks apart
inline Smem7 smem7(int fmt, bool int8, int npad, int warps, int chunk, int own_tiles, int sources, int kept_tiles) {
    const size_t x = (size_t)(warps / team7(fmt)) * kDepth7 * (fmt == 3 ? kTile3 : kTile2);
    const size_t sx = x + (size_t)chunk * npad * 1024, red = sx + (int8 ? (size_t)chunk * 4 * npad * 8 : 0);
    const size_t keep = red + (size_t)own_tiles * sources * 16 * red_stride7(npad) * 4;
    const size_t bars = (keep + (size_t)kept_tiles * 16 * npad * 4 + 15) / 16 * 16;
    const Smem7 s = {(uint32_t)x, (uint32_t)sx, (uint32_t)red, (uint32_t)keep, (uint32_t)bars, bars + (size_t)(warps * kDepth7 + 1) * 8 + 8};
    return s;
}

// int8: batch row `row` of column tile nt, 32 columns of one group per lane (runs t and t + 4 of 16), to 15-bit
// block fixed point: X = round(x 2^s) with the group maximum in [2^13, 2^14), X = 256 hi + lo with both bytes signed, high
// bytes in the even MMA columns, low bytes in the odd ones.
template <int FMT, int NT>
__device__ __forceinline__ void convert7(const uint4 (&r)[2][2], int grp, int nt, int row, int t, unsigned char* xs, int2* records) {
    uint32_t v[2][8];
    uint32_t m2 = 0u;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        v[i][0] = r[i][0].x; v[i][1] = r[i][0].y; v[i][2] = r[i][0].z; v[i][3] = r[i][0].w;
        v[i][4] = r[i][1].x; v[i][5] = r[i][1].y; v[i][6] = r[i][1].z; v[i][7] = r[i][1].w;
#pragma unroll
        for (int e = 0; e < 8; ++e) m2 = __vmaxu2(m2, v[i][e] & 0x7fff7fffu);
    }
    uint32_t mxb = max(m2 & 0xffffu, m2 >> 16);          // fp16 patterns order like the values
    mxb = max(mxb, __shfl_xor_sync(0xffffffffu, mxb, 1));
    mxb = max(mxb, __shfl_xor_sync(0xffffffffu, mxb, 2));
    int s = 0;
    if (mxb != 0u) {
        const int ef = (int)(mxb >> 10);
        const int ex = ef ? ef - 15 : (31 - __clz((int)mxb)) - 24;
        s = 13 - ex;
    }
    const float scale = __uint_as_float((uint32_t)(127 + s) << 23);
    uint32_t sum = 0u;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        uint32_t B[16];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            // adding 1.5 * 2^23 rounds to the nearest integer and leaves it in the low bits
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&v[i][e]));
            B[2 * e] = __float_as_uint(fmaf(f.x, scale, 12582912.f));
            B[2 * e + 1] = __float_as_uint(fmaf(f.y, scale, 12582912.f));
            sum += B[2 * e] + B[2 * e + 1];
        }
        uint32_t lo[4], hi[4];                           // four columns each
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            lo[q] = __byte_perm(__byte_perm(B[4 * q], B[4 * q + 1], 0x0040), __byte_perm(B[4 * q + 2], B[4 * q + 3], 0x0040), 0x5410);
            hi[q] = __byte_perm(__byte_perm(B[4 * q] + 0x80u, B[4 * q + 1] + 0x80u, 0x0051),
                                __byte_perm(B[4 * q + 2] + 0x80u, B[4 * q + 3] + 0x80u, 0x0051), 0x5410);
        }
        if (nt < NT) {
            const int run = t + 4 * i;
            unsigned char* base = xs + (size_t)(grp * NT + nt) * 1024;
            if constexpr (FMT == 3) {
                // k-step cc = run / 2, lanes t' = 2 (run % 2) + 0 | 1: columns 0-3 and 8-11 | 4-7 and 12-15
                unsigned char* d = base + (run >> 2) * 512 + (8 * row + 2 * (run & 1)) * 16 + ((run >> 1) & 1) * 8;
                *reinterpret_cast<uint2*>(d) = make_uint2(hi[0], hi[2]);
                *reinterpret_cast<uint2*>(d + 16) = make_uint2(hi[1], hi[3]);
                *reinterpret_cast<uint2*>(d + 64) = make_uint2(lo[0], lo[2]);
                *reinterpret_cast<uint2*>(d + 80) = make_uint2(lo[1], lo[3]);
            } else {
                // run = 4 (t' % 2) + 2 L + t' / 2, k-steps 2 L + 0 | 1, lane t': columns 0-7 | 8-15
                unsigned char* d = base + ((run >> 1) & 1) * 512 + (8 * row + 2 * (run & 1) + (run >> 2)) * 16;
                *reinterpret_cast<uint4*>(d) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                *reinterpret_cast<uint4*>(d + 64) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            }
        }
    }
    int isum = (int)(sum - 32u * 0x4B400000u);
    isum += __shfl_xor_sync(0xffffffffu, isum, 1);
    isum += __shfl_xor_sync(0xffffffffu, isum, 2);
    if (t == 0 && nt < NT) records[grp * (4 * NT) + 4 * nt + row] = make_int2((int)((uint32_t)(127 - s) << 23), isum);
}

// int8: one group of a tile for NT column tiles.  Fields 0, 1 (the planes of row 2 g) are one MMA chain, field 2 and the
// unmasked byte (all four fields) the other: three masks per code word.
template <int NT>
__device__ __forceinline__ void group_int8(const uint32_t (&word)[8], const unsigned char* xb, const unsigned char* quad, const int2* rec,
                                           float (&y)[NT][2]) {
    int ca[NT][4], cb[NT][4];
#pragma unroll
    for (int kp = 0; kp < 2; ++kp) {
        uint4 b[NT];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) b[nt] = *reinterpret_cast<const uint4*>(xb + nt * 1024 + kp * 512);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const uint32_t w1 = word[4 * kp + 2 * s], w2 = word[4 * kp + 2 * s + 1];
            const uint32_t a0 = w1 & 0x03030303u, a1 = w1 & 0x0c0c0c0cu, a2 = w2 & 0x03030303u, a3 = w2 & 0x0c0c0c0cu;
            const uint32_t e0 = w1 & 0x30303030u, e2 = w2 & 0x30303030u;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const uint32_t b0 = s ? b[nt].z : b[nt].x, b1 = s ? b[nt].w : b[nt].y;
                if (kp + s == 0) {
                    mma_u8s8_first(ca[nt], a0, a1, a2, a3, b0, b1);
                    mma_u8s8_first(cb[nt], e0, w1, e2, w2, b0, b1);
                } else {
                    mma_u8s8(ca[nt], a0, a1, a2, a3, b0, b1);
                    mma_u8s8(cb[nt], e0, w1, e2, w2, b0, b1);
                }
            }
        }
    }
    const uint2 sc = *reinterpret_cast<const uint2*>(quad);
    const float2 s0 = __half22float2(*reinterpret_cast<const __half2*>(&sc.x));      // row 2 g: alpha1, alpha2
    const float2 s1 = __half22float2(*reinterpret_cast<const __half2*>(&sc.y));      // row 2 g + 1
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        // Q_f = 4^f sum t X (columns 2 t high, 2 t + 1 low byte of batch row t; codes are trit + 1)
        const int2 m = rec[4 * nt];
        const int Q0 = (ca[nt][0] << 8) + (ca[nt][1] - m.y), Q1 = (ca[nt][2] << 8) + (ca[nt][3] - 4 * m.y);
        const int Q2 = (cb[nt][0] << 8) + (cb[nt][1] - 16 * m.y);
        const int Q3 = (cb[nt][2] << 8) + (cb[nt][3] - 85 * m.y) - Q0 - Q1 - Q2;
        const float cx = __int_as_float(m.x);
        y[nt][0] = fmaf(cx, fmaf(0.25f * s0.y, (float)Q1, s0.x * (float)Q0), y[nt][0]);
        y[nt][1] = fmaf(0.0625f * cx, fmaf(0.25f * s1.y, (float)Q3, s1.x * (float)Q2), y[nt][1]);
    }
}

// fp16: the trits of field F of the even or odd bytes of a code word (two columns), times 2: a code at the top of a half, inverted, is
// the sign and the top bit of the exponent (00 -> -2, 01 -> -0, 10 -> 2).  Exact and normal, and all of it on a pipe that
// runs beside the MMAs (FMAs do not: 8 cycles + 2; made with one FMA per two trits 14336 x 4096 took 14.7 and 20.4 us at 8 and 16
// rows, against 14.3 and 19.9).  The codes themselves, masked subnormals, as operand A and the sum of x taken off
// afterwards took 13.0 and 18.8, but a sum then has x where the trit is 0, and the MMA cuts products with a
// subnormal factor off where it would if that factor were 2^-14: 2.6e-6 of the result on normal x, 0.1 of it next to columns
// of 30000.
template <int F, bool ODD>
__device__ __forceinline__ uint32_t trits(uint32_t word) {
    return ~(word << ((ODD ? 6 : 14) - 2 * F)) & 0xc000c000u;
}

// One launch.  The shares are divided on the host (a dozen integer divisions per warp were half a microsecond of a launch): tile0
// and the tiles (8 row pairs) of a cluster, the superblocks of a rank, C = 1 << lg_csize, kw = 1 << lg_kw; all_tiles: of
// the matrix; chunk: superblocks of activations held at a time.
struct Args7 {
    const unsigned char* codes;
    const __half* X;
    __half* Y;
    int n, k, m, nrp, tile0, t_base, t_rem, all_tiles, sbs, s_base, s_rem;
    int slices, last_active, last_unit;                // format 2
    int lg_csize, lg_kw, chunk, early, spin_limit, inject;
    Smem7 at;
    int* status_word;
};

template <int FMT, bool INT8, int NT>
__global__ void __launch_bounds__(max_warps7(INT8, NT) * 32, 1)
gemm7_kernel(const __grid_constant__ Args7 a) {
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int ROWS = INT8 ? 4 : 8;                   // batch rows per MMA column tile
    constexpr int NPAD = ROWS * NT, RS = NPAD + 2;
    constexpr int NY = INT8 ? 2 : 4;                     // sums of a lane and column tile
    constexpr int kTileBytes = FMT == 3 ? kTile3 : kTile2, TEAM = team7(FMT);
    const int warps = blockDim.x >> 5, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int csize = 1 << a.lg_csize, crank = (int)blockIdx.x & (csize - 1), cl = (int)blockIdx.x >> a.lg_csize;
    // this cluster's tiles, this rank's superblocks, this warp's share of both
    const int t_lo = a.tile0 + cl * a.t_base + min(cl, a.t_rem), T = a.t_base + (cl < a.t_rem ? 1 : 0);
    constexpr int S = FMT == 3 ? 1 : 4;                  // superblocks that stay together
    const int sb_lo = S * (crank * a.s_base + min(crank, a.s_rem));
    const int sb_hi = min(a.sbs, sb_lo + S * (a.s_base + (crank < a.s_rem ? 1 : 0)));
    const int kw = 1 << a.lg_kw, tw = warps >> a.lg_kw, kl = warp & (kw - 1), tl = warp >> a.lg_kw;
    const int sources = csize << a.lg_kw;
    const Smem7& so = a.at;
    const uint32_t ring = smem_u32(smem) + (uint32_t)(warp / TEAM * kDepth7 * kTileBytes), xs = smem_u32(smem + so.x), red = smem_u32(smem + so.red);
    unsigned char* ring_p = smem + (size_t)(warp / TEAM) * kDepth7 * kTileBytes;
    int2* records = reinterpret_cast<int2*>(smem + so.sx);                // int8: (2^-s, sum of the integers)
    const uint32_t bars = smem_u32(smem + so.bars) + 8 * (warp / TEAM) * kDepth7, r_full = smem_u32(smem + so.bars) + 8 * warps * kDepth7;
    const int own_tiles = (T - crank + csize - 1) >> a.lg_csize;               // tiles crank, crank + csize, ... of the cluster

    if (a.early) asm volatile("griddepcontrol.launch_dependents;");
    if (lane == 0 && warp % TEAM == 0) {
#pragma unroll
        for (int d = 0; d < kDepth7; ++d) mbar_init(bars + 8 * d, 1);
        if (warp == 0) mbar_init(r_full, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (warp == 0 && csize > 1) mbar_expect_tx(r_full, (uint32_t)(own_tiles * sources * 16 * NPAD * 4));
    }
    __syncwarp();

    // producer (of this warp, or of the team: its first warp): the unit (tile, superblock or slice) that is requested next
    int pj = 0, ps = 0, ps0 = 0, ps1 = 0, pslot = 0;
    auto start_chunk = [&](int s0, int s1) {
        ps0 = FMT == 3 ? s0 + kl : s0;
        ps1 = s1;
        ps = ps0;
        pj = ps0 < s1 && tl < tw ? tl : T;
    };
    auto unit_src3 = [&](int j, int sb) { return a.codes + ((size_t)sb * a.all_tiles + t_lo + j) * kTile3; };
    auto issue = [&]() {
        if (pj < T) {
            if constexpr (FMT == 3) {
                if (lane == 0) mbar_expect_tx(bars + 8 * pslot, kTile3);
                if (lane == 0) bulk_copy_g2s(ring + pslot * kTile3, unit_src3(pj, ps), kTile3, bars + 8 * pslot);
            } else {
                // lane = row pair; past the end: the last one again
                const int slice = ps >> 2, unit_bytes = slice == a.slices - 1 ? a.last_unit : kUnit2;
                if (kl == 0) {
                    if (lane == 0) mbar_expect_tx(bars + 8 * pslot, 8u * (uint32_t)unit_bytes);
                    __syncwarp();
                    if (lane < 8)
                        bulk_copy_g2s(ring + pslot * kTile2 + lane * kPair2,
                                      a.codes + (size_t)slice * a.nrp * kUnit2 + (size_t)min(8 * (t_lo + pj) + lane, a.nrp - 1) * unit_bytes,
                                      (uint32_t)unit_bytes, bars + 8 * pslot);
                }
            }
            ps += kw;
            if (ps >= ps1) { ps = ps0; pj += tw; }
        }
        pslot = pslot + 1 == kDepth7 ? 0 : pslot + 1;
    };

    start_chunk(sb_lo, min(sb_hi, sb_lo + a.chunk));
    if (FMT == 3 && !a.early && lane == 0 && pj < T) bulk_prefetch_l2(unit_src3(pj, ps), kTile3);
    bool met = csize == 1;
    __syncthreads();
    if (!met) cluster_arrive();                          // awaited before the first store into another rank
    if (!a.early) {
        // the next kernel may start when everything before this one is complete, as after a plain launch
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;");
    }

    bool failed = a.inject != 0;
    int cslot = 0;
    uint32_t phase = 0;
    for (int s0 = sb_lo, ch = 0;; s0 += a.chunk, ++ch) {
        const int s1 = min(sb_hi, s0 + a.chunk), ns = max(0, s1 - s0);
        const bool last = s0 + a.chunk >= sb_hi;
        if (ch > 0) {
            __syncthreads();                             // everybody is done with the activations of the chunk before
            start_chunk(s0, s1);
        }
#pragma unroll
        for (int d = 0; d < kDepth7; ++d) issue();
        if (a.early && ch == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
        {
            // the activations: a warp takes eight batch rows of one group, a lane two runs of 16 columns of one row.  CTAs
            // start at different places: all of them read the same lines.
            // (int8: two column tiles of four rows at a time; the last one may be half a pair)
            // (one column tile: two groups at a time instead)
            constexpr int NP = INT8 ? (NT + 1) / 2 : NT;
            constexpr bool kPairs = INT8 && NT == 1;
            const int tasks = kPairs ? 2 * ns : ns * 4 * NP, rot = tasks ? (cl * 5) % tasks : 0;
            constexpr int U = 4;                         // tasks whose loads are in flight
            for (int w0 = warp; w0 < tasks; w0 += U * warps) {
                uint4 r[U][2][2];
#pragma unroll
                for (int q = 0; q < U; ++q) {
                    const int wr = w0 + q * warps + rot, w = wr < tasks ? wr : wr - tasks;
                    const int mi = kPairs ? g & 3 : 8 * (w % NP) + g, col = kSuper3 * s0 + 128 * (kPairs ? 2 * w + (g >> 2) : w / NP) + 16 * t;
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        r[q][i][0] = r[q][i][1] = make_uint4(0u, 0u, 0u, 0u);
                        if (w0 + q * warps < tasks && mi < a.m && col < a.k) {
                            const uint4* src = reinterpret_cast<const uint4*>(a.X + (size_t)mi * a.k + col + 64 * i);
                            r[q][i][0] = __ldcg(src);
                            r[q][i][1] = __ldcg(src + 1);
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < U; ++q) {
                    if (w0 + q * warps >= tasks) break;
                    const int wr = w0 + q * warps + rot, w = wr < tasks ? wr : wr - tasks;
                    if constexpr (INT8) {
                        convert7<FMT, NT>(r[q], kPairs ? 2 * w + (g >> 2) : w / NP, kPairs ? 0 : 2 * (w % NP) + (g >> 2), g & 3, t, smem + so.x, records);
                        continue;
                    }
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const uint4 lo = r[q][i][0], hi = r[q][i][1];
                        const uint32_t v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                        // four columns (p, q) of a k-step: even ones, then odd ones
                        uint32_t ev[4], od[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            ev[e] = __byte_perm(v[2 * e], v[2 * e + 1], 0x5410);
                            od[e] = __byte_perm(v[2 * e], v[2 * e + 1], 0x7632);
                        }
                        const int run = t + 4 * i;       // 16-column run of the group
                        uint32_t d0, d1;
                        {
                            // fragment (cc = run / 2, lane t' = 2 (run % 2) + 0 | 1): columns 0-3 and 8-11 | 4-7 and 12-15
                            d0 = xs + (uint32_t)((w * 4 + (run >> 1)) * 512 + (g * 4 + 2 * (run & 1)) * 16);
                            d1 = d0 + 16;
                            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(d0), "r"(ev[0]), "r"(od[0]), "r"(ev[2]), "r"(od[2]) : "memory");
                            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(d1), "r"(ev[1]), "r"(od[1]), "r"(ev[3]), "r"(od[3]) : "memory");
                        }
                    }
                }
            }
        }
        __syncthreads();

        int round = 0;
        for (int j = tl < tw ? tl : T; j < T; j += tw, ++round) {
            // fp16: rows 2 g (0, 1) and 2 g + 1 (2, 3), batch rows 8 nt + 2 t, + 1; int8: rows 2 g, 2 g + 1, batch row 4 nt + t
            float y[NT][NY];
            float* kept = reinterpret_cast<float*>(smem + so.keep) + (size_t)(round * warps + warp) * 16 * NPAD + lane;
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int i = 0; i < NY; ++i) y[nt][i] = ch > 0 ? kept[(nt * NY + i) * 32] : 0.f;
            for (int sb = s0 + kl; sb - kl % TEAM < s1; sb += kw) {
                if (!wait_bounded<false>(bars + 8 * cslot, phase, failed ? 256 : a.spin_limit)) failed = true;
                const unsigned char* tile = ring_p + cslot * kTileBytes;
                const unsigned char* xb = smem + so.x + (size_t)(sb - s0) * (NPAD * 1024) + lane * 16;
                auto group = [&](int G, const uint32_t (&word)[8], const unsigned char* quad) {
                    if constexpr (INT8) {
                        group_int8<NT>(word, xb + G * (NT * 1024), quad, records + ((sb - s0) * 4 + G) * NPAD + t, y);
                    } else {
                    float ca[NT][4], cb[NT][4];
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        uint4 b[NT];
#pragma unroll
                        for (int nt = 0; nt < NT; ++nt) b[nt] = *reinterpret_cast<const uint4*>(xb + ((G * NT + nt) * 4 + kk) * 512);
#pragma unroll
                        for (int s = 0; s < 2; ++s) {
                            const uint32_t w = word[2 * kk + s];
                            const uint32_t e0 = trits<0, false>(w), e1 = trits<1, false>(w), e2 = trits<2, false>(w), e3 = trits<3, false>(w);
                            const uint32_t o0 = trits<0, true>(w), o1 = trits<1, true>(w), o2 = trits<2, true>(w), o3 = trits<3, true>(w);
#pragma unroll
                            for (int nt = 0; nt < NT; ++nt) {
                                if (kk + s == 0) {
                                    mma_f16_first(ca[nt], e0, e1, o0, o1, b[nt].x, b[nt].y);
                                    mma_f16_first(cb[nt], e2, e3, o2, o3, b[nt].x, b[nt].y);
                                } else {
                                    mma_f16(ca[nt], e0, e1, o0, o1, s ? b[nt].z : b[nt].x, s ? b[nt].w : b[nt].y);
                                    mma_f16(cb[nt], e2, e3, o2, o3, s ? b[nt].z : b[nt].x, s ? b[nt].w : b[nt].y);
                                }
                            }
                        }
                    }
                    const uint2 sc = *reinterpret_cast<const uint2*>(quad);
                    const float2 s0v = __half22float2(*reinterpret_cast<const __half2*>(&sc.x));     // row 2 g: alpha1, alpha2
                    const float2 s1v = __half22float2(*reinterpret_cast<const __half2*>(&sc.y));     // row 2 g + 1
                    const float k0 = 0.5f * s0v.x, k1 = 0.5f * s0v.y, k2 = 0.5f * s1v.x, k3 = 0.5f * s1v.y;
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        y[nt][0] = fmaf(k1, ca[nt][2], fmaf(k0, ca[nt][0], y[nt][0]));
                        y[nt][1] = fmaf(k1, ca[nt][3], fmaf(k0, ca[nt][1], y[nt][1]));
                        y[nt][2] = fmaf(k3, cb[nt][2], fmaf(k2, cb[nt][0], y[nt][2]));
                        y[nt][3] = fmaf(k3, cb[nt][3], fmaf(k2, cb[nt][1], y[nt][3]));
                    }
                    }
                };
                if constexpr (FMT == 3) {
                    // the entries (chunk 2 cc + t / 2, 4 g + 2 u + t % 2) hold words of groups u and 2 + u
#pragma unroll 1
                    for (int u = 0; u < 2; ++u) {
                        uint4 v[4];
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc)
                            v[cc] = *reinterpret_cast<const uint4*>(tile + (2 * cc + (t >> 1)) * 512 + (4 * g + 2 * u + (t & 1)) * 16);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t word[8];
#pragma unroll
                            for (int cc = 0; cc < 4; ++cc) {
                                word[2 * cc] = h ? v[cc].y : v[cc].x;
                                word[2 * cc + 1] = h ? v[cc].w : v[cc].z;
                            }
                            group(2 * h + u, word, tile + kTileCodes3 + (4 * g + 2 * h + u) * 8);
                        }
                    }
                } else {
                    // atom (i, l) is columns 64 l + 16 i of the slice; lane t: i = 2 L + t / 2, l = t % 2 of the group
                    const int A = (sb >> 2) == a.slices - 1 ? a.last_active : 32, G0 = 4 * (sb & 3), groups = min(4, A / 2 - G0);
                    const unsigned char* atoms = tile + g * kPair2 + ((t >> 1) * A + (t & 1)) * 16;
#pragma unroll 1
                    for (int G = 0; G < groups; ++G) {   // (none in a superblock past the end)
                        const uint4 p = *reinterpret_cast<const uint4*>(atoms + 32 * (G0 + G));
                        const uint4 q = *reinterpret_cast<const uint4*>(atoms + 32 * (G0 + G) + 32 * A);
                        const uint32_t word[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
                        group(G, word, tile + g * kPair2 + 64 * A + (G0 + G) * 8);
                    }
                }
                // every lane has read the slot
                if constexpr (TEAM == 1) __syncwarp();
                else asm volatile("bar.sync %0, %1;" ::"r"(1 + warp / TEAM), "n"(32 * TEAM) : "memory");
                issue();
                if (++cslot == kDepth7) { cslot = 0; phase ^= 1u; }
            }
            if (!last) {
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int i = 0; i < NY; ++i) kept[(nt * NY + i) * 32] = y[nt][i];
                continue;
            }
            // push the partial sums to the rank that owns the tile
            if (!met) { cluster_wait(); met = true; }
            const int owner = j & (csize - 1), src = crank * kw + kl;
            // first of this lane's sums, in floats
            const int slot = (((j >> a.lg_csize) * sources + src) * 16 + 2 * g) * RS + (INT8 ? t : 2 * t);
            if (failed) {
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int i = 0; i < NY; ++i) y[nt][i] = __int_as_float(0x7fc00000);
            }
            if (csize == 1) {                            // this CTA's own memory (st.async only between the ranks of a cluster)
                float* dst = reinterpret_cast<float*>(smem + so.red) + slot;
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    if constexpr (INT8) {
                        dst[4 * nt] = y[nt][0];
                        dst[4 * nt + RS] = y[nt][1];
                    } else {
                        *reinterpret_cast<float2*>(dst + 8 * nt) = make_float2(y[nt][0], y[nt][1]);
                        *reinterpret_cast<float2*>(dst + 8 * nt + RS) = make_float2(y[nt][2], y[nt][3]);
                    }
                }
            } else {
                const uint32_t dst = cluster_addr(red + 4u * slot, (uint32_t)owner), bar = cluster_addr(r_full, (uint32_t)owner);
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    if constexpr (INT8) {
                        st_async1(dst + 16 * nt, bar, y[nt][0]);
                        st_async1(dst + 16 * nt + RS * 4, bar, y[nt][1]);
                    } else {
                        st_async2(dst + 32 * nt, bar, y[nt][0], y[nt][1]);
                        st_async2(dst + 32 * nt + RS * 4, bar, y[nt][2], y[nt][3]);
                    }
                }
            }
        }
        if (last) break;
    }
    if (!met) cluster_wait();
    // all partial sums of this rank's tiles: added in the order of the superblock shares, one rounding
    bool arrived = true;
    if (csize == 1) __syncthreads();
    else arrived = wait_bounded<true>(r_full, 0u, a.spin_limit);
    if (!arrived) failed = true;
    const float* mine = reinterpret_cast<const float*>(smem + so.red);
    // a half warp per (tile, batch row), lanes = rows
    for (int jj = 0, mi = 2 * warp + (lane >> 4);; mi += 2 * warps) {
        while (mi >= a.m) { mi -= a.m; ++jj; }
        if (jj >= own_tiles) break;
        const int r = lane & 15, row = 16 * (t_lo + crank + jj * csize) + r;
        const float* p = mine + (size_t)(jj * sources * 16 + r) * RS + mi;
        float s = 0.f;
        for (int q = 0; q < sources; ++q) s += p[q * 16 * RS];
        if (row < a.n) a.Y[(size_t)mi * a.n + row] = arrived ? __float2half_rn(s) : __ushort_as_half((unsigned short)0x7fffu);
    }
    if (failed) {
        if (lane == 0) atomicExch(a.status_word, (int)PTQTP_ERR_CUDA);
        // a copy whose wait gave up may still be in flight: give it time to land before the memory is released
        for (int i = 0; i < 64; ++i) __nanosleep(1000);
    }
    // a rank that gave up on partial sums must not leave before the others have stopped sending
    if (csize > 1) {
        __syncwarp();
        cluster_arrive();
        cluster_wait();
    }
}

// Clusters of csize CTAs that fit on the device at once (one CTA per SM; asked of the runtime once per device and size: every plan
// asks for several sizes, and every call makes a few plans, so what is known is read without a lock).
template <int FMT, bool INT8, int NT>
int max_clusters(int csize) {
    static std::atomic<int> known[64][4] = {};
    int dev = 0;
    const int lg = csize == 1 ? 0 : csize == 2 ? 1 : csize == 4 ? 2 : 3;
    if (csize == 1) return sm_count();
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return sm_count() / csize;
    int n = known[dev][lg].load(std::memory_order_relaxed);
    if (!n) {
        if (configure_once<gemm7_kernel<FMT, INT8, NT>>() != PTQTP_OK) return sm_count() / csize;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(sm_count() / csize * csize);
        cfg.blockDim = dim3(max_warps7(INT8, NT) * 32);
        cfg.dynamicSmemBytes = kSmem7;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = csize;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, gemm7_kernel<FMT, INT8, NT>, &cfg) != cudaSuccess || n < 1) { (void)cudaGetLastError(); n = sm_count() / csize; }
        n = n < sm_count() / csize ? n : sm_count() / csize;
        known[dev][lg].store(n, std::memory_order_relaxed);
    }
    return n;
}

// The launch shape of a matrix (rows in tiles of 16, superblocks): clusters, CTAs per cluster, warps that split K.
struct Plan7 {
    int csize, clusters, kw, per_cluster, share, blocks;
};
template <int FMT, bool INT8>
Plan7 plan7(int tiles, int sbs) {
    Plan7 best = {};
    double best_cost = 0.0;
    for (int c = 1; c <= 8; c *= 2) {
        constexpr int S = FMT == 3 ? 1 : 4;              // superblocks that stay together
        const int blocks = (sbs + S - 1) / S;
        if (c > 1 && c > blocks) break;
        Plan7 p;
        p.csize = c;
        p.clusters = min(max_clusters<FMT, INT8, 1>(c), tiles);
        p.per_cluster = (tiles + p.clusters - 1) / p.clusters;
        p.blocks = blocks;
        p.share = S * ((blocks + c - 1) / c);
        p.kw = FMT == 3 ? 1 : 4;                         // format 2: the warps of a team
        double units = 0.0;
        for (int kw = 1; FMT == 3 && kw <= 8; kw *= 2) {
            const int tw = 16 / kw;
            const double u = (double)((p.per_cluster + tw - 1) / tw) * ((p.share + kw - 1) / kw) + 0.02 * kw;
            if (kw == 1 || u < units) { units = u; p.kw = kw; }
        }
        // tiles of the busiest CTA; a superblock of activations costs about half a tile's time to bring in; a cluster costs
        // the time of a few tiles to start and to meet; two column tiles should fit at once
        double cost = p.per_cluster * (double)p.share + 0.5 * p.share + (c > 1 ? 2.0 : 0.0);
        if (smem7(FMT, INT8, INT8 ? 8 : 16, 8, p.share, (min(p.per_cluster, 32) + c - 1) / c, c * p.kw, 0).total > kSmem7) cost *= 2.0;
        if (best_cost == 0.0 || cost < best_cost) { best_cost = cost; best = p; }
    }
    return best;
}

// What one launch takes: column tiles (rows of X), warps, superblocks of activations at a time, tiles of a cluster, rounds of
// tiles whose sums wait for the next chunk (0: no chunks).
struct Fit7 {
    int nt, warps, chunk, per_cluster, rounds;
};
template <int FMT, bool INT8>
size_t total7(const Plan7& p, int nt, int warps, int chunk, int tiles, int rounds) {
    return smem7(FMT, INT8, (INT8 ? 4 : 8) * nt, warps, chunk, (tiles + p.csize - 1) / p.csize, p.csize * p.kw, rounds * warps).total;
}
// As many rows of X (up to 32, or 16 for int8) as leave room for all of a rank's activations beside the warps' rings, then as
// many tiles as leave room for their partial sums: a matrix too tall for one launch takes several, a row too long
// even for one column tile is taken in chunks.
template <int FMT, bool INT8>
Fit7 fit7(const Plan7& p, int m) {
    constexpr int ROWS = INT8 ? 4 : 8, S = FMT == 3 ? 1 : 4;             // S: superblocks that stay together
    Fit7 f = {};
    f.chunk = p.share;
    for (int n = min(4, (m + ROWS - 1) / ROWS); n >= 1 && !f.nt; --n)
        for (int w = max_warps7(INT8, n); w >= 8 && !f.nt; w -= 8)
            for (int seg = 1; seg <= p.per_cluster; seg *= 2) {
                const int tiles = (p.per_cluster + seg - 1) / seg;
                if (seg > 1 && tiles < 2 * w) break;     // a launch of its own only for some rounds of work
                if (total7<FMT, INT8>(p, n, w, p.share, tiles, 0) <= kSmem7) { f.nt = n; f.warps = w; f.per_cluster = tiles; break; }
            }
    if (!f.nt) {
        f.nt = 1;
        f.warps = 8;
        f.per_cluster = min(p.per_cluster, 16);
        f.rounds = (f.per_cluster + f.warps / p.kw - 1) / (f.warps / p.kw);
        while (f.chunk > S && total7<FMT, INT8>(p, 1, f.warps, f.chunk, f.per_cluster, f.rounds) > kSmem7) f.chunk -= S;
    } else if (f.warps == 16 && 8 >= p.kw * f.per_cluster) {
        f.warps = 8;                                     // no more warps than tiles to start on, but eight to bring in the activations
    }
    return f;
}

template <int FMT, bool INT8, int NT>
ptqtp_status launch_nt7(Args7 a, const Plan7& p, const Fit7& f, int clusters, cudaStream_t st) {
    ptqtp_status s = configure_once<gemm7_kernel<FMT, INT8, NT>>();
    if (s != PTQTP_OK) return s;
    a.chunk = f.chunk;
    // Overlap levels 1 and 2: worth it when the launch fills the device, or leaves room for a whole one beside it.  In between the first
    // CTAs of the next launch take the idle SMs and wait there while the rest queue for the others: 128 CTAs at level 2, 2048 x 4096
    // at 3 rows of format 2 6.0 us against 5.1 in stream order, 2048 x 2048 at 8 rows of format 3 5.2 against 4.2; 32 CTAs (512 x
    // 1024, 2 rows) 3.0 against 3.4, all SMs (14336 x 4096, 4 rows) 9.2 against 9.6.
    const bool overlap = clusters == max_clusters<FMT, INT8, NT>(p.csize) || 2 * clusters * p.csize <= sm_count();
    a.early = overlap_enabled() && overlap && !consume_pack(st) ? 1 : 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters * p.csize);
    cfg.blockDim = dim3(f.warps * 32);
    cfg.dynamicSmemBytes = a.at.total;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = p.csize;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, gemm7_kernel<FMT, INT8, NT>, a);
    if (e != cudaSuccess) { set_last_cuda_error(e); (void)cudaGetLastError(); return PTQTP_ERR_CUDA; }
    return PTQTP_OK;
}

template <int FMT, bool INT8>
ptqtp_status run7(Args7 a, int m, const uint16_t* X, uint16_t* Y, cudaStream_t st) {
    int* status_word = nullptr;                           // shared with the GEMV kernels (ptqtp_kernel_status)
    if (gemv_status_word(&status_word) != PTQTP_OK) return PTQTP_ERR_CUDA;
    constexpr int ROWS = INT8 ? 4 : 8;
    const Plan7 p = plan7<FMT, INT8>(a.all_tiles, a.sbs);
    auto lg = [](int v) { return v == 1 ? 0 : v == 2 ? 1 : v == 4 ? 2 : 3; };
    a.lg_csize = lg(p.csize);
    a.lg_kw = lg(p.kw);
    a.s_base = p.blocks / p.csize;
    a.s_rem = p.blocks % p.csize;
    a.spin_limit = wait_poll_limit();
    a.status_word = status_word;
    const Fit7 f = fit7<FMT, INT8>(p, m);
    const int own_cap = (f.per_cluster + p.csize - 1) / p.csize;
    const int tiles_per_launch = f.per_cluster * p.clusters;
    const int launches = (m + ROWS * f.nt - 1) / (ROWS * f.nt);
    for (int tile0 = 0; tile0 < a.all_tiles; tile0 += tiles_per_launch) {
        a.tile0 = tile0;
        const int tiles = min(tiles_per_launch, a.all_tiles - tile0), clusters = min(p.clusters, tiles);
        a.t_base = tiles / clusters;
        a.t_rem = tiles % clusters;
        for (int i = 0, done = 0; i < launches; ++i) {
            const int rows = (m - done + launches - i - 1) / (launches - i), ntl = (rows + ROWS - 1) / ROWS;
            a.X = reinterpret_cast<const __half*>(X) + (size_t)done * a.k;
            a.Y = reinterpret_cast<__half*>(Y) + (size_t)done * a.n;
            a.m = rows;
            a.inject = take_injected_wait_failure() ? 1 : 0;
            a.at = smem7(FMT, INT8, ROWS * ntl, f.warps, f.chunk, own_cap, p.csize * p.kw, f.rounds * f.warps);
            const ptqtp_status s = ntl == 1 ? launch_nt7<FMT, INT8, 1>(a, p, f, clusters, st)
                                 : ntl == 2 ? launch_nt7<FMT, INT8, 2>(a, p, f, clusters, st)
                                 : ntl == 3 ? launch_nt7<FMT, INT8, 3>(a, p, f, clusters, st)
                                            : launch_nt7<FMT, INT8, 4>(a, p, f, clusters, st);
            if (s != PTQTP_OK) return s;
            done += rows;
        }
    }
    return PTQTP_OK;
}

bool one_launch7(int fmt, bool int8, int tiles, int sbs, int m) {
    const Fit7 f = fmt == 2 ? fit7<2, true>(plan7<2, true>(tiles, sbs), m)
                 : int8 ? fit7<3, true>(plan7<3, true>(tiles, sbs), m) : fit7<3, false>(plan7<3, false>(tiles, sbs), m);
    return m <= f.nt * (int8 ? 4 : 8);
}

}  // namespace

bool gemm7_one_launch(const Layout3& L, int m, bool int8) { return one_launch7(3, int8, L.nrb, L.sbs, m); }
bool gemm7_one_launch(const Layout2& L, int m) {
    return one_launch7(2, true, (L.nrp + kTileRp3 - 1) / kTileRp3, (L.k + kSuper3 - 1) / kSuper3, m);
}
// Clusters of eight CTAs (15 of them find room: 28 SMs idle) whose ranks have unequal shares of the slices: the other kernels on format
// 2 are faster there (14 slices: 8192 x 28672 at 2 rows 46 us against 40 on the register-stationary kernel, at 8 rows 67 against
// 62 on the workspace kernel; 16384 x 28672 85 against 78 and 129 against 103; 16 slices: 8192 x 32768 46 against 51, 65
// against 68).
bool gemm7_uneven(const Layout2& L) {
    if (L.slices <= 8 || L.slices % 8 == 0) return false;
    return plan7<2, true>((L.nrp + kTileRp3 - 1) / kTileRp3, (L.k + kSuper3 - 1) / kSuper3).csize == 8;
}

// What a call takes in a chain at level 0, where another kernel could take it: 9 to 16 rows of format 2, 17 to 32 rows of format 3 in
// fp16.  Start, a cluster's meeting, the activations of a rank, its tiles, bytes.  Within 6 % on average of 1254 calls on format 2, 7 %
// of 837 on format 3, 128 to 28672 rows by 256 to 28672 columns.
double gemm7_us(const Layout2& L, int m) {
    const int tiles = (L.nrp + kTileRp3 - 1) / kTileRp3, sbs = (L.k + kSuper3 - 1) / kSuper3;
    const Plan7 p = plan7<2, true>(tiles, sbs);
    const Fit7 f = fit7<2, true>(p, m);
    const int launches = (m + 4 * f.nt - 1) / (4 * f.nt), share = min(p.share, sbs), units = p.per_cluster * (p.share / 4);
    const double mb = 1e-6 * (double)L.total, c = p.csize > 1 ? 1.0 : 0.0;
    return launches * ((m + launches - 1) / launches <= 12 ? 2.0 + 0.47 * c + 0.56 * share + 0.53 * units + 0.27 * mb
                                                           : 1.65 + 0.69 * c + 0.67 * share + 0.73 * units + 0.33 * mb);
}
double gemm7_us(const Layout3& L, int m) {
    const Plan7 p = plan7<3, false>(L.nrb, L.sbs);
    const Fit7 f = fit7<3, false>(p, m);
    const int tw = max(1, f.warps / p.kw), units = (f.per_cluster + tw - 1) / tw * ((p.share + p.kw - 1) / p.kw);
    const int groups = min(4 * p.share, L.k / kGroup), per = p.per_cluster;
    const double mb = 1e-6 * (double)L.total, c = p.csize > 1 ? 1.0 : 0.0;
    return m <= 24 ? 1.45 + 0.55 * c + 0.19 * groups + 0.92 * units + 0.28 * per + 0.35 * mb
                   : 1.85 + 0.45 * c + 0.185 * groups + 0.97 * units + 0.23 * per + 0.64 * mb;
}

// 1 <= m <= 64 rows of X (16-byte aligned).
ptqtp_status launch_gemm7(const Layout3& L, const void* packed, int m, const uint16_t* X, uint16_t* Y, bool int8, cudaStream_t st) {
    if (m < 1 || m > 64) return PTQTP_ERR_SHAPE;
    Args7 a = {};
    a.codes = static_cast<const unsigned char*>(packed) + L.codes_off;
    a.n = L.n; a.k = L.k; a.nrp = L.nrp; a.all_tiles = L.nrb; a.sbs = L.sbs;
    return int8 ? run7<3, true>(a, m, X, Y, st) : run7<3, false>(a, m, X, Y, st);
}

ptqtp_status launch_gemm7(const Layout2& L, const void* packed, int m, const uint16_t* X, uint16_t* Y, cudaStream_t st) {
    if (m < 1 || m > 64) return PTQTP_ERR_SHAPE;
    Args7 a = {};
    a.codes = static_cast<const unsigned char*>(packed) + L.codes_off;
    a.n = L.n; a.k = L.k; a.nrp = L.nrp; a.all_tiles = (L.nrp + kTileRp3 - 1) / kTileRp3; a.sbs = (L.k + kSuper3 - 1) / kSuper3;
    a.slices = L.slices; a.last_active = L.last_active; a.last_unit = L.last_unit;
    return run7<2, true>(a, m, X, Y, st);
}

}  // namespace ptqtp
