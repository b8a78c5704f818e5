// Pack / unpack kernels of the PTQTP-B200 format 3 (layout described in ptqtp.h).
// A run of 16 columns of one scale group is two words of each of two neighbouring lane entries, so a thread takes a row pair,
// chunk and group pair of a tile: eight 16-byte loads (two rows, two planes, the two groups of the pair), 32
// contiguous bytes of the blob.  Eight lanes cover 128 contiguous bytes of a row.  Bound by memory: 14336 x 4096
// packs in 26.7 us and unpacks in 25.6 (5.6 and 5.9 TB/s; 61.9 and 112 with four-byte accesses and byte-wise coding).  Packing takes a
// tile per CTA (two tiles 27.5; four 32.9; a loop of CTAs that stay, the next tile's loads in flight, 41; streaming stores of the blob
// 26.2, but who reads it next finds it in L2 without them); unpacking two (one tile: 25.4 there, but 4.2 against 3.9 on 1024 x 4096).
// Launched as dependents that wait first, mostly: call after call of the binding 27.1 us packing and 26.9 unpacking 14336 x 4096 (28.8 and 28.7 with
// plain launches).
#include "trit_bytes.h"

namespace ptqtp {

namespace {

constexpr int kTileThreads3 = 128, kThreadsPack3 = 128, kThreadsUnpack3 = 256;

// Thread -> tile (row block by row block, so that neighbours read the same rows), chunk, row pair, group pair.
struct Run3 {
    int sb, rb, c, g, u;
    size_t tile_off;                  // byte offset of the tile from the start of the codes
    bool live;
};
__device__ __forceinline__ Run3 run_of(const Layout3& L) {
    const size_t tile = (size_t)blockIdx.x * (blockDim.x / kTileThreads3) + threadIdx.x / kTileThreads3;
    const int r = threadIdx.x % kTileThreads3;
    Run3 p;
    p.rb = (int)(tile / L.sbs);
    p.sb = (int)(tile - (size_t)p.rb * L.sbs);
    p.c = r & 7;
    p.g = (r >> 3) & 7;
    p.u = r >> 6;
    p.live = p.rb < L.nrb;
    p.tile_off = tile_offset3(L, p.rb, p.sb);
    return p;
}

__global__ void __launch_bounds__(kThreadsPack3)
pack3_kernel(Layout3 L, const int8_t* __restrict__ T1, const int8_t* __restrict__ T2, const uint16_t* __restrict__ a1,
             const uint16_t* __restrict__ a2, unsigned char* __restrict__ packed, int32_t* dev_status) {
    in_order(T1, T2, a1, a2);
    unsigned char* codes = packed + L.codes_off;
    bool bad = false;
    const Run3 p = run_of(L);
    if (p.live) {
        const int row = 2 * (p.rb * kTileRp3 + p.g);
        uint4 v[2][4];                                   // [group u | 2 + u][(row, plane 1), (row, plane 2), (row + 1, ...)]
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int col = p.sb * kSuper3 + 128 * (2 * h + p.u) + 16 * p.c;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const bool in = row + r < L.n && col < L.k;      // K is a multiple of 128: a run is in or out
                const size_t at = (size_t)(row + r) * L.k + col;
                v[h][2 * r] = in ? __ldcs(reinterpret_cast<const uint4*>(T1 + at)) : make_uint4(0u, 0u, 0u, 0u);
                v[h][2 * r + 1] = in ? __ldcs(reinterpret_cast<const uint4*>(T2 + at)) : make_uint4(0u, 0u, 0u, 0u);
            }
        }
        const uint4 lo = pair_words(v[0][0], v[0][1], v[0][2], v[0][3], bad), hi = pair_words(v[1][0], v[1][1], v[1][2], v[1][3], bad);
        // entry t = 2 u: columns 0-3 and 8-11 of the run, t = 2 u + 1: columns 4-7 and 12-15; words (s, h)
        uint4* dst = reinterpret_cast<uint4*>(codes + p.tile_off + (p.c * 32 + 4 * p.g + 2 * p.u) * 16);
        dst[0] = make_uint4(lo.x, hi.x, lo.z, hi.z);
        dst[1] = make_uint4(lo.y, hi.y, lo.w, hi.w);
    }

    // scale quads: 32 per tile, quad 4 g + t = row pair g of the tile, group t of the superblock
    const int groups = L.k / kGroup, l = threadIdx.x % kTileThreads3;
    if (p.live && l < 32) {
        const int g = l >> 2, grp = 4 * p.sb + (l & 3);
        uint16_t s[4] = {0, 0, 0, 0};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int row = 2 * (p.rb * kTileRp3 + g) + r;
            if (row < L.n && grp < groups) {
                s[2 * r] = __ldcg(a1 + (size_t)row * groups + grp);
                s[2 * r + 1] = __ldcg(a2 + (size_t)row * groups + grp);
            }
        }
        *reinterpret_cast<uint2*>(codes + p.tile_off + kTileCodes3 + l * 8) =
            make_uint2((uint32_t)s[0] | ((uint32_t)s[1] << 16), (uint32_t)s[2] | ((uint32_t)s[3] << 16));
    }

    if (blockIdx.x == 0 && threadIdx.x < PTQTP_HEADER_BYTES / 4) {
        Header h;
        const char m[8] = {'P', 'T', 'Q', 'T', 'P', 'B', '2', '\0'};
        for (int i = 0; i < 8; ++i) h.magic[i] = m[i];
        h.version = kVersion; h.format = PTQTP_FORMAT_V3;
        h.n = L.n; h.k = L.k; h.group = kGroup; h.k_pad = L.sbs * kSuper3;
        h.codes_off = L.codes_off; h.scales_off = kTile3; h.total = L.total;
        const uint32_t* hw = reinterpret_cast<const uint32_t*>(&h);
        const int i = threadIdx.x;
        reinterpret_cast<uint32_t*>(packed)[i] = i < (int)(sizeof(Header) / 4) ? hw[i] : 0u;
    }
    if (bad && dev_status) atomicExch(dev_status, (int)PTQTP_ERR_TRIT);
}

__global__ void __launch_bounds__(kThreadsUnpack3)
unpack3_kernel(Layout3 L, const unsigned char* __restrict__ packed, int8_t* __restrict__ T1, int8_t* __restrict__ T2,
               uint16_t* __restrict__ a1, uint16_t* __restrict__ a2, int32_t* dev_status) {
    in_order(packed);
    if (blockIdx.x == 0 && threadIdx.x == 0 && dev_status) {
        const Header* h = reinterpret_cast<const Header*>(packed);
        const char m[8] = {'P', 'T', 'Q', 'T', 'P', 'B', '2', '\0'};
        bool ok = h->version == kVersion && h->format == PTQTP_FORMAT_V3 && h->n == L.n && h->k == L.k &&
                  h->group == kGroup && h->k_pad == L.sbs * kSuper3 && h->codes_off == L.codes_off &&
                  h->scales_off == (uint64_t)kTile3 && h->total == L.total;
        for (int i = 0; i < 8; ++i) ok = ok && h->magic[i] == m[i];
        if (!ok) atomicExch(dev_status, (int)PTQTP_ERR_FORMAT);
    }
    const unsigned char* codes = packed + L.codes_off;
    const Run3 p = run_of(L);
    if (p.live) {
        const int row = 2 * (p.rb * kTileRp3 + p.g);
        const uint4* src = reinterpret_cast<const uint4*>(codes + p.tile_off + (p.c * 32 + 4 * p.g + 2 * p.u) * 16);
        const uint4 e0 = __ldcs(src), e1 = __ldcs(src + 1);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int col = p.sb * kSuper3 + 128 * (2 * h + p.u) + 16 * p.c;
            const uint4 w = h ? make_uint4(e0.y, e1.y, e0.w, e1.w) : make_uint4(e0.x, e1.x, e0.z, e1.z);
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (row + r < L.n && col < L.k) {
                    const size_t at = (size_t)(row + r) * L.k + col;
                    __stcs(reinterpret_cast<uint4*>(T1 + at), trits_of(w, 2 * r));
                    __stcs(reinterpret_cast<uint4*>(T2 + at), trits_of(w, 2 * r + 1));
                }
        }
    }

    const int groups = L.k / kGroup, l = threadIdx.x % kTileThreads3, grp = 4 * p.sb + (l & 3);
    if (p.live && l < 32 && grp < groups) {
        const uint2 s = __ldcg(reinterpret_cast<const uint2*>(codes + p.tile_off + kTileCodes3 + l * 8));
        const uint32_t v[2] = {s.x, s.y};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int row = 2 * (p.rb * kTileRp3 + (l >> 2)) + r;
            if (row < L.n) {
                a1[(size_t)row * groups + grp] = (uint16_t)(v[r] & 0xffffu);
                a2[(size_t)row * groups + grp] = (uint16_t)(v[r] >> 16);
            }
        }
    }
}

// A plain launch where the CTAs of this launch fill between a half and three quarters of the device's places, so that only some of the
// next launch's find room beside them: packing 1708 x 4096 4.8 to 5.0 us, 5.2 as a dependent launch (469 x 4096 3.5 instead of 4.0, 2410 x 4096
// 5.4 instead of 5.6, 13506 x 4096 23.1 instead of 23.4), unpacking 2410 x 4096 5.2 and 6.6, 11196 x 640 4.4 and 5.4 (1860 x 4096 4.6
// instead of 4.8, 4042 x 4096 7.3 instead of 7.4, 13506 x 4096 23.2 instead of 23.6).  resident: CTAs per SM, by the registers.
bool dependent3(unsigned ctas, unsigned resident) {
    const unsigned wave = resident * (unsigned)sm_count();
    return 2 * ctas <= wave || 4 * ctas > 3 * wave;
}
constexpr unsigned kResidentPack3 = 10, kResidentUnpack3 = 8;      // 48 and 32 registers a thread
unsigned grid_for3(const Layout3& L, int threads) {
    const size_t per_cta = threads / kTileThreads3;
    return (unsigned)(((size_t)L.nrb * L.sbs + per_cta - 1) / per_cta);
}

}  // namespace

ptqtp_status launch_pack3(const Layout3& L, const int8_t* T1, const int8_t* T2, const uint16_t* a1,
                          const uint16_t* a2, void* packed, int32_t* dev_status, cudaStream_t st) {
    const unsigned grid = grid_for3(L, kThreadsPack3);
    return launch_in_order_if(dependent3(grid, kResidentPack3), pack3_kernel, grid, kThreadsPack3, 0, st, L, T1, T2, a1, a2, static_cast<unsigned char*>(packed),
                              dev_status);
}

ptqtp_status launch_unpack3(const Layout3& L, const void* packed, int8_t* T1, int8_t* T2, uint16_t* a1,
                            uint16_t* a2, int32_t* dev_status, cudaStream_t st) {
    const unsigned grid = grid_for3(L, kThreadsUnpack3);
    return launch_in_order_if(dependent3(grid, kResidentUnpack3), unpack3_kernel, grid, kThreadsUnpack3, 0, st, L, static_cast<const unsigned char*>(packed), T1, T2,
                              a1, a2, dev_status);
}

}  // namespace ptqtp
