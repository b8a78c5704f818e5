// Pack / unpack kernels of the PTQTP-B200 format 2 (layout described in ptqtp.h).
// A thread handles 16-byte atoms: 16 columns of one row pair, both planes.  Atoms are numbered along the rows, so that
// neighbouring lanes read neighbouring columns (numbered in storage order they would read every fourth 16 bytes).  Bound by memory: in a
// chain of calls 13506 x 4096 packs in 23.0 us and unpacks in 22.9 (24.8 and 22.9 with two atoms per packing thread, 24.6 and 22.9 with
// that, CTAs of 256 threads and plain launches; 43.7 and 42.5 for 14336 x 4096 with atoms in storage order, a division in 64 bits for each and
// byte-wise coding).  Streaming stores of the blob would bring 2 %, but who reads it next finds it in L2 without them (a call of
// ptqtp_unpack right after 55 us with the host's part, 61 from memory).
#include "trit_bytes.h"

namespace ptqtp {

namespace {

constexpr int kThreadsP2 = 128;

__device__ __forceinline__ int active_of(const Layout2& L, int slice) {
    return slice == L.slices - 1 ? L.last_active : 32;
}

// Row pair and column of an atom, numbered row pair by row pair along the columns.  I: an index type that holds the number of
// atoms (32 bits where they do: the division is a tenth of the cost).
template <class I, int A>
__device__ __forceinline__ bool atom_of(const Layout2& L, int nth, int& rp, int& col) {
    const I a = (I)blockIdx.x * (kThreadsP2 * A) + nth * kThreadsP2 + threadIdx.x, per_rp = (I)(L.k / 16);
    const I q = a / per_rp;
    rp = (int)q;
    col = 16 * (int)(a - q * per_rp);
    return q < (I)L.nrp;
}
// Byte offset of the atom from the start of the codes: atom (i, l) is columns 64 l + 16 i of its slice.
__device__ __forceinline__ size_t atom_offset(const Layout2& L, int rp, int col) {
    const int slice = col / kSlice2, c = col % kSlice2;
    return unit_offset(L, rp, slice) + (size_t)((c / 16 % 4) * active_of(L, slice) + c / kLane2) * 16;
}

template <class I>
__global__ void __launch_bounds__(kThreadsP2)
pack2_kernel(Layout2 L, const int8_t* __restrict__ T1, const int8_t* __restrict__ T2, const uint16_t* __restrict__ a1,
             const uint16_t* __restrict__ a2, unsigned char* __restrict__ packed, int32_t* dev_status) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    in_order(T1, T2, a1, a2);
    unsigned char* codes = packed + L.codes_off;
    bool bad = false;

    int rp, col;
    if (atom_of<I, 1>(L, 0, rp, col)) {
        uint4 v[4];                                // (row, plane 1), (row, plane 2), (row + 1, plane 1), (row + 1, plane 2)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const bool in = 2 * rp + r < L.n;
            const size_t at = (size_t)(2 * rp + r) * L.k + col;
            v[2 * r] = in ? __ldcs(reinterpret_cast<const uint4*>(T1 + at)) : make_uint4(0u, 0u, 0u, 0u);
            v[2 * r + 1] = in ? __ldcs(reinterpret_cast<const uint4*>(T2 + at)) : make_uint4(0u, 0u, 0u, 0u);
        }
        *reinterpret_cast<uint4*>(codes + atom_offset(L, rp, col)) = pair_words(v[0], v[1], v[2], v[3], bad);
    }

    // scale quads: one per row pair and 128-column group, after the codes of their slice unit
    const int groups = L.k / kGroup;
    const size_t n_quads = (size_t)L.nrp * groups;
    for (size_t q = tid; q < n_quads; q += stride) {
        const int rp = (int)(q / groups), g = (int)(q % groups);
        const int slice = g / 16, gl = g % 16;
        const int active = active_of(L, slice);
        uint16_t s[4] = {0, 0, 0, 0};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int row = 2 * rp + r;
            if (row < L.n) {
                s[2 * r] = __ldcg(a1 + (size_t)row * groups + g);
                s[2 * r + 1] = __ldcg(a2 + (size_t)row * groups + g);
            }
        }
        unsigned char* dst = codes + unit_offset(L, rp, slice) + (size_t)active * 64 + gl * 8;
        *reinterpret_cast<uint2*>(dst) = make_uint2((uint32_t)s[0] | ((uint32_t)s[1] << 16),
                                                    (uint32_t)s[2] | ((uint32_t)s[3] << 16));
    }

    // padding bytes at the end of a last unit whose content is not a multiple of 16 bytes
    const int last_content = L.last_active * 64 + L.last_active * 4;
    if (last_content < L.last_unit) {
        for (size_t rp = tid; rp < (size_t)L.nrp; rp += stride) {
            unsigned char* dst = codes + unit_offset(L, (int)rp, L.slices - 1);
            for (int b = last_content; b < L.last_unit; ++b) dst[b] = 0;
        }
    }

    if (blockIdx.x == 0 && threadIdx.x < PTQTP_HEADER_BYTES / 4) {
        Header h;
        const char m[8] = {'P', 'T', 'Q', 'T', 'P', 'B', '2', '\0'};
        for (int i = 0; i < 8; ++i) h.magic[i] = m[i];
        h.version = kVersion; h.format = PTQTP_FORMAT_V2;
        h.n = L.n; h.k = L.k; h.group = kGroup; h.k_pad = L.slices * kSlice2;
        h.codes_off = L.codes_off; h.scales_off = L.strip; h.total = L.total;
        const uint32_t* hw = reinterpret_cast<const uint32_t*>(&h);
        const int i = threadIdx.x;
        reinterpret_cast<uint32_t*>(packed)[i] = i < (int)(sizeof(Header) / 4) ? hw[i] : 0u;
    }
    if (bad && dev_status) atomicExch(dev_status, (int)PTQTP_ERR_TRIT);
}

template <class I, int A>
__global__ void __launch_bounds__(kThreadsP2)
unpack2_kernel(Layout2 L, const unsigned char* __restrict__ packed, int8_t* __restrict__ T1, int8_t* __restrict__ T2,
               uint16_t* __restrict__ a1, uint16_t* __restrict__ a2, int32_t* dev_status) {
    in_order(packed);
    if (blockIdx.x == 0 && threadIdx.x == 0 && dev_status) {
        const Header* h = reinterpret_cast<const Header*>(packed);
        const char m[8] = {'P', 'T', 'Q', 'T', 'P', 'B', '2', '\0'};
        bool ok = h->version == kVersion && h->format == PTQTP_FORMAT_V2 && h->n == L.n && h->k == L.k &&
                  h->group == kGroup && h->k_pad == L.slices * kSlice2 && h->codes_off == L.codes_off &&
                  h->scales_off == L.strip && h->total == L.total;
        for (int i = 0; i < 8; ++i) ok = ok && h->magic[i] == m[i];
        if (!ok) atomicExch(dev_status, (int)PTQTP_ERR_FORMAT);
    }
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned char* codes = packed + L.codes_off;

    int rp[A], col[A];
    bool live[A];
    uint4 w[A];
#pragma unroll
    for (int n = 0; n < A; ++n) {
        live[n] = atom_of<I, A>(L, n, rp[n], col[n]);
        if (live[n]) w[n] = __ldcs(reinterpret_cast<const uint4*>(codes + atom_offset(L, rp[n], col[n])));
    }
#pragma unroll
    for (int n = 0; n < A; ++n)
#pragma unroll
        for (int r = 0; r < 2; ++r)
            if (live[n] && 2 * rp[n] + r < L.n) {
                const size_t at = (size_t)(2 * rp[n] + r) * L.k + col[n];
                __stcs(reinterpret_cast<uint4*>(T1 + at), trits_of(w[n], 2 * r));
                __stcs(reinterpret_cast<uint4*>(T2 + at), trits_of(w[n], 2 * r + 1));
            }

    const int groups = L.k / kGroup;
    const size_t n_quads = (size_t)L.nrp * groups;
    for (size_t q = tid; q < n_quads; q += stride) {
        const int rp = (int)(q / groups), g = (int)(q % groups);
        const int slice = g / 16, gl = g % 16;
        const int active = active_of(L, slice);
        const uint2 s = __ldcg(reinterpret_cast<const uint2*>(codes + unit_offset(L, rp, slice) + (size_t)active * 64 + gl * 8));
        const uint32_t v[2] = {s.x, s.y};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int row = 2 * rp + r;
            if (row < L.n) {
                a1[(size_t)row * groups + g] = (uint16_t)(v[r] & 0xffffu);
                a2[(size_t)row * groups + g] = (uint16_t)(v[r] >> 16);
            }
        }
    }
}

// One grid for all atoms; the scale quads (an eighth as many) are strided over it.
unsigned ctas_for2(const Layout2& L, int atoms) {
    const size_t per_cta = (size_t)kThreadsP2 * atoms;
    return (unsigned)(((size_t)L.nrp * (L.k / 16) + per_cta - 1) / per_cta);
}
bool index32_2(const Layout2& L) { return (size_t)L.nrp * (L.k / 16) < ((size_t)1 << 32) - 2 * kThreadsP2; }
constexpr unsigned kResident2 = 16;                // CTAs per SM: 128 threads of 32 registers at most

// Packing as a dependent launch: where the CTAs of two launches find room beside each other (468 x 4096 2.7 us instead of 3.1), and from three
// waves on (8054 x 4096 13.6 instead of 14.0).  In between the next launch's CTAs leave no room for the rest of this one's
// or start unevenly: 1438 x 4096 4.8 us against 4.1 with plain launches, 9195 x 640 6.3 and 4.6, 28195 x 640 11.9 and 8.9 (with K a
// multiple of 2048 dependent launches would be the better ones again from one wave on, 3708 x 4096 7.0 and 7.4).
bool pack_dependent2(unsigned ctas) {
    const unsigned wave = kResident2 * (unsigned)sm_count();
    return 2 * ctas <= wave || ctas >= 3 * wave;
}
// Unpacking: two atoms per thread where each SM gets two CTAs or more and the CTAs of two launches find room beside each other (860 x 6272
// 3.8 us instead of 4.2), and from a wave and a half on (8778 x 4096 11.8 and 12.2); one in between (2410 x 4096 4.5, with two atoms 5.6)
// and below (191 x 1024 2.6 and 2.9).  (Packing takes one everywhere: 1860 x 4096 4.6 with one, 5.4 with two, 13506 x 4096 23.0 and 24.8.)
bool two_atoms2(const Layout2& L) {
    const unsigned sms = (unsigned)sm_count(), wave = kResident2 * sms, ctas = ctas_for2(L, 2);
    return ctas >= 2 * sms && (2 * ctas <= wave || 2 * ctas >= 3 * wave);
}

}  // namespace

ptqtp_status launch_pack2(const Layout2& L, const int8_t* T1, const int8_t* T2, const uint16_t* a1,
                          const uint16_t* a2, void* packed, int32_t* dev_status, cudaStream_t st) {
    const unsigned ctas = ctas_for2(L, 1);
    return launch_in_order_if(pack_dependent2(ctas), index32_2(L) ? pack2_kernel<uint32_t> : pack2_kernel<size_t>, ctas, kThreadsP2, 0, st, L, T1, T2, a1, a2,
                              static_cast<unsigned char*>(packed), dev_status);
}

ptqtp_status launch_unpack2(const Layout2& L, const void* packed, int8_t* T1, int8_t* T2, uint16_t* a1,
                            uint16_t* a2, int32_t* dev_status, cudaStream_t st) {
    const bool two = two_atoms2(L);
    auto kern = !two ? unpack2_kernel<uint32_t, 1> : index32_2(L) ? unpack2_kernel<uint32_t, 2> : unpack2_kernel<size_t, 2>;
    return launch_in_order(kern, ctas_for2(L, two ? 2 : 1), kThreadsP2, 0, st, L, static_cast<const unsigned char*>(packed), T1, T2, a1, a2, dev_status);
}

}  // namespace ptqtp
