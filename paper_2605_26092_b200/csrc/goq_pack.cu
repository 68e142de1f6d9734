// goq_pack / goq_unpack kernels: quantizer output <-> the tile16 packed layout.
// The fields are those of Sections 3.2-3.4 of the paper (code per weight, 6-bit exchange record
// per 8 weights, fp16 coefficient pair per macro-block); unpack also derives b2 the way
// Section 3.3 (Theorem 1) defines it, so tests can compare it with an independent decode.
#include "goq_common.cuh"
#include "goq_internal.h"

namespace goq {

// One warp per half record (8 rows x 128 k): lane (g, t) packs the four words 4 lane .. 4 lane + 3, which are consecutive in the
// record (row g, micro-blocks t, 4 + t, 8 + t, 12 + t), and stores them with one 16-byte store, 512 bytes a warp; its loads of
// the codes take whole 32-byte sectors (four lanes x 8 bytes of a row). The warp also writes its rows' coefficient pairs. One
// launch; bound by memory: codes, records and pairs in, the record out.
// VEC: the code rows are 8-byte aligned (k_in is a multiple of 8, so it is up to the array's address).
constexpr int kPackWarps = 8;
template <int WB, bool VEC>
__global__ void __launch_bounds__(kPackWarps * 32)
pack_kernel(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ meta, const uint16_t* __restrict__ coef,
            uint8_t* __restrict__ packed, int n_out, int k_in, int k_blocks, long long n_half, int group_log2, int unit_bytes,
            int meta_off, int k1) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const long long id = (long long)blockIdx.x * kPackWarps + (threadIdx.x >> 5);
    if (id >= n_half) return;
    // half-records are numbered tile by tile, half by half, k-block by k-block: neighbouring warps read neighbouring columns
    const long long th = id / k_blocks;
    const int bk = (int)(id - th * k_blocks), v = (int)(th & 1), row0 = (int)(th >> 1) * kTileRows + 8 * v, row = row0 + g;
    uint8_t* unit = packed + ((th >> 1) * k_blocks + bk) * (long long)unit_bytes;
    constexpr uint32_t kZero = (1u << (WB - 1)) - 1u, kMask = ((1u << WB) - 1u) * 0x01010101u;
    uint32_t word[4], rec[4];
    const bool row_in = row < n_out;
    const uint8_t* row_meta = meta + (size_t)row * (k_in / 8) + bk * (kBlockK / 8);
    uint32_t mw[4] = {0u, 0u, 0u, 0u};   // the row's 16 records of this k-block, where they are one aligned load
    const bool meta16 = VEC && (k_in & (kBlockK - 1)) == 0 && (reinterpret_cast<uintptr_t>(meta) & 15u) == 0;
    if (meta16 && row_in) {
        const uint4 q = *reinterpret_cast<const uint4*>(row_meta);
        mw[0] = q.x; mw[1] = q.y; mw[2] = q.z; mw[3] = q.w;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int mb = bk * (kBlockK / 8) + 4 * c + t;
        uint32_t lo = kZero * 0x01010101u, hi = lo, m = 0;
        if (row_in && mb * 8 < k_in) {
            const uint8_t* src = codes + (size_t)row * k_in + (size_t)mb * 8;
            if constexpr (VEC) {
                const uint2 q = __ldcs(reinterpret_cast<const uint2*>(src));
                lo = q.x; hi = q.y;
            } else {
                lo = src[0] | (src[1] << 8) | (src[2] << 16) | ((uint32_t)src[3] << 24);
                hi = src[4] | (src[5] << 8) | (src[6] << 16) | ((uint32_t)src[7] << 24);
            }
            m = k1 ? 0u : (meta16 ? mw[c] >> (8 * t) : (uint32_t)row_meta[4 * c + t]) & 63u;   // single-basis weights carry no exchange record
        }
        lo &= kMask; hi &= kMask;
        lo |= lo >> 4; hi |= hi >> 4;                               // bytes -> nibbles
        word[c] = __byte_perm(lo, hi, 0x6420);
        rec[c] = m;
        if constexpr (WB <= 3) word[c] |= scatter_meta(m);
    }
    reinterpret_cast<uint4*>(unit)[v * 32 + lane] = make_uint4(word[0], word[1], word[2], word[3]);
    if constexpr (WB == 4)
        *reinterpret_cast<uint32_t*>(unit + meta_off + v * 128 + lane * 4) = rec[0] | (rec[1] << 8) | (rec[2] << 16) | (rec[3] << 24);
    const int gpb = kBlockK >> group_log2, groups_in = k_in >> group_log2;
    for (int i = lane; i < 8 * gpb; i += 32) {   // pair jj of row r at word jj * 16 + r of the coefficient plane
        const int jj = i >> 3, r = i & 7, j = bk * gpb + jj;
        uint32_t cf = 0;
        if (row0 + r < n_out && j < groups_in) {
            const uint16_t* c = coef + ((size_t)(row0 + r) * groups_in + j) * 2;
            cf = (uint32_t)c[0] | (k1 ? 0u : ((uint32_t)c[1] << 16));   // single-basis weights: c2 = 0
        }
        reinterpret_cast<uint32_t*>(unit + kCodeBytesPerUnit)[jj * 16 + 8 * v + r] = cf;
    }
}

__global__ void unpack_kernel(const uint8_t* __restrict__ packed, uint8_t* __restrict__ codes_b1,
                              uint8_t* __restrict__ codes_b2, int n_out, int k_in, int k_pad, int wbits,
                              int unit_bytes, int meta_off) {
    const int mbs = k_in / 8;
    size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)n_out * mbs) return;
    int row = (int)(idx / mbs), mb = (int)(idx % mbs);
    const uint8_t* unit = packed + unit_offset(row >> 4, mb >> 4, k_pad / kBlockK, unit_bytes);
    const int wi = word_in_unit(row, mb);
    uint32_t w = reinterpret_cast<const uint32_t*>(unit)[wi];
    uint32_t m = (wbits <= 3) ? gather_meta(w) : (uint32_t)unit[meta_off + wi];
    const uint32_t cmask = (wbits <= 3) ? 0x77777777u : 0xFFFFFFFFu;
    uint32_t cw = w & cmask;
    const uint32_t emax = (1u << (wbits - 1)) - 1u;
    size_t o = (size_t)row * k_in + (size_t)mb * 8;
    if (codes_b1) {
#pragma unroll
        for (int i = 0; i < 8; ++i) codes_b1[o + i] = (uint8_t)((cw >> (4 * i)) & 15u);
    }
    if (codes_b2) {
        int s = (int)(m & 3u) + 1;
        uint32_t src = xor_permute_nibbles(cw, s);
        uint32_t flips = flip_mask(m);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            uint32_t c = (src >> (4 * i)) & 15u;
            uint32_t sign = c >> (wbits - 1), e = c & emax;
            uint8_t out;
            if (sign == 0 && e == emax) out = 0x80;
            else out = (uint8_t)(((sign ^ ((flips >> i) & 1u)) << 3) | e);
            codes_b2[o + i] = out;
        }
    }
}

__global__ void unpack_coef_kernel(const uint8_t* __restrict__ packed, uint16_t* __restrict__ coef, int n_out,
                                   int groups_in, int gpb, int k_blocks, int unit_bytes) {
    size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)n_out * groups_in) return;
    int row = (int)(idx / groups_in), j = (int)(idx % groups_in);
    const uint8_t* unit = packed + unit_offset(row >> 4, j / gpb, k_blocks, unit_bytes);
    uint32_t v = reinterpret_cast<const uint32_t*>(unit + kCodeBytesPerUnit)[(j % gpb) * 16 + (row & 15)];
    coef[idx * 2] = (uint16_t)(v & 0xFFFFu);
    coef[idx * 2 + 1] = (uint16_t)(v >> 16);
}

template <int WB>
static void launch_pack_wb(const Geometry& g, const uint8_t* codes, const uint8_t* meta, const uint16_t* coef, uint8_t* base,
                           cudaStream_t st) {
    const long long n_half = (long long)g.n_units * 2;
    const unsigned blocks = (unsigned)((n_half + kPackWarps - 1) / kPackWarps);
    int lg = 3;
    while ((1 << lg) < g.group) ++lg;
    if ((reinterpret_cast<uintptr_t>(codes) & 7u) == 0)
        pack_kernel<WB, true><<<blocks, kPackWarps * 32, 0, st>>>(codes, meta, coef, base, g.n_out, g.k_in, g.k_blocks, n_half, lg,
                                                                  g.unit_bytes, g.meta_off, g.k1);
    else
        pack_kernel<WB, false><<<blocks, kPackWarps * 32, 0, st>>>(codes, meta, coef, base, g.n_out, g.k_in, g.k_blocks, n_half, lg,
                                                                   g.unit_bytes, g.meta_off, g.k1);
}

cudaError_t launch_pack(const Geometry& g, const uint8_t* codes, const uint8_t* meta, const uint16_t* coef,
                        void* packed, cudaStream_t st) {
    auto* base = (uint8_t*)packed;
    if (g.wbits == 2) launch_pack_wb<2>(g, codes, meta, coef, base, st);
    else if (g.wbits == 3) launch_pack_wb<3>(g, codes, meta, coef, base, st);
    else launch_pack_wb<4>(g, codes, meta, coef, base, st);
    return cudaGetLastError();
}

cudaError_t launch_unpack(const Geometry& g, const void* packed, uint8_t* b1, uint8_t* b2, uint16_t* coef,
                          cudaStream_t st) {
    auto* base = (const uint8_t*)packed;
    if (b1 || b2) {
        size_t n = (size_t)g.n_out * (g.k_in / 8);
        unpack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(base, b1, b2, g.n_out, g.k_in, g.k_pad, g.wbits,
                                                                  g.unit_bytes, g.meta_off);
    }
    if (coef) {
        size_t n = (size_t)g.n_out * (g.k_in / g.group);
        unpack_coef_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(base, coef, g.n_out, g.k_in / g.group,
                                                                       g.groups_per_block, g.k_blocks, g.unit_bytes);
    }
    return cudaGetLastError();
}

}  // namespace goq
