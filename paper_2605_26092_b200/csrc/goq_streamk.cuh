// Even split of a layer's units (128 output channels x one 128-wide k-block) over the CTAs of a launch, and the deterministic
// sum of the channel tiles that several CTAs share; used by the tensor-core kernels for few tokens.
//
// Units are numbered token tile by token tile, channel tile by channel tile, k-block by k-block; CTA c of G takes
// [U c / G, U (c+1) / G). A CTA parks the part of a tile it has only a share of (its range's first and last tile at most) as fp32
// [token][128 channels] in scratch; `finish_kernel`, launched behind as a programmatic dependent, adds the parts of every shared
// tile in CTA order and stores. (Adding in the CTA that came last instead needs no second launch, but leaves the sum of a tile to
// one SM: 1024 x 8192 at 256 tokens, where eight tiles have 19 parts of 128 KB each, took 71 us, now 28.)
#pragma once
#include "goq_tc_core.cuh"

namespace goq {
namespace streamk {

constexpr int kTileN = 128;   // output channels of a unit

__device__ __forceinline__ int range_begin(int c, int units, int n_ctas) { return (int)((long long)units * c / n_ctas); }

// A part: a run of k-blocks of one tile inside a CTA's range
struct Part { int tile, kb, n; };
__device__ __forceinline__ Part part_at(int u, int u1, int k_blocks) {
    Part p;
    p.tile = u / k_blocks;
    p.kb = u - p.tile * k_blocks;
    p.n = min(k_blocks - p.kb, u1 - u);
    return p;
}

// y[token][channel..channel + 3], vector stores where the output allows them
struct Output {
    void* y;
    int y_dtype, n_out;
    __device__ __forceinline__ void store4(int tok, int ch, float4 f) const {
        const size_t o = (size_t)tok * n_out + ch;
        const bool f32 = y_dtype == GOQ_F32;
        const bool vec = ch + 4 <= n_out && (n_out & 3) == 0 && (reinterpret_cast<uintptr_t>(y) & (f32 ? 15u : 7u)) == 0;
        if (f32) {
            float* d = reinterpret_cast<float*>(y);
            if (vec) *reinterpret_cast<float4*>(d + o) = f;
            else {
                if (ch + 0 < n_out) d[o + 0] = f.x;
                if (ch + 1 < n_out) d[o + 1] = f.y;
                if (ch + 2 < n_out) d[o + 2] = f.z;
                if (ch + 3 < n_out) d[o + 3] = f.w;
            }
        } else {
            uint16_t* d = reinterpret_cast<uint16_t*>(y);
            const uint32_t h01 = tc::pack_bf16x2(f.x, f.y), h23 = tc::pack_bf16x2(f.z, f.w);
            if (vec) *reinterpret_cast<uint2*>(d + o) = make_uint2(h01, h23);
            else {
                if (ch + 0 < n_out) d[o + 0] = (uint16_t)(h01 & 0xFFFFu);
                if (ch + 1 < n_out) d[o + 1] = (uint16_t)(h01 >> 16);
                if (ch + 2 < n_out) d[o + 2] = (uint16_t)(h23 & 0xFFFFu);
                if (ch + 3 < n_out) d[o + 3] = (uint16_t)(h23 >> 16);
            }
        }
    }
    __device__ __forceinline__ void store1(int tok, int ch, float f) const {
        const size_t o = (size_t)tok * n_out + ch;
        if (y_dtype == GOQ_F32) reinterpret_cast<float*>(y)[o] = f;
        else reinterpret_cast<uint16_t*>(y)[o] = (uint16_t)(tc::pack_bf16x2(f, 0.f) & 0xFFFFu);
    }
};

struct FinishParams {
    const float* partial;   // [CTA][2][n_cols][128]: a CTA's first part, its last one
    const float* scale;     // per-token factor of the sums
    void* y;
    int y_dtype, n_out, m, n_cols, tiles_x, k_blocks, units, n_ctas;
};
constexpr int kFinishThreads = 256, kFinishTokens = 16;   // of a CTA: 16 tokens of a tile, two tokens x four channels a thread

// grid: (channel tiles x token tiles, token slices). Bound by the parts' way through L2. `after_wait`: called once the kernels before are complete;
// gives the slice's tokens whose sums are not wanted, a bit each.
template <class F>
__device__ __forceinline__ void finish_tile(const FinishParams& p, F&& after_wait) {
    const int tile = blockIdx.x, ch = (threadIdx.x & 31) * 4;
    // the CTAs that share the tile, and where the first of them keeps its part (every other one starts inside the tile, so it is
    // that CTA's first)
    const int c_lo = (int)((((long long)tile * p.k_blocks + 1) * p.n_ctas - 1) / p.units);
    const int c_hi = (int)((((long long)(tile + 1) * p.k_blocks) * p.n_ctas - 1) / p.units);
    const int slot = range_begin(c_lo, p.units, p.n_ctas) == tile * p.k_blocks ? 0 : 1;
    const int tok0 = (tile / p.tiles_x) * p.n_cols, cols = min(p.n_cols, p.m - tok0);
    const int col = blockIdx.y * kFinishTokens + (threadIdx.x >> 5);
    const int col2 = min(col + kFinishTokens / 2, cols - 1);
    const size_t park = (size_t)p.n_cols * kTileN, stride = 2 * park;
    const float* lo = p.partial + ((size_t)c_lo * 2 + slot) * park + ch;
    const float* rest = p.partial + (size_t)(c_lo + 1) * stride + ch;
    // Every CTA waits, also one that finds nothing to add: what follows on the stream is ordered behind this grid alone, and a grid of
    // CTAs that return at once would be complete while the kernel before it still runs.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t skip = after_wait();
    if (c_lo == c_hi || col >= cols) return;   // one CTA had the whole tile and has stored it; no such token
    float4 f0 = __ldcg(reinterpret_cast<const float4*>(lo + (size_t)col * kTileN));
    float4 f1 = __ldcg(reinterpret_cast<const float4*>(lo + (size_t)col2 * kTileN));
    const float s0 = __ldcg(p.scale + tok0 + col), s1 = __ldcg(p.scale + tok0 + col2);
#pragma unroll 8
    for (int c = c_lo + 1; c <= c_hi; ++c, rest += stride) {   // CTA order
        const float4 a = __ldcg(reinterpret_cast<const float4*>(rest + (size_t)col * kTileN));
        const float4 b = __ldcg(reinterpret_cast<const float4*>(rest + (size_t)col2 * kTileN));
        f0.x += a.x; f0.y += a.y; f0.z += a.z; f0.w += a.w;
        f1.x += b.x; f1.y += b.y; f1.z += b.z; f1.w += b.w;
    }
    const Output out = {p.y, p.y_dtype, p.n_out};
    const int ch0 = (tile % p.tiles_x) * kTileN + ch;
    const int bit = threadIdx.x >> 5;
    if (!((skip >> bit) & 1u)) out.store4(tok0 + col, ch0, make_float4(f0.x * s0, f0.y * s0, f0.z * s0, f0.w * s0));
    if (col + kFinishTokens / 2 < cols && !((skip >> (bit + kFinishTokens / 2)) & 1u)) out.store4(tok0 + col2, ch0, make_float4(f1.x * s1, f1.y * s1, f1.z * s1, f1.w * s1));
}
static __global__ void __launch_bounds__(kFinishThreads) finish_kernel(const FinishParams p) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    finish_tile(p, [] { return 0u; });
}

}  // namespace streamk
}  // namespace goq
