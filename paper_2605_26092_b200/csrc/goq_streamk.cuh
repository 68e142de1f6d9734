// Even split of a layer's units (128 output channels x one 128-wide k-block) over the CTAs of a launch, and the deterministic
// sum of the channel tiles that several CTAs share; used by the tensor-core kernels for few tokens.
//
// Units are numbered token tile by token tile, channel tile by channel tile, k-block by k-block; CTA c of G takes
// [U c / G, U (c+1) / G). A CTA parks the part of a tile it has only a share of (its range's first and last tile at most) as fp32
// [token][128 channels] in scratch. At its end it counts itself in at both tiles; the CTA that comes last adds all parts in CTA
// order, with all its threads, and stores.
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

// device-scope fetch-add: releases this thread's earlier writes (and those ordered before it by a barrier), acquires the others'
__device__ __forceinline__ int atomic_add_acq_rel(int* addr, int v) {
    int old;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(addr), "r"(v) : "memory");
    return old;
}

// The range's first and last tile: the CTAs that share it, where the first of them keeps its part (every other sharer starts
// inside the tile, so it is that CTA's first part), and which channel quarters this CTA has to finish.
struct SharedTile { int tile, c_lo, c_hi, first_slot, last_of[4]; };

// Filled by lanes 0 and 1 of a warp that has time before the main loop (the divisions are slow).
__device__ __forceinline__ void describe_shared(SharedTile (&fin)[2], int lane, int u0, int u1, int units, int k_blocks, int n_ctas) {
    if (lane >= 2) return;
    const int tile = (lane ? u1 - 1 : u0) / k_blocks;
    const int c_lo = (int)((((long long)tile * k_blocks + 1) * n_ctas - 1) / units);
    fin[lane].tile = tile;
    fin[lane].c_lo = c_lo;
    fin[lane].c_hi = (int)((((long long)(tile + 1) * k_blocks) * n_ctas - 1) / units);
    fin[lane].first_slot = range_begin(c_lo, units, n_ctas) == tile * k_blocks ? 0 : 1;
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

// After the CTA's own work, by all its threads (contains barriers). park_floats: floats of one parked part, two parts a CTA.
// scale: per-token factor of the sums (nullptr: 1).
template <int THREADS>
__device__ __forceinline__ void finish_shared(SharedTile (&fin)[2], const float* partial, size_t park_floats, int* counters,
                                              int tiles_x, int n_cols, int m, const float* scale, const Output& out) {
    const int tid = threadIdx.x;
    if (tid < 8) {   // the parked parts are ordered before by the caller's barrier; the fetch-add releases them
        const int f = tid >> 2, quarter = tid & 3;
        bool mine = false;
        if (fin[f].c_hi > fin[f].c_lo && !(f == 1 && fin[0].tile == fin[1].tile)) {
            int* counter = &counters[fin[f].tile * 4 + quarter];
            mine = atomic_add_acq_rel(counter, 1) == fin[f].c_hi - fin[f].c_lo;
            if (mine) *counter = 0;
        }
        fin[f].last_of[quarter] = mine ? 1 : 0;
    }
    __syncthreads();
    for (int f = 0; f < 2; ++f) {
        if (!(fin[f].last_of[0] | fin[f].last_of[1] | fin[f].last_of[2] | fin[f].last_of[3])) continue;
        const int tile = fin[f].tile, c_lo = fin[f].c_lo, c_hi = fin[f].c_hi;
        const int tok0 = (tile / tiles_x) * n_cols, elems = min(n_cols, m - tok0) * 32, ch0 = (tile % tiles_x) * kTileN;
        const float4* first_part = reinterpret_cast<const float4*>(partial + ((size_t)c_lo * 2 + fin[f].first_slot) * park_floats);
        const float4* other = reinterpret_cast<const float4*>(partial);
        const size_t stride = park_floats / 2;   // two parts a CTA, four floats a vector
        for (int idx0 = tid; idx0 < elems; idx0 += THREADS * 2) {   // two elements (four channels of a token) a thread in flight
            const int idx[2] = {idx0, min(idx0 + THREADS, elems - 1)};
            float4 f0 = __ldcg(first_part + idx[0]), f1 = __ldcg(first_part + idx[1]);
#pragma unroll 4
            for (int c = c_lo + 1; c <= c_hi; ++c) {   // CTA order
                const float4 a = __ldcg(other + c * stride + idx[0]), b = __ldcg(other + c * stride + idx[1]);
                f0.x += a.x; f0.y += a.y; f0.z += a.z; f0.w += a.w;
                f1.x += b.x; f1.y += b.y; f1.z += b.z; f1.w += b.w;
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int col = idx[j] >> 5, c4 = (idx[j] & 31) * 4;
                if (idx0 + j * THREADS >= elems || !fin[f].last_of[c4 >> 5]) continue;
                const float s = scale ? __ldcg(scale + tok0 + col) : 1.0f;
                const float4 v = j ? f1 : f0;
                out.store4(tok0 + col, ch0 + c4, make_float4(v.x * s, v.y * s, v.z * s, v.w * s));
            }
        }
    }
}

}  // namespace streamk
}  // namespace goq
