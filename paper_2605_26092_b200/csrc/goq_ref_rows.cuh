// What the two kernels of the REF solve share: eight rows of W at a time against a column's Gram matrix (or observations) in shared memory, on the float64
// tensor pipe.
#pragma once
#include <cuda_fp16.h>
#include "goq_common.cuh"

namespace goq {
namespace quant {

// value of code c on the b-bit asymmetric lattice (Section 3.2): (-1)^sign 2^-e, the smallest positive bin being zero
__device__ __forceinline__ double lattice_value(int c, int wbits) {
    const int emax = (1 << (wbits - 1)) - 1, sg = c >> (wbits - 1), e = c & emax;
    if (!sg && e == emax) return 0.0;
    const double mag = __longlong_as_double((long long)(1023 - e) << 52);   // 2^-e
    return sg ? -mag : mag;
}
constexpr int kRefWarps = 16;
__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}
template <int NB> struct RefSmem {   // NB = group / 8
    static constexpr int kStride = NB * 8 + 4;                         // floats per staged row: fragment reads are conflict-free
    static constexpr int kFrags = NB * (NB + 1);                       // 4 x 8 operand fragments of H (of X: at most NB * NB)
    static constexpr size_t kBytes = (size_t)kFrags * 32 * sizeof(double) + (size_t)kRefWarps * 16 * kStride * sizeof(float);
};
// Row tiles [rt_lo, rt_hi) of column j: c* of eight rows each, a tile a warp (warps 0..15 of the CTA). frag: H as operand fragments (DIRECT: the observations);
// stage: 16 rows of kStride floats a warp.
template <int WB, int NB, bool DIRECT>
__device__ __forceinline__ void solve_rows(const double* frag, float* stage, const float* __restrict__ w, const uint8_t* __restrict__ codes,
                                           const uint8_t* __restrict__ meta, int m, double lambda, uint16_t* __restrict__ coef, double* __restrict__ c_out,
                                           int n_out, int k_in, int j, int rt_lo, int rt_hi) {
    constexpr unsigned kFull = 0xFFFFFFFFu;
    constexpr int G = NB * 8, kStride = RefSmem<NB>::kStride;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lr = lane >> 2, lc = lane & 3, nj = k_in / G;
    // this warp's eight rows: b1 and b2 as a bf16 pair (PoT values are exact in it), and w
    uint32_t* vb = reinterpret_cast<uint32_t*>(stage + warp * 16 * kStride);
    float* vw = stage + warp * 16 * kStride + 8 * kStride;
    auto low = [](uint32_t p) { return (double)__uint_as_float(p << 16); };
    auto high = [](uint32_t p) { return (double)__uint_as_float(p & 0xFFFF0000u); };
    const bool codes8 = (reinterpret_cast<uintptr_t>(codes) & 7u) == 0;
    for (int rt = rt_lo + warp; rt < rt_hi; rt += kRefWarps) {
        __syncwarp();
        for (int i = lane; i < 8 * NB; i += 32) {
            const int r = i / NB, t = i - r * NB, row = rt * 8 + r;
            uint32_t* dst = vb + r * kStride + t * 8;
            if (row < n_out) {   // b2 by the recorded exchange (Section 3.3)
                const size_t o = (size_t)row * k_in + (size_t)j * G + t * 8;
                uint32_t cw[2];
                if (codes8) { const uint2 q = *reinterpret_cast<const uint2*>(codes + o); cw[0] = q.x; cw[1] = q.y; }
                else {
                    cw[0] = codes[o] | (codes[o + 1] << 8) | (codes[o + 2] << 16) | ((uint32_t)codes[o + 3] << 24);
                    cw[1] = codes[o + 4] | (codes[o + 5] << 8) | (codes[o + 6] << 16) | ((uint32_t)codes[o + 7] << 24);
                }
                const uint32_t rec = meta[o / 8], s = (rec & 3u) + 1u, flips = flip_mask(rec);
#pragma unroll
                for (int e = 0; e < 8; ++e) dst[e] = __float_as_uint((float)lattice_value((int)((cw[e >> 2] >> (8 * (e & 3))) & 255u), WB)) >> 16;
                uint32_t y[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) y[e] = dst[e ^ s] ^ (((flips >> e) & 1u) << 15);
#pragma unroll
                for (int e = 0; e < 8; ++e) dst[e] |= y[e] << 16;
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) dst[e] = 0u;
            }
        }
#pragma unroll
        for (int q0 = 0; q0 < 2 * NB; q0 += 8) {   // up to eight loads of a lane in flight (one after another they were most of a small solve)
            float v[8];
#pragma unroll
            for (int q = 0; q < 8 && q0 + q < 2 * NB; ++q) {
                const int i = lane + (q0 + q) * 32, r = i / G, k = i - r * G, row = rt * 8 + r;
                v[q] = row < n_out ? w[(size_t)row * k_in + (size_t)j * G + k] : 0.f;
            }
#pragma unroll
            for (int q = 0; q < 8 && q0 + q < 2 * NB; ++q) {
                const int i = lane + (q0 + q) * 32, r = i / G;
                vw[r * kStride + (i - r * G)] = v[q];
            }
        }
        __syncwarp();
        double g11 = 0, g12 = 0, g22 = 0, r1 = 0, r2 = 0;
        const uint32_t* fb = vb + lr * kStride + lc;
        const float* fw = vw + lr * kStride + lc;
        const int n_blocks = DIRECT ? (m + 7) / 8 : NB;
        // two blocks of 8 output columns at a time: they share the row operands
#pragma unroll 1
        for (int ib = 0; ib < n_blocks; ib += 2) {
            double c[2][3][2];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int q = 0; q < 3; ++q) c[h][q][0] = c[h][q][1] = 0.0;
            const bool two = NB > 1 && ib + 1 < n_blocks;
            const double* f0 = frag + (DIRECT ? ib * 2 * NB : ib * (ib + 1)) * 32 + lane;
            const double* f1 = frag + (DIRECT ? (ib + 1) * 2 * NB : (ib + 1) * (ib + 2)) * 32 + lane;
            const int s0 = DIRECT ? 2 * NB : 2 * (ib + 1), s1 = DIRECT ? 2 * NB : 2 * (ib + 2);
#pragma unroll 2
            for (int s = 0; s < s0; ++s) {
                const uint32_t p = fb[4 * s];
                const double a1 = low(p), a2 = high(p), a3 = (double)fw[4 * s];
                const double b0 = f0[s * 32];
                dmma(c[0][0], a1, b0); dmma(c[0][1], a2, b0); dmma(c[0][2], a3, b0);
                if (two) {
                    const double b1 = f1[s * 32];
                    dmma(c[1][0], a1, b1); dmma(c[1][1], a2, b1); dmma(c[1][2], a3, b1);
                }
            }
            if (two && !DIRECT) {
#pragma unroll
                for (int s = s1 - 2; s < s1; ++s) {
                    const double b1 = f1[s * 32];
                    const uint32_t p = fb[4 * s];
                    dmma(c[1][0], low(p), b1); dmma(c[1][1], high(p), b1); dmma(c[1][2], (double)fw[4 * s], b1);
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h == 1 && !two) break;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const double p = c[h][0][e], q = c[h][1][e], t = c[h][2][e];
                    if constexpr (DIRECT) {
                        g11 = fma(p, p, g11); g12 = fma(p, q, g12); g22 = fma(q, q, g22); r1 = fma(p, t, r1); r2 = fma(q, t, r2);
                    } else {
                        const int at = lr * kStride + (ib + h) * 8 + 2 * lc + e;
                        const double b1 = low(vb[at]), b2 = high(vb[at]), ww = (double)vw[at];
                        g11 = fma(b1, p, g11); g22 = fma(b2, q, g22);
                        g12 = fma(b1, q, fma(b2, p, g12));
                        r1 = fma(b1, t, fma(ww, p, r1));
                        r2 = fma(b2, t, fma(ww, q, r2));
                    }
                }
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            g11 += __shfl_xor_sync(kFull, g11, o); g12 += __shfl_xor_sync(kFull, g12, o); g22 += __shfl_xor_sync(kFull, g22, o);
            r1 += __shfl_xor_sync(kFull, r1, o); r2 += __shfl_xor_sync(kFull, r2, o);
        }
        if constexpr (!DIRECT) { g11 *= 2.0; g22 *= 2.0; }
        const int row = rt * 8 + lr;
        if (lc == 0 && row < n_out) {
            const double a = g11 + lambda, d = g22 + lambda, det = a * d - g12 * g12;
            const double c1 = (d * r1 - g12 * r2) / det, c2 = (a * r2 - g12 * r1) / det;
            const size_t o = ((size_t)row * nj + j) * 2;
            coef[o] = __half_as_ushort(__double2half(c1));
            coef[o + 1] = __half_as_ushort(__double2half(c2));
            if (c_out) { c_out[o] = c1; c_out[o + 1] = c2; }
        }
    }
}

}  // namespace quant
}  // namespace goq
