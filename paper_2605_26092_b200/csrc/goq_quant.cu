// The steps either side of the inner product, on the device:
//   quantize_geo_kernel      Sections 3.2-3.4 (GEO mode): primary PoT code by round-to-nearest, orthogonal residual (Eq. 1),
//                            analytical sign inference and pattern selection per micro-block (Section 3.3, steps 1-3),
//                            decoupled least-squares coefficients (Eq. 2). One warp per macro-block.
//   solve_ref_kernel         Section 3.4, REF mode (Eq. 3): 2 x 2 ridge regression per macro-block on calibration inputs.
//   quantize_act_kernel      Section 3.5: X~ and s_x of Eq. 4 (per-token symmetric 8-bit integers).
// All decisions that end in an integer (a code, a pattern, a sign, a quantised activation) are taken in float64, the
// precision of the reference they are checked against; the work is bound by reading the inputs once.
#include <cuda_fp16.h>
#include "goq_common.cuh"
#include "goq_internal.h"
#include "goq_ref_rows.cuh"
#include <type_traits>

namespace goq {
namespace quant {

constexpr int kWarps = 8;
constexpr unsigned kFull = 0xFFFFFFFFu;

// ---- GEO quantizer -----------------------------------------------------------------------------------------
// A lane owns a whole micro-block (8 weights), so all four pair patterns stay inside the thread; the LPG = group / 8 lanes
// of a macro-block share its sums. Everything is flat: macro-blocks do not straddle rows, so lane l of a warp takes
// micro-block base + l whatever the shape. Bound: instruction issue, with the float64 pipe (about 85 operations per
// micro-block) and the memory system near behind. What keeps float64 work down without changing one result:
//   - codes need no division (rtn_codes), the two quotients share one reciprocal (quotient), ||b1||^2 is summed in integers (norm_units);
//   - every product has a power of two as a factor, hence is exact; ||b2||^2 = ||b1||^2 (b2 is a signed permutation
//     of b1), <w, b2> is the sum of the chosen patterns' |d|;
// Sums are added in a fixed order: elements 0..3 and 4..7 of a micro-block apart, each over the lanes from the farthest
// partner down, then the halves.
// Measured, 11008 x 4096 W3 g128: 84 us (two float64 divisions, ||b1||^2 in float64 and the sums of |d| as two halves: 92; one lane per four weights, with a
// float64 quotient per weight and a warp-wide float64 reduction for every sum: 438). 62 registers and 32 warps an SM, issue slots ~70 % busy: the number
// of instructions counts. Not kept: the next micro-block's loads in flight (24 warps 89 us, 32 warps with spills 98), 32-byte loads (88).
template <int LPG>
__device__ __forceinline__ double group_sum2(double p0, double p1) {
    if constexpr (LPG == 1) {
        return p0 + p1;
    } else {
        constexpr int o0 = LPG / 2;
        const bool up = (threadIdx.x & o0) != 0;   // the first step splits the halves over the lanes: one exchange instead of two
        double v = (up ? p1 : p0) + __shfl_xor_sync(kFull, up ? p0 : p1, o0);
#pragma unroll
        for (int o = o0 / 2; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        return v + __shfl_xor_sync(kFull, v, o0);
    }
}

// a / b rounded to nearest, as a division would, given r = 1/b to about 2^-42. b = ||b1||^2 is an integer of at most 21 bits times a power of two. Then
//   q = a r is off by at most 2^11 ulp, so a - q b fits 53 bits and the fma gives it exactly, and the corrected quotient is off by 2^-31 ulp before its one
//   rounding; a / b itself is never a midpoint of two doubles (54-bit odd times b has more bits than a) and at least 2^-22 ulp away from one.
// No underflow: a is a multiple of 2^-156. An infinite a stays what it is.
__device__ __forceinline__ double quotient(double a, double b, double r) {
    const double q = a * r;
    return fabs(q) <= 1.7976931348623157e308 ? fma(fma(-q, b, a), r, q) : q;
}
// sum over a micro-block of (b1 2^emax)^2: the magnitudes as bytes
template <int WB>
__device__ __forceinline__ uint32_t norm_units(uint32_t code) {
    // W3 codes 0..7: 8 4 2 0 8 4 2 1;  W2 codes 0..3: 2 0 2 1;  W4 by e: 128 64 32 16 8 4 2 and 0 (the zero; -2^-7, code 15, is counted apart)
    constexpr uint32_t t0 = WB == 3 ? 0x00020408u : WB == 2 ? 0x01020002u : 0x10204080u, t1 = WB == 3 ? 0x01020408u : WB == 2 ? 0u : 0x00020408u;
    const uint32_t sel = WB == 4 ? code & 0x77777777u : code;
    const uint32_t a = __byte_perm(t0, t1, sel), b = __byte_perm(t0, t1, sel >> 16);
    uint32_t n = __dp4a(a, a, __dp4a(b, b, 0u));
    if constexpr (WB == 4) {
        const uint32_t two = code & (code >> 1);
        n += __popc(two & (two >> 2) & 0x11111111u);
    }
    return n;
}

// Codes of a micro-block, a nibble each: nearest lattice state in linear distance, exact ties to the state of smaller
// magnitude (Section 3.2). Between 2^-(e+1) and 2^-e the midpoint is 0.75 * 2^-e; the zero meets the smallest negative
// magnitude at 2^-(emax+1) and the smallest positive one (there is no +2^-emax) at 2^-emax. `th` holds these midpoints times
// s_norm, rounded DOWN to fp32: for an fp32 number a, a > t and a > round_down(t) are the same, so every decision is the
// exact one and nothing is divided. A code is a sum of predicates: e counts the midpoints |w| does not exceed, and the sign bit
// is set only below the negative zero bin (between it and 0, |w| exceeds no midpoint of either sign and e = emax, the zero).
template <int WB> struct Midpoints {
    static constexpr int emax = (1 << (WB - 1)) - 1;
    float both[emax > 1 ? emax - 1 : 1], last_neg, last_pos, zero_neg;
};
template <int WB>
__device__ __forceinline__ Midpoints<WB> midpoints(float s) {
    constexpr int emax = Midpoints<WB>::emax;
    Midpoints<WB> m;
    float t = 0.75f;
#pragma unroll
    for (int i = 0; i < emax - 1; ++i, t *= 0.5f) m.both[i] = __fmul_rd(t, s);
    m.last_neg = __fmul_rd(t, s);
    m.last_pos = __fmul_rd(1.0f / (float)(1 << emax), s);
    m.zero_neg = __fmul_rd(1.0f / (float)(2 << emax), s);
    return m;
}
template <int WB>
__device__ __forceinline__ uint32_t rtn_codes(const float (&w)[8], const Midpoints<WB>& m) {
    constexpr int emax = Midpoints<WB>::emax;
    uint32_t code = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float a = fabsf(w[i]);
        const bool neg = w[i] < -m.zero_neg;
#pragma unroll
        for (int q = 0; q < emax - 1; ++q)
            if (!(a > m.both[q])) code += 1u << (4 * i);
        if (!(a > (neg ? m.last_neg : m.last_pos))) code += 1u << (4 * i);
        if (neg) code += (1u << (WB - 1)) << (4 * i);
    }
    return code;
}
// The values of eight codes as the high words of doubles (the low words are zero). W <= 3: sign/exponent bytes by table.
template <int WB>
__device__ __forceinline__ void code_values(uint32_t code, double (&x)[8]) {
    if constexpr (WB <= 3) {
        // W3 codes 0..7: +1 +.5 +.25 0 -1 -.5 -.25 -.125;  W2 codes 0..3: +1 0 -1 -.5
        constexpr uint32_t t0 = WB == 3 ? 0x00D0E0F0u : 0xE0F000F0u, t1 = WB == 3 ? 0xC0D0E0F0u : 0u;
        constexpr uint32_t s0 = WB == 3 ? 0x003F3F3Fu : 0xBFBF003Fu, s1 = WB == 3 ? 0xBFBFBFBFu : 0u;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t sel = h ? code >> 16 : code;
            const uint32_t t = __byte_perm(t0, t1, sel), sg = __byte_perm(s0, s1, sel);
            const uint32_t v01 = __byte_perm(t, sg, 0x5140), v23 = __byte_perm(t, sg, 0x7362);
            x[4 * h + 0] = __hiloint2double((int)(v01 << 16), 0);
            x[4 * h + 1] = __hiloint2double((int)(v01 & 0xFFFF0000u), 0);
            x[4 * h + 2] = __hiloint2double((int)(v23 << 16), 0);
            x[4 * h + 3] = __hiloint2double((int)(v23 & 0xFFFF0000u), 0);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t c = (code >> (4 * i)) & 15u;
            x[i] = __hiloint2double(c == 7u ? 0 : (int)(((1023u - (c & 7u)) << 20) | ((c & 8u) << 28)), 0);
        }
    }
}

template <int WB, int LPG, bool K1>
__global__ void __launch_bounds__(kWarps * 32, 4)
quantize_geo_kernel(const float* __restrict__ w, uint8_t* __restrict__ codes, uint8_t* __restrict__ meta,
                    uint16_t* __restrict__ coef, long long n_micro) {
    const int in_group = threadIdx.x & (LPG - 1);
    const long long mb = (long long)blockIdx.x * (kWarps * 32) + threadIdx.x;   // this lane's micro-block
    const bool on = mb < n_micro;
    float wf[8];
    {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (on) {
            const float4* src = reinterpret_cast<const float4*>(w) + mb * 2;
            a = __ldcs(src); b = __ldcs(src + 1);
        }
        wf[0] = a.x; wf[1] = a.y; wf[2] = a.z; wf[3] = a.w;
        wf[4] = b.x; wf[5] = b.y; wf[6] = b.z; wf[7] = b.w;
    }
    // Section 3.2: s_norm = ||w||_inf, b1 = Q(w / s_norm)
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) s = fmaxf(s, fabsf(wf[i]));
#pragma unroll
    for (int o = LPG / 2; o; o >>= 1) s = fmaxf(s, __shfl_xor_sync(kFull, s, o));
    const uint32_t code = rtn_codes<WB>(wf, midpoints<WB>(s));
    double x[8], p[2] = {0.0, 0.0};
    code_values<WB>(code, x);
#pragma unroll
    for (int i = 0; i < 8; ++i) p[i >> 2] = fma((double)wf[i], x[i], p[i >> 2]);   // exact product
    uint32_t nu = norm_units<WB>(code);
#pragma unroll
    for (int o = LPG / 2; o; o >>= 1) nu += __shfl_xor_sync(kFull, nu, o);
    const float nb = (float)nu * (1.0f / (float)(1 << (2 * Midpoints<WB>::emax)));   // ||b1||^2: at most 128 and 21 bits, exact
    double rb = (double)__fdividef(1.0f, nb);
    rb = fma(fma(-rb, (double)nb, 1.0), rb, rb);   // one Newton step: 2^-21 -> 2^-42
    // zero-norm bypass: an all-zero block keeps c1 = c2 = 0
    const double c1 = nb == 0.f ? 0.0 : quotient(group_sum2<LPG>(p[0], p[1]), (double)nb, rb);
    double c2 = 0.0;
    uint32_t rec = 0;
    if constexpr (!K1) {
        // Eq. 1: r = w - c1 b1. Section 3.3, steps 1-2: d = x_i r_j - x_j r_i per pair, eta* = sgn d, A_s = sum |d|, s* = first maximiser
        double r[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) r[i] = fma(-c1, x[i], (double)wf[i]);
        double best = -1.0;
#pragma unroll
        for (int sp = 1; sp <= 4; ++sp) {
            double d[4];
            int n = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int j = i ^ sp;   // pairs in ascending order of their lower index
                // exact products; the added zero keeps d from being -0, so that its sign bit is "d < 0"
                if (i < j) { d[n] = fma(x[i], r[j], fma(-x[j], r[i], 0.0)); ++n; }
            }
            const double a = sp < 4 ? (fabs(d[0]) + fabs(d[1])) + (fabs(d[2]) + fabs(d[3]))
                                    : ((fabs(d[0]) + fabs(d[1])) + fabs(d[2])) + fabs(d[3]);
            uint32_t f = 0;   // flag of pair p at bit 2 + p
#pragma unroll
            for (int q = 3; q >= 0; --q) f = __funnelshift_l((uint32_t)__double2hiint(d[q]), f, 1);
            f = f * 4u + (uint32_t)(sp - 1);
            if (a > best) { best = a; rec = f; }
        }
        // step 3 and Eq. 2: with eta = sgn d, <w, b2> of the micro-block is the chosen pattern's sum |d| (<b1, b2> = 0)
        double wb2 = best;
#pragma unroll
        for (int o = LPG / 2; o; o >>= 1) wb2 += __shfl_xor_sync(kFull, wb2, o);
        c2 = nb == 0.f ? 0.0 : quotient(wb2, (double)nb, rb);
        if (nb == 0.f) rec = 0;   // s_norm = 0 iff b1 = 0: the largest weight never rounds to zero
    }
    if (!on) return;
    const uint32_t even = code & 0x0F0F0F0Fu, odd = (code >> 4) & 0x0F0F0F0Fu;   // nibbles -> bytes
    const uint32_t lo = __byte_perm(even, odd, 0x5140), hi = __byte_perm(even, odd, 0x7362);
    uint32_t* dst = reinterpret_cast<uint32_t*>(codes) + mb * 2;
    if ((reinterpret_cast<uintptr_t>(codes) & 7u) == 0) *reinterpret_cast<uint2*>(dst) = make_uint2(lo, hi);
    else { dst[0] = lo; dst[1] = hi; }
    meta[mb] = (uint8_t)rec;
    if (in_group == 0) {
        uint16_t* c = coef + mb / LPG * 2;
        c[0] = __half_as_ushort(__double2half(c1));
        c[1] = __half_as_ushort(__double2half(c2));
    }
}

// ---- REF mode (Eq. 3) --------------------------------------------------------------------------------------
// c* = (A^T A + lambda I)^-1 A^T Y with A = [X_q b1, X_q b2] (M x 2), Y = X_q w, per row and macro-block column j, in float64.
// The calibration rows enter only through the Gram matrix G = X_q^T X_q of the column (g x g), which all output rows share:
//   b1^T G b1, b1^T G b2, b2^T G b2, b1^T G w, b2^T G w  are the five entries of the normal equations. With H = the lower
// triangle of G and half its diagonal, G = H + H^T and b^T G c = b.(H c) + (H b).c, so a row costs the three triangular products
// H b1, H b2, H w: 1.5 g^2 multiply-adds whatever M is, against 3 M g for the observations one by one. With M <= g / 2 the
// latter is the cheaper (DIRECT), and is used.
// Both are matrix products with the columns' G (or X) as the shared operand and run on the float64 tensor pipe
// (mma.m8n8k4): same rate as scalar float64 on this part, but an eighth of the operand traffic and no conversions of shared
// values in the inner loop. CTA = 16 warps on one macro-block column and a range of 8-row tiles; G is formed once per CTA.
// Bound: the float64 pipe.
constexpr int kRefChunk = 64;   // observations staged at a time while G is formed
template <int WB, int NB, bool DIRECT>
__global__ void __launch_bounds__(kRefWarps * 32, 1)
solve_ref_kernel(const float* __restrict__ w, const uint8_t* __restrict__ codes, const uint8_t* __restrict__ meta,
                 const float* __restrict__ xc, int m, double lambda, uint16_t* __restrict__ coef, double* __restrict__ c_out,
                 int n_out, int k_in) {
    constexpr int G = NB * 8, kStride = RefSmem<NB>::kStride;
    extern __shared__ __align__(16) unsigned char smem_ref[];
    double* frag = reinterpret_cast<double*>(smem_ref);
    float* stage = reinterpret_cast<float*>(frag + RefSmem<NB>::kFrags * 32);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, lr = lane >> 2, lc = lane & 3;
    const int j = blockIdx.x;
    const float* xj = xc + (size_t)j * G;

    if constexpr (DIRECT) {   // operand = the observations: fragment (block of 8 observations, 4 channels), element (channel, observation)
#pragma unroll 4
        for (int i = threadIdx.x; i < ((m + 7) / 8) * 8 * G; i += kRefWarps * 32) {
            const int o = i / G, k = i - o * G;
            frag[((o >> 3) * (2 * NB) + (k >> 2)) * 32 + (o & 7) * 4 + (k & 3)] = o < m ? (double)xj[(size_t)o * k_in + k] : 0.0;
        }
        __syncthreads();
    } else {
        // G, lower block triangle, element blocks of 8 x 8. Up to 8 block rows: warp w takes block row w. With 16: warp w < 8 takes
        // blocks 0..7 of row 15 - w, warp 8 + v the rest of row 15 - v and row v (8 or 9 blocks each).
        constexpr int kAcc = NB < 8 ? NB : 8;
        const int v = warp & 7;
        const bool second = NB == 16 && warp >= 8;
        const int row_a = NB == 16 ? 15 - v : warp, b0 = second ? 8 : 0;   // blocks b0 .. of row_a, and blocks 0..v of row v
        double acc_a[kAcc][2], acc_b[kAcc][2];
#pragma unroll
        for (int b = 0; b < kAcc; ++b) acc_a[b][0] = acc_a[b][1] = acc_b[b][0] = acc_b[b][1] = 0.0;
        for (int o0 = 0; o0 < m; o0 += kRefChunk) {
            __syncthreads();
#pragma unroll
            for (int q = 0; q < (kRefChunk * G) / (kRefWarps * 32); ++q) {   // all of a thread's loads in flight
                const int i = (int)threadIdx.x + q * (kRefWarps * 32), o = i / G, k = i - o * G;
                stage[o * kStride + k] = (o0 + o < m) ? xj[(size_t)(o0 + o) * k_in + k] : 0.f;
            }
            __syncthreads();
            if (warp < NB) {
#pragma unroll 1
                for (int s = 0; s < kRefChunk / 4; ++s) {
                    const float* xs = stage + (s * 4 + lc) * kStride + lr;
                    const double fa = (double)xs[row_a * 8];
#pragma unroll
                    for (int b = 0; b < kAcc; ++b)
                        if (b0 + b <= row_a) dmma(acc_a[b], fa, (double)xs[(b0 + b) * 8]);
                    if (second) {
                        const double fb = (double)xs[v * 8];
#pragma unroll
                        for (int b = 0; b < kAcc; ++b)
                            if (b <= v) dmma(acc_b[b], fb, (double)xs[b * 8]);
                    }
                }
            }
        }
        if (warp < NB) {
            // element (row lr, columns 2 lc, 2 lc + 1) of block (ib, b) -> H as an operand fragment: element (k, i)
            auto put = [&](int ib, int b, const double (&c)[2]) {
                const int k = 2 * lc;
                double2 h = make_double2(c[0], c[1]);
                if (ib == b) {
                    h.x = k > lr ? 0.0 : (k == lr ? 0.5 * h.x : h.x);
                    h.y = k + 1 > lr ? 0.0 : (k + 1 == lr ? 0.5 * h.y : h.y);
                }
                *reinterpret_cast<double2*>(frag + (ib * (ib + 1) + 2 * b + (k >> 2)) * 32 + lr * 4 + (k & 3)) = h;
            };
#pragma unroll
            for (int b = 0; b < kAcc; ++b) if (b0 + b <= row_a) put(row_a, b0 + b, acc_a[b]);
            if (second) {
#pragma unroll
                for (int b = 0; b < kAcc; ++b) if (b <= v) put(v, b, acc_b[b]);
            }
        }
        __syncthreads();
    }

    const int n_rt = (n_out + 7) / 8;
    solve_rows<WB, NB, DIRECT>(frag, stage, w, codes, meta, m, lambda, coef, c_out, n_out, k_in, j, (int)((long long)n_rt * blockIdx.y / gridDim.y),
                               (int)((long long)n_rt * (blockIdx.y + 1) / gridDim.y));
}

// ---- activation quantizer (Section 3.5: X~, s_x) -----------------------------------------------------------
// Per token: s_x = max |x| / q_max (1 for an all-zero token), x~ = clamp(rne(x / s_x), +-q_max), q_max = 2^(bits-1) - 1, in int8
// containers whatever the width; float64 decides. Bound: memory, 5 bytes an fp32 element. So a row is read once and kept in
// registers between the maximum and the rounding (a warp or a CTA per token by the row's length), and the float64 division is
// made only where it can matter: x * (q_max / max|x|) in fp32 is within 127 * 3 * 2^-24 < 1e-4 of x / s_x, so any quotient further
// than that from a half rounds the same way; the others, and everything that is not finite, take the division.
// Measured, 12608 x 768 fp32: 17.9 us (a division per element, two passes: 39.5); 12608 x 3072 with the maxima given: 43.4 us (88.6).
__device__ __forceinline__ float load_act(const float* p) { return *p; }
__device__ __forceinline__ float load_act(const uint16_t* p) { return bf16_to_f32(*p); }

struct Scale {
    double s, qmax;
    float inv;    // 0: always divide
    __device__ __forceinline__ Scale(double amax, double q) : s(amax == 0.0 ? 1.0 : amax / q), qmax(q) {
        const float r = (float)q / (float)amax;   // (the maximum is an fp32 number: one rounding, as a float64 quotient's would be)
        inv = (r > 1e-36f && r < 1e36f) ? r : 0.f;
    }
    __device__ __forceinline__ int exact(double x) const {
        const double q = rint(x / s);   // round half to even
        return (int)fmin(qmax, fmax(-qmax, q));
    }
    __device__ __forceinline__ int operator()(float x) const {
        const float v = x * inv, r = rintf(v);
        if (inv != 0.f && fabsf(v - r) < 0.4999f) return (int)fminf((float)qmax, fmaxf(-(float)qmax, r));   // (a given maximum may be too small)
        return exact((double)x);
    }
};

// Four elements of a row as fp32
__device__ __forceinline__ float4 load4(const float* p) { return __ldcs(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 load4(const uint16_t* p) {
    const uint2 v = __ldcs(reinterpret_cast<const uint2*>(p));
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xFFFF0000u));
}
// NaN elements do not take part in the maximum (fmax); they round to -q_max like every comparison that fails
__device__ __forceinline__ float max4(float4 v) { return fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))); }
__device__ __forceinline__ uint32_t quant4(const Scale& sc, float4 v) {
    return (uint32_t)(sc(v.x) & 255) | ((uint32_t)(sc(v.y) & 255) << 8) | ((uint32_t)(sc(v.z) & 255) << 16) | ((uint32_t)(sc(v.w) & 255) << 24);
}

// Vector rows (k a multiple of 4, aligned). WARPS: warps that share a token (1 or 8); HOLD: vectors a lane keeps.
template <typename T, int WARPS, int HOLD>
__global__ void __launch_bounds__(256)
quantize_act_vec_kernel(const T* __restrict__ x, int m, int k4, const float* __restrict__ amax_in, int8_t* __restrict__ xq,
                        float* __restrict__ sx, double qmax) {
    constexpr int kThreads = WARPS * 32;
    const int tok = WARPS == 1 ? (int)(blockIdx.x * 8 + (threadIdx.x >> 5)) : (int)blockIdx.x, tid = threadIdx.x & (kThreads - 1);
    if (WARPS == 1 && tok >= m) return;
    const T* row = x + (size_t)tok * k4 * 4;
    uint32_t* out = reinterpret_cast<uint32_t*>(xq) + (size_t)tok * k4;
    float4 held[HOLD];
#pragma unroll
    for (int h = 0; h < HOLD; ++h) {
        const int i = tid + h * kThreads;
        held[h] = i < k4 ? load4(row + (size_t)i * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float a;
    if (amax_in) {
        a = amax_in[tok];
    } else {
        a = 0.f;
#pragma unroll
        for (int h = 0; h < HOLD; ++h) a = fmaxf(a, max4(held[h]));
        for (int i = tid + HOLD * kThreads; i < k4; i += kThreads) a = fmaxf(a, max4(load4(row + (size_t)i * 4)));
#pragma unroll
        for (int o = 16; o; o >>= 1) a = fmaxf(a, __shfl_xor_sync(kFull, a, o));
        if constexpr (WARPS > 1) {
            __shared__ float red[WARPS];
            if ((tid & 31) == 0) red[tid >> 5] = a;
            __syncthreads();
#pragma unroll
            for (int w = 0; w < WARPS; ++w) a = fmaxf(a, red[w]);
        }
    }
    const Scale sc((double)a, qmax);
#pragma unroll
    for (int h = 0; h < HOLD; ++h)
        if (tid + h * kThreads < k4) out[tid + h * kThreads] = quant4(sc, held[h]);
    for (int i = tid + HOLD * kThreads; i < k4; i += kThreads) out[i] = quant4(sc, load4(row + (size_t)i * 4));
    if (tid == 0) sx[tok] = (float)sc.s;
}

// Any row: one CTA per token, element by element
template <typename T>
__global__ void __launch_bounds__(256)
quantize_act_kernel(const T* __restrict__ x, int k, const float* __restrict__ amax_in, int8_t* __restrict__ xq, float* __restrict__ sx,
                    double qmax) {
    __shared__ float red[8];
    const int tok = blockIdx.x, tid = threadIdx.x;
    const T* row = x + (size_t)tok * k;
    float a = 0.f;
    if (amax_in) {
        a = amax_in[tok];
    } else {
        for (int i = tid; i < k; i += 256) a = fmaxf(a, fabsf(load_act(row + i)));
#pragma unroll
        for (int o = 16; o; o >>= 1) a = fmaxf(a, __shfl_xor_sync(kFull, a, o));
        if ((tid & 31) == 0) red[tid >> 5] = a;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 8; ++i) a = fmaxf(a, red[i]);
    }
    const Scale sc((double)a, qmax);
    for (int i = tid; i < k; i += 256) xq[(size_t)tok * k + i] = (int8_t)sc(load_act(row + i));
    if (tid == 0) sx[tok] = (float)sc.s;
}

}  // namespace quant

// ---- launchers -----------------------------------------------------------------------------------------------
template <int WB, int LPG>
static void launch_geo(const Geometry& g, const float* w, uint8_t* codes, uint8_t* meta, uint16_t* coef, cudaStream_t st) {
    const long long n_micro = (long long)g.n_out * (g.k_in / 8);
    constexpr int kPerBlock = quant::kWarps * 32;
    const unsigned blocks = (unsigned)((n_micro + kPerBlock - 1) / kPerBlock);
    if (g.k1) quant::quantize_geo_kernel<WB, LPG, true><<<blocks, quant::kWarps * 32, 0, st>>>(w, codes, meta, coef, n_micro);
    else quant::quantize_geo_kernel<WB, LPG, false><<<blocks, quant::kWarps * 32, 0, st>>>(w, codes, meta, coef, n_micro);
}
template <int WB>
static void launch_geo_group(const Geometry& g, const float* w, uint8_t* codes, uint8_t* meta, uint16_t* coef, cudaStream_t st) {
    switch (g.group) {
        case 8: launch_geo<WB, 1>(g, w, codes, meta, coef, st); break;
        case 16: launch_geo<WB, 2>(g, w, codes, meta, coef, st); break;
        case 32: launch_geo<WB, 4>(g, w, codes, meta, coef, st); break;
        case 64: launch_geo<WB, 8>(g, w, codes, meta, coef, st); break;
        default: launch_geo<WB, 16>(g, w, codes, meta, coef, st); break;
    }
}
cudaError_t launch_quantize_geo(const Geometry& g, const float* w, uint8_t* codes, uint8_t* meta, uint16_t* coef, cudaStream_t st) {
    if (g.wbits == 2) launch_geo_group<2>(g, w, codes, meta, coef, st);
    else if (g.wbits == 3) launch_geo_group<3>(g, w, codes, meta, coef, st);
    else launch_geo_group<4>(g, w, codes, meta, coef, st);
    return cudaGetLastError();
}
template <int WB, int NB>
static cudaError_t launch_ref(const Geometry& g, const float* w, const uint8_t* codes, const uint8_t* meta, const float* x_calib,
                              int m, double lambda, uint16_t* coef, double* c_out, cudaStream_t st) {
    const bool direct = 2 * m <= NB * 8;
    auto kernel = direct ? quant::solve_ref_kernel<WB, NB, true> : quant::solve_ref_kernel<WB, NB, false>;
    const size_t smem = quant::RefSmem<NB>::kBytes;
    static SmemAttrCache cache[2];
    if (cudaError_t e = ensure_dynamic_smem(kernel, smem, cache[direct ? 1 : 0])) return e;
    const int sms = sm_count();
    // Row chunks per column: every CTA forms its column's G again, so few chunks save work and many fill the chip. Take the
    // split whose waves cost least in float64 tensor clocks (4 per m8n8k4 and SM, a row tile's loads and epilogue about 400). Row
    // tiles go in rounds of 16 warps; a CTA with fewer is bound by one warp's chain of products instead, about four tiles' clocks.
    const int cols = g.k_in / g.group, tiles = (g.n_out + 7) / 8, slots = sms;
    const double form = direct ? 500.0 : 4.0 * (NB * (NB + 1) / 2) * ((m + 63) / 64 * 16) + 1500.0;
    const double tile = 12.0 * (direct ? (m + 7) / 8 * 2 * NB : NB * (NB + 1)) + 400.0;
    int best = 1;
    double best_cost = 0.0;
    for (int c = 1; c <= tiles && c <= 65535 && c <= 4 * slots; ++c) {
        const double waves = (double)(((long long)cols * c + slots - 1) / slots);
        const int per = (tiles + c - 1) / c;
        const int paid = per >= quant::kRefWarps ? (per + quant::kRefWarps - 1) / quant::kRefWarps * quant::kRefWarps : (per > 4 ? per : 4);
        const double cost = waves * (form + paid * tile);
        if (c == 1 || cost < best_cost) { best = c; best_cost = cost; }
    }
    kernel<<<dim3(cols, best), quant::kRefWarps * 32, smem, st>>>(w, codes, meta, x_calib, m, lambda, coef, c_out, g.n_out, g.k_in);
    return cudaGetLastError();
}
template <int WB>
static cudaError_t launch_ref_group(const Geometry& g, const float* w, const uint8_t* codes, const uint8_t* meta, const float* x_calib,
                                    int m, double lambda, uint16_t* coef, double* c_out, cudaStream_t st) {
    switch (g.group) {
        case 8: return launch_ref<WB, 1>(g, w, codes, meta, x_calib, m, lambda, coef, c_out, st);
        case 16: return launch_ref<WB, 2>(g, w, codes, meta, x_calib, m, lambda, coef, c_out, st);
        case 32: return launch_ref<WB, 4>(g, w, codes, meta, x_calib, m, lambda, coef, c_out, st);
        case 64: return launch_ref<WB, 8>(g, w, codes, meta, x_calib, m, lambda, coef, c_out, st);
        default: return launch_ref<WB, 16>(g, w, codes, meta, x_calib, m, lambda, coef, c_out, st);
    }
}
cudaError_t launch_solve_ref(const Geometry& g, const float* w, const uint8_t* codes, const uint8_t* meta, const float* x_calib,
                             int m, double lambda, uint16_t* coef, double* c_out, cudaStream_t st) {
    if (g.wbits == 2) return launch_ref_group<2>(g, w, codes, meta, x_calib, m, lambda, coef, c_out, st);
    if (g.wbits == 3) return launch_ref_group<3>(g, w, codes, meta, x_calib, m, lambda, coef, c_out, st);
    return launch_ref_group<4>(g, w, codes, meta, x_calib, m, lambda, coef, c_out, st);
}
cudaError_t launch_quantize_act(const void* x, int x_dtype, int m, int k, int abits, const float* amax, int8_t* xq, float* sx,
                                cudaStream_t st) {
    const double qmax = (double)((1 << (abits - 1)) - 1);
    const size_t elem = x_dtype == GOQ_F32 ? 4 : 2;
    const bool vec = k % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & (4 * elem - 1)) == 0 && (reinterpret_cast<uintptr_t>(xq) & 3u) == 0;
    auto go = [&](auto* p) {
        using T = std::remove_const_t<std::remove_pointer_t<decltype(p)>>;
        if (!vec) quant::quantize_act_kernel<T><<<m, 256, 0, st>>>(p, k, amax, xq, sx, qmax);
        else if (k <= 1024)   // a warp per token: 8 vectors a lane cover the row
            quant::quantize_act_vec_kernel<T, 1, 8><<<(m + 7) / 8, 256, 0, st>>>(p, m, k / 4, amax, xq, sx, qmax);
        else                  // a CTA per token: 4096 elements in registers
            quant::quantize_act_vec_kernel<T, 8, 4><<<m, 256, 0, st>>>(p, m, k / 4, amax, xq, sx, qmax);
    };
    if (x_dtype == GOQ_F32) go((const float*)x);
    else go((const uint16_t*)x);
    return cudaGetLastError();
}

}  // namespace goq
