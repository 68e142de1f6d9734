// Device helpers of the integer-operand decode kernels (a chain of linears, one linear): the even split of a linear's unit records
// over the CTAs, the decode of a micro-block word into int8 operands, the coefficient stage, the conversion of activations to
// block fixed point and the hand-over of tile parts inside a CTA.
#pragma once
#include "goq_stream_core.cuh"

namespace goq {
namespace chain {

constexpr int kNW = 16;                      // consumer warps
constexpr int kStageRecs = kNW;              // records of a ring stage
constexpr int kTileSlots = 4;                // in-CTA reduction slots (tile parts in flight)
constexpr int kXPad = 32;                    // bytes between activation planes beyond k_pad: keeps the B-fragment loads conflict-free
constexpr int kMaxKBlocks = 96;              // activation scales kept per k-block: k_in <= 12288
constexpr int kGlobalSpin = 1 << 20;
constexpr int kMaxStages = 8;

// Split of a last stage of n < 16 records over the 16 consumer warps: 16 / n warps share a record, each a run of its four chunks.
struct TailShare { unsigned short v[16][16]; };
constexpr TailShare make_tail_share() {
    TailShare t{};
    for (int n = 1; n < 16; ++n) {
        const int wpr = 16 / n;
        for (int w = 0; w < 16; ++w) {
            const int rloc = w / wpr, sub = w - rloc * wpr;
            const int cb = 4 * sub / wpr, ce = 4 * (sub + 1) / wpr;
            t.v[n][w] = (unsigned short)(rloc < n ? (rloc | (cb << 4) | (ce << 7)) : 15);   // 15: no share (first chunk = end chunk = 0)
        }
    }
    return t;
}
static __constant__ TailShare c_tail_share = make_tail_share();

// ---- small helpers ---------------------------------------------------------------------------------
template <int WB> struct IntTables;
template <> struct IntTables<3> { static constexpr uint32_t P0 = 0x00020408u, P1 = 0xFFFEFCF8u; };  // 8 4 2 0 -8 -4 -2 -1
template <> struct IntTables<2> { static constexpr uint32_t P0 = 0xFFFE0002u, P1 = 0u; };           // 2 0 -2 -1

// volatile: stays behind the waits (also volatile) that make the activation planes valid
__device__ __forceinline__ uint2 lds64(uint32_t addr) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ void mma_s8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ int ld_acquire_gpu(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// mbarrier operations by 32-bit shared-window address (no generic-to-shared conversion in the hot loop)
__device__ __forceinline__ bool try_wait_a(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void arrive_a(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// bounded wait, gives up when another thread has (inlined: a call would sit on the critical path)
__device__ __forceinline__ bool wait_a(uint32_t bar, uint32_t parity, volatile int* abort_flag, int limit) {
    for (int it = 0; it < limit; ++it) {
        if (try_wait_a(bar, parity)) return true;
        if ((it & 63) == 63 && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}
__device__ __forceinline__ float lds_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int limit) {
    for (int it = 0; it < limit; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63) == 63 && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}

// One micro-block word -> int8 operands (value * 2^emax): b1 (pa: weights 0..3, pb: 4..7), the routed bytes of
// b2 (qa, qb) and the same bytes at the sign-flipped positions only (fa, fb).
template <int WB, bool K1>
__device__ __forceinline__ void decode_word(uint32_t w, uint32_t lut_lane, uint32_t& pa, uint32_t& pb, uint32_t& qa,
                                            uint32_t& qb, uint32_t& fa, uint32_t& fb) {
    const uint32_t m = w & 0x77777777u, mh = m >> 16;
    pa = prmt_b32(IntTables<WB>::P0, IntTables<WB>::P1, m);
    pb = prmt_b32(IntTables<WB>::P0, IntTables<WB>::P1, mh);
    if constexpr (K1) {   // single-basis weights (Section 3.1, w_hat = c1 b1): no second operand
        qa = qb = fa = fb = 0u;
    } else {
        const uint32_t h = (w & 0x88888888u) * kHashMul;
        const uint4 e = lds128(((h >> 19) & 0x1F80u) | lut_lane);   // selectors x, y; 0xFF at the flipped bytes z, w
        qa = prmt_b32(pa, pb, e.x);
        qb = prmt_b32(pa, pb, e.y);
        fa = qa & e.z;
        fb = qb & e.w;
    }
}

// The range of CTA `cta` of `G` over `units` records, and the order it is walked in.
struct Walk {
    unsigned a, b, L;        // range [a, b), length
    unsigned L1, s1;         // the first L1 positions are records s1, s1+1, ... (the open tile at the end of the range); then a, a+1, ...
    int Ta, Tb, P;           // first and last tile touched, number of tile parts
    bool rot;
};
// No division anywhere: every warp works this out at the start of every linear, on the critical path of a chain of small ones.
__device__ __forceinline__ unsigned mul_shift32(unsigned n, unsigned long long magic) { return (unsigned)(((unsigned long long)n * magic) >> 32); }
// `it`: units, uq, ur (quotient and remainder of units by the number of CTAs), k_blocks, kb_magic
template <class Item>
__device__ __forceinline__ Walk make_walk(const Item& it, int cta, unsigned long long g_magic) {
    Walk w;
    // floor(units c / G) = c (units / G) + floor(c (units % G) / G)
    w.a = (unsigned)cta * it.uq + mul_shift32((unsigned)cta * it.ur, g_magic);
    w.b = (unsigned)(cta + 1) * it.uq + mul_shift32((unsigned)(cta + 1) * it.ur, g_magic);
    w.L = w.b - w.a;
    w.L1 = 0; w.s1 = 0; w.Ta = 0; w.Tb = 0; w.P = 0; w.rot = false;
    if (w.L) {
        const unsigned kb = (unsigned)it.k_blocks;
        w.Ta = (int)mul_shift32(w.a, it.kb_magic);
        w.Tb = (int)mul_shift32(w.b - 1, it.kb_magic);
        w.P = w.Tb - w.Ta + 1;
        w.rot = w.Tb > w.Ta && w.b != mul_shift32(w.b, it.kb_magic) * kb;
        if (w.rot) { w.s1 = (unsigned)w.Tb * kb; w.L1 = w.b - w.s1; }
    }
    return w;
}
__device__ __forceinline__ unsigned walk_record(const Walk& w, unsigned j) { return j < w.L1 ? w.s1 + j : w.a + (j - w.L1); }
__device__ __forceinline__ int walk_part_of_tile(const Walk& w, int T) { return w.rot ? (T == w.Tb ? 0 : 1 + T - w.Ta) : T - w.Ta; }
__device__ __forceinline__ int walk_tile_of_part(const Walk& w, int q) { return w.rot ? (q == 0 ? w.Tb : w.Ta + q - 1) : w.Ta + q; }

// ---- hand-over of one tile part (kept out of line) ------------------------------------------------------
// A consumer warp parks its sums of part number sq (counted per CTA over the whole chain) in reduction slot sq % kTileSlots
// and arrives on the slot's mbarrier; the control warp adds the 16 partials, stores or passes on the result and then
// frees the slot. Returns false after a give-up.
struct FlushCtx {
    uint32_t red_addr;        // shared-window addresses: no 64-bit pointers are kept alive across the record loop
    uint32_t part_bar_addr;
    volatile int* done_gen;
    volatile int* abort_flag;
    int spin;
};
struct Sums4 { float v[4]; };   // by value: the accumulators never have their address taken, so they stay in registers
__device__ __forceinline__ void sts_f32(uint32_t addr, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
template <int NG>
__device__ __forceinline__ bool flush_part(const FlushCtx& c, unsigned sq, Sums4 sums) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int rs = (int)(sq % kTileSlots);
    if (*c.abort_flag) return false;
    if (sq >= (unsigned)kTileSlots) {   // the slot's previous part must have been taken over
        int spins = 0;
        while (c.done_gen[rs] != (int)(sq - kTileSlots + 1)) {
            if (*c.abort_flag || ++spins > c.spin) { *c.abort_flag = 1; return false; }
            __nanosleep(20);
        }
    }
    const uint32_t rb = c.red_addr + (uint32_t)(((rs * kNW + warp) * (NG * 64) + g * 4 + t) * 4);
#pragma unroll
    for (int cg = 0; cg < NG; ++cg) {
        sts_f32(rb + (cg * 64) * 4, sums.v[2 * cg]);
        sts_f32(rb + (cg * 64 + 32) * 4, sums.v[2 * cg + 1]);
    }
    __syncwarp();
    if (lane == 0) arrive_a(c.part_bar_addr + rs * 8);   // releases the warp's stores (ordered before it by the barrier above)
    return true;
}

// sums of one macro-block -> fp32, times the coefficients (outside the inner product, Eq. 4)
template <int NG, bool K1>
__device__ __forceinline__ void group_end(int (&s1)[NG][4], int (&s2)[NG][4], int (&s3)[NG][4], uint32_t cfa, uint32_t cfb, float (&rec)[NG][2]) {
    const float c1a = __half2float(__ushort_as_half((unsigned short)(cfa & 0xFFFFu)));
    const float c2a = __half2float(__ushort_as_half((unsigned short)(cfa >> 16)));
    const float c1b = __half2float(__ushort_as_half((unsigned short)(cfb & 0xFFFFu)));
    const float c2b = __half2float(__ushort_as_half((unsigned short)(cfb >> 16)));
#pragma unroll
    for (int cg = 0; cg < NG; ++cg) {
        // columns 2t, 2t+1 hold the high and low activation slices of one token: S = 256 S_hi + S_lo, exact in int32
        if constexpr (K1) {
            rec[cg][0] += c1a * (float)(s1[cg][0] * 256 + s1[cg][1]);
            rec[cg][1] += c1b * (float)(s1[cg][2] * 256 + s1[cg][3]);
        } else {
            rec[cg][0] += c1a * (float)(s1[cg][0] * 256 + s1[cg][1]) + c2a * (float)((s2[cg][0] - 2 * s3[cg][0]) * 256 + (s2[cg][1] - 2 * s3[cg][1]));
            rec[cg][1] += c1b * (float)(s1[cg][2] * 256 + s1[cg][3]) + c2b * (float)((s2[cg][2] - 2 * s3[cg][2]) * 256 + (s2[cg][3] - 2 * s3[cg][3]));
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) s1[cg][r] = s2[cg][r] = s3[cg][r] = 0;
    }
}

// Sixteen lanes hold the 128 activations of one token and k-block, 8 each (v): Q = rne(x 2^s), the block's largest magnitude in
// [2^14, 2^15), as two int8 planes at hi / hi + plane (byte offsets of this lane's 8), and the scale that undoes it in *scale
// (2^-s, and 2^-emax for the integer weights). `in`: this lane's token exists.
template <int WB>
__device__ __forceinline__ void convert_chunk(const uint4 v, const bool in, unsigned char* hi, int plane, float* scale) {
    const int lane = threadIdx.x & 31;
    const uint32_t in32[4] = {v.x, v.y, v.z, v.w};
    // magnitudes order like their bit patterns: two at a time
    uint32_t amax = __vmaxu2(__vmaxu2(in32[0] & 0x7FFF7FFFu, in32[1] & 0x7FFF7FFFu), __vmaxu2(in32[2] & 0x7FFF7FFFu, in32[3] & 0x7FFF7FFFu));
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) amax = __vmaxu2(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, o));
    amax = max(amax & 0xFFFFu, amax >> 16);
    int sfield = 268 - (int)(amax >> 7);
    sfield = sfield < 1 ? 1 : (sfield > 253 ? 253 : sfield);
    const float mult = __uint_as_float((uint32_t)sfield << 23);
    // Q = rne(x 2^s) without a convert: adding 1.5 * 2^23 leaves the integer in the low mantissa bits. With 128 more in
    // the constant the low 16 bits are 256 hi + (lo + 128) for the split Q = 256 hi + lo, lo in [-128, 127]: the high
    // byte is hi as it stands and the low byte is lo with its top bit flipped. Clamped as raw bits (monotonic):
    // Q = 32640 (all-ones mantissa at the block's top exponent) would need hi = 128; inf and nan saturate.
    uint32_t v16[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint32_t bits = (j & 1) ? (in32[j >> 1] & 0xFFFF0000u) : (in32[j >> 1] << 16);
        const int raw = __float_as_int(fmaf(__uint_as_float(bits), mult, 12582912.0f + 128.0f));
        v16[j] = (uint32_t)max(0x4B400000 + 128 - 32640, min(0x4B400000 + 128 + 32639, raw));
    }
    uint32_t q0[2], q1[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t t01 = prmt_b32(v16[4 * h], v16[4 * h + 1], 0x5410u), t23 = prmt_b32(v16[4 * h + 2], v16[4 * h + 3], 0x5410u);
        q0[h] = prmt_b32(t01, t23, 0x7531u);                   // the four high bytes
        q1[h] = prmt_b32(t01, t23, 0x6420u) ^ 0x80808080u;     // the four low bytes, as signed
    }
    if (in) {
        *reinterpret_cast<uint2*>(hi) = make_uint2(q0[0], q0[1]);
        *reinterpret_cast<uint2*>(hi + plane) = make_uint2(q1[0], q1[1]);
        if ((lane & 15) == 0) *scale = __uint_as_float((uint32_t)(254 - sfield) << 23) * (1.0f / (float)(1 << ((1 << (WB - 1)) - 1)));
    }
}

}  // namespace chain
}  // namespace goq
