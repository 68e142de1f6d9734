// A warp's share of Eq. 4 with bf16 tensor-core fragments (wbits 2..4, group >= 32): a unit record (16 rows x 128 k) from global memory, its decode, and its sums for
// up to 16 tokens. Lane (g, t) owns whole micro-blocks of rows g and g + 8 of the weights and 8 of every 32 k of tokens g, g + 8.
#pragma once
#include "goq_stream_core.cuh"

namespace goq {
namespace gmma {

// weights of a record as a lane holds them: 8 micro-block words, (W4) their records, the coefficient pairs of rows g and g + 8
template <int WB, int GPB> struct Record {
    uint4 w0, w1;
    uint32_t m0, m1;
    uint32_t ca[GPB], cb[GPB];
    __device__ __forceinline__ void load(const uint8_t* unit, int meta_off) {
        const int lane = threadIdx.x & 31, g = lane >> 2;
        w0 = __ldcs(reinterpret_cast<const uint4*>(unit) + lane);
        w1 = __ldcs(reinterpret_cast<const uint4*>(unit) + 32 + lane);
        if constexpr (WB == 4) {
            m0 = __ldcs(reinterpret_cast<const uint32_t*>(unit + meta_off) + lane);
            m1 = __ldcs(reinterpret_cast<const uint32_t*>(unit + meta_off + 128) + lane);
        }
        const uint32_t* c = reinterpret_cast<const uint32_t*>(unit + kCodeBytesPerUnit) + g;
#pragma unroll
        for (int jj = 0; jj < GPB; ++jj) { ca[jj] = __ldcs(c + jj * 16); cb[jj] = __ldcs(c + jj * 16 + 8); }
    }
};

// One micro-block word -> bf16x2 operands R (b1, elements 2q, 2q + 1) and Q (b2). `entry`: the record's table entry.
template <int WB>
__device__ __forceinline__ void expand(uint32_t w, uint32_t ha, uint32_t hb, uint32_t la, uint32_t lb, const uint4 e, uint32_t (&R)[4], uint32_t (&Q)[4]) {
    R[0] = prmt_b32(la, ha, 0x5140u); R[1] = prmt_b32(la, ha, 0x7362u);
    R[2] = prmt_b32(lb, hb, 0x5140u); R[3] = prmt_b32(lb, hb, 0x7362u);
    const uint32_t qha = prmt_b32(ha, hb, e.x) ^ e.z, qhb = prmt_b32(ha, hb, e.y) ^ e.w;
    const uint32_t qla = prmt_b32(la, lb, e.x), qlb = prmt_b32(la, lb, e.y);
    Q[0] = prmt_b32(qla, qha, 0x5140u); Q[1] = prmt_b32(qla, qha, 0x7362u);
    Q[2] = prmt_b32(qlb, qhb, 0x5140u); Q[3] = prmt_b32(qlb, qhb, 0x7362u);
}
template <int WB>
__device__ __forceinline__ void decode(uint32_t w, uint32_t record, const unsigned char* lut, uint32_t lane16, uint32_t (&R)[4], uint32_t (&Q)[4]) {
    const uint32_t m = w & 0x77777777u, mh = m >> 16;
    uint32_t ha, hb, la, lb, slot_off;
    if constexpr (WB <= 3) {
        ha = prmt_b32(PotBytes<WB>::H0, PotBytes<WB>::H1, m); hb = prmt_b32(PotBytes<WB>::H0, PotBytes<WB>::H1, mh);
        la = prmt_b32(PotBytes<WB>::L0, PotBytes<WB>::L1, m); lb = prmt_b32(PotBytes<WB>::L0, PotBytes<WB>::L1, mh);
        slot_off = (((w - m) * kHashMul) >> 19) & 0x1F80u;
    } else {
        // code = sign << 3 | e, value (-1)^sign 2^-e, sign 0 with e = 7 is the zero. bf16(2^-e) = (127 - e) << 7: the low byte does not
        // depend on the sign; the high byte comes from a table per sign (the positive one holds 0 at e = 7), chosen per byte by a
        // mask that prmt's sign-replicate mode makes of the sign bits (top bit of each byte of w: odd weights; of w << 4: even).
        // The zero's low byte 0x00 (e odd) makes it +0 and, flipped, -0.
        constexpr uint32_t PH0 = 0x3E3E3F3Fu, PH1 = 0x003C3D3Du, NH0 = 0xBEBEBFBFu, NH1 = 0xBCBCBDBDu, LL = 0x00800080u;
        const uint32_t s_odd = prmt_b32(w, 0u, 0xBA98u), s_even = prmt_b32(w << 4, 0u, 0xBA98u);
        const uint32_t ma = prmt_b32(s_even, s_odd, 0x5140u), mb = prmt_b32(s_even, s_odd, 0x7362u);
        ha = (prmt_b32(PH0, PH1, m) & ~ma) | (prmt_b32(NH0, NH1, m) & ma);
        hb = (prmt_b32(PH0, PH1, mh) & ~mb) | (prmt_b32(NH0, NH1, mh) & mb);
        la = prmt_b32(LL, LL, m); lb = prmt_b32(LL, LL, mh);
        slot_off = (record & 63u) << 7;
    }
    const uint4 e = *reinterpret_cast<const uint4*>(lut + (slot_off | lane16));
    expand<WB>(w, ha, hb, la, lb, e, R, Q);
}

// the record table (64 x kLutCopies entries) by all threads of the CTA
template <int WB>
__device__ __forceinline__ void fill_table(unsigned char* lut) {
    for (int i = threadIdx.x; i < 64 * kLutCopies; i += blockDim.x) {
        int slot = i / kLutCopies;
        if constexpr (WB == 4) slot = (int)record_slot((uint32_t)slot);   // table in record order
        const uint32_t* e = c_exchange_lut.v[slot];
        *reinterpret_cast<uint4*>(lut + (size_t)i * 16) = make_uint4(e[0], e[1], e[2], e[3]);
    }
}
// xp: each token's row + 8 t. Past the end of a row: zeros (the weights there are zero too)
template <int NT>
__device__ __forceinline__ void load_activations(const uint16_t* const (&xp)[NT], int bk, int k_in, uint4 (&xa)[NT][4]) {
    const int t = threadIdx.x & 3, k0 = bk * kBlockK;
    const bool inside = k0 + kBlockK <= k_in;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            xa[nt][c] = make_uint4(0u, 0u, 0u, 0u);
            if (inside || k0 + c * 32 + t * 8 < k_in) xa[nt][c] = *reinterpret_cast<const uint4*>(xp[nt] + k0 + c * 32);
        }
}
// acc[nt][r]: row g + 8 (r >> 1), token 8 nt + 2 t + (r & 1)
template <int WB, int NT, int CPG>
__device__ __forceinline__ void add_record(const Record<WB, 4 / CPG>& rec, const uint4 (&xa)[NT][4], const unsigned char* lut, uint32_t lane16, float (&acc)[NT][4]) {
    const uint32_t w0[4] = {rec.w0.x, rec.w0.y, rec.w0.z, rec.w0.w}, w1[4] = {rec.w1.x, rec.w1.y, rec.w1.z, rec.w1.w};
    float d1[NT][4], d2[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int r = 0; r < 4; ++r) d1[nt][r] = d2[nt][r] = 0.f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint32_t R0[4], Q0[4], R1[4], Q1[4];
        decode<WB>(w0[c], WB == 4 ? rec.m0 >> (8 * c) : 0u, lut, lane16, R0, Q0);
        decode<WB>(w1[c], WB == 4 ? rec.m1 >> (8 * c) : 0u, lut, lane16, R1, Q1);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const uint4 x = xa[nt][c];
            mma_bf16(d1[nt], R0[0], R1[0], R0[1], R1[1], x.x, x.y);
            mma_bf16(d2[nt], Q0[0], Q1[0], Q0[1], Q1[1], x.x, x.y);
            mma_bf16(d1[nt], R0[2], R1[2], R0[3], R1[3], x.z, x.w);
            mma_bf16(d2[nt], Q0[2], Q1[2], Q0[3], Q1[3], x.z, x.w);
        }
        if (((c + 1) % CPG) == 0) {
            const int jj = c / CPG;
            const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&rec.ca[jj]));   // (c1, c2) of row g, of row g + 8
            const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&rec.cb[jj]));
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                acc[nt][0] += a.x * d1[nt][0] + a.y * d2[nt][0];
                acc[nt][1] += a.x * d1[nt][1] + a.y * d2[nt][1];
                acc[nt][2] += b.x * d1[nt][2] + b.y * d2[nt][2];
                acc[nt][3] += b.x * d1[nt][3] + b.y * d2[nt][3];
#pragma unroll
                for (int r = 0; r < 4; ++r) d1[nt][r] = d2[nt][r] = 0.f;
            }
        }
    }
}

}  // namespace gmma
}  // namespace goq
