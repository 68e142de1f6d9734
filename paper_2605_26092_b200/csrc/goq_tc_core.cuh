// Device helpers shared by the tcgen05 kernels: mbarrier / TMA wrappers with bounded waits, tensor memory, shared-memory
// operand descriptors, and the decode of a micro-block word into fp16 operands (Section 3.3 of the paper: b2 is b1 routed by
// "partner i XOR s" with pair signs).
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include "goq_common.cuh"

namespace goq {
namespace tc {

constexpr int kLutCopies = 8;   // record table, one copy per lane & 7: lookups are bank-conflict free
constexpr int kLutBytes = 64 * kLutCopies * 16;
constexpr int kSpin = 1 << 22;

__device__ __forceinline__ uint32_t s32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s32(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(s32(b)), "r"(parity) : "memory");
    return ok != 0;
}
// probe without suspending (try_wait holds an early caller back for microseconds)
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(s32(b)), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag, int limit = kSpin) {
    for (int it = 0; it < limit; ++it) {
        if (mbar_try(b, parity)) return true;
        if ((it & 63) == 63 && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}
// Copies and MMAs in flight must land before a CTA that has given up lets go of its shared and tensor memory. Their barriers may count
// arrivals that never come, so this waits a time that none of them takes (a millisecond). Every thread calls it, behind the last barrier.
__device__ __forceinline__ void settle_after_give_up() {
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    __syncthreads();
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(s32(dst)),
                 "l"(src), "r"(bytes), "r"(s32(bar)) : "memory");
}
// 2-D tiled TMA load (no multicast): coordinates {c0 = k element, c1 = token row}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int c0, int c1, uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(s32(dst)), "l"(map), "r"(c0), "r"(c1), "r"(s32(bar)) : "memory");
}
// ... 3-D: packed records, {c0 = 8-byte element of a piece, c1 = piece of the row of records, c2 = row tile}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(s32(dst)), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(s32(bar)) : "memory");
}
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ uint32_t after_wait(uint32_t addr) {
    uint32_t r;
    asm volatile("mov.u32 %0, %1;" : "=r"(r) : "r"(addr) : "memory");
    return r;
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint32_t pack_f16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// true in one lane of a warp that runs as one
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

// ---- tensor memory and MMA ---------------------------------------------------------------------
template <int COLS>
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_slot) {  // whole warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(smem_slot)), "n"(COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
template <int COLS>
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr) {  // whole warp
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "n"(COLS) : "memory");
}
// K-major operand tile with 128-byte swizzle: rows of 128 bytes, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);        // start address
    d |= (uint64_t)1 << 16;                          // leading byte offset (unused for this layout)
    d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset between 8-row groups
    d |= (uint64_t)1 << 46;                          // descriptor version for sm_100
    d |= (uint64_t)2 << 61;                          // SWIZZLE_128B
    return d;
}
// kind::f16 instruction descriptor: fp32 accumulate, fp16 x fp16 (format fields 0), both K-major, M = 128
__host__ __device__ constexpr uint32_t idesc_f16(uint32_t n) { return (1u << 4) | ((n >> 3) << 17) | ((128u >> 4) << 24); }
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}


// ---- record decode (same tables as the decode GEMV) --------------------------------------------
// High byte of the fp16 number of every PoT state, by code (the low byte of a power of two is zero).
template <int WB> struct PotBytes;
template <> struct PotBytes<3> {  // +1 +.5 +.25 0 -1 -.5 -.25 -.125
    static constexpr uint32_t H0 = 0x0034383Cu, H1 = 0xB0B4B8BCu;
};
template <> struct PotBytes<2> {  // +1 0 -1 -.5
    static constexpr uint32_t H0 = 0xB8BC003Cu, H1 = 0u;
};
// W4: code = sign << 3 | e, value (-1)^sign 2^-e (fp16 high byte (15 - e) << 2), sign 0 with e = 7 is the zero state
struct PotBytes4 {
    static constexpr uint32_t PH0 = 0x3034383Cu, PH1 = 0x0024282Cu, NH0 = 0xB0B4B8BCu, NH1 = 0xA0A4A8ACu;
};
constexpr uint32_t kHashMul = 0x01008420u;  // (record bits in place) * kHashMul >> 26 is a bijection onto 0..63

struct ExchangeLut { uint32_t v[64][4]; };
constexpr ExchangeLut make_exchange_lut() {
    ExchangeLut t{};
    for (uint32_t meta = 0; meta < 64; ++meta) {
        const int s = (int)(meta & 3u) + 1;
        // flips: bit i = 1 iff b2 element i has the opposite sign of the b1 element routed to it
        uint32_t flips = 0;
        int p = 0;
        for (int i = 0; i < 8; ++i) {
            const int j = i ^ s;
            if (i < j) {
                const uint32_t f = (meta >> (2 + p)) & 1u;  // 1 iff eta = -1
                flips |= (f ^ 1u) << i;                     // y_i = -eta x_j
                flips |= f << j;                            // y_j =  eta x_i
                ++p;
            }
        }
        uint32_t sel_a = 0, sel_b = 0, f_a = 0, f_b = 0, spread = 0;
        for (int i = 0; i < 4; ++i) {
            sel_a |= (uint32_t)(i ^ s) << (4 * i);
            sel_b |= (uint32_t)((4 + i) ^ s) << (4 * i);
            f_a |= ((flips >> i) & 1u) << (8 * i + 7);
            f_b |= ((flips >> (4 + i)) & 1u) << (8 * i + 7);
        }
        for (int i = 0; i < 6; ++i) spread |= ((meta >> i) & 1u) << (4 * i + 3);
        const uint32_t slot = (uint32_t)(spread * kHashMul) >> 26;
        t.v[slot][0] = sel_a; t.v[slot][1] = sel_b; t.v[slot][2] = f_a; t.v[slot][3] = f_b;
    }
    return t;
}
static __constant__ ExchangeLut c_lut = make_exchange_lut();

__device__ __forceinline__ uint32_t hmul2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t hfma2(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}
// One micro-block word -> the fp16 values of b1 (R) and b2 (Q), two weights per register: the high byte of every value comes from
// a byte table (a power of two's low byte is zero).
// W <= 3: the exchange record sits in the spare bit of the word's nibbles and is hashed into the table slot. W = 4: the
// nibbles are full (the sign is bit 3), the record comes from the unit's byte plane (`record`) and the table is filled
// in record order; the high byte is taken from a positive or a negative table per weight, chosen by a byte mask that
// prmt's sign-replicate mode makes of the sign bits (top bit of each byte of w: odd weights; of w << 4: even weights).
// ADD: the table lies at any 1 KiB boundary (one more addition a word).
template <int WB, bool ADD = false>
__device__ __forceinline__ void expand_bases(uint32_t w, uint32_t record, uint32_t lut_lane, uint32_t (&R)[4], uint32_t (&Q)[4]) {
    const uint32_t m = w & 0x77777777u, mh = m >> 16;
    uint32_t ha, hb, slot_off;
    if constexpr (WB <= 3) {
        ha = prmt(PotBytes<WB>::H0, PotBytes<WB>::H1, m);
        hb = prmt(PotBytes<WB>::H0, PotBytes<WB>::H1, mh);
        slot_off = (((w - m) * kHashMul) >> 19) & 0x1F80u;
    } else {
        const uint32_t s_odd = prmt(w, 0u, 0xBA98u), s_even = prmt(w << 4, 0u, 0xBA98u);
        const uint32_t ma = prmt(s_even, s_odd, 0x5140u), mb = prmt(s_even, s_odd, 0x7362u);   // weights 0..3, 4..7
        ha = (prmt(PotBytes4::PH0, PotBytes4::PH1, m) & ~ma) | (prmt(PotBytes4::NH0, PotBytes4::NH1, m) & ma);
        hb = (prmt(PotBytes4::PH0, PotBytes4::PH1, mh) & ~mb) | (prmt(PotBytes4::NH0, PotBytes4::NH1, mh) & mb);
        slot_off = (record & 63u) << 7;
    }
    const uint4 e = lds128(ADD ? slot_off + lut_lane : slot_off | lut_lane);  // table is 8 KiB aligned, lut_lane selects the copy
    const uint32_t qa = prmt(ha, hb, e.x) ^ e.z, qb = prmt(ha, hb, e.y) ^ e.w;   // b2: permuted, pair signs applied
    // bytes {0, h[2q], 0, h[2q+1]}: weights 2q, 2q+1 as one f16x2 word
    R[0] = prmt(ha, 0u, 0x1404u); R[1] = prmt(ha, 0u, 0x3424u); R[2] = prmt(hb, 0u, 0x1404u); R[3] = prmt(hb, 0u, 0x3424u);
    Q[0] = prmt(qa, 0u, 0x1404u); Q[1] = prmt(qa, 0u, 0x3424u); Q[2] = prmt(qb, 0u, 0x1404u); Q[3] = prmt(qb, 0u, 0x3424u);
}
// w_hat = c1*b1 + c2*b2 in fp16. c1, c2: the coefficient in both halves of a register. c1*b1 is a power-of-two scaling (exact)
// and the fused multiply-add rounds once: the same value as fp32 arithmetic rounded to fp16.
template <int WB, bool ADD = false>
__device__ __forceinline__ void expand_what(uint32_t w, uint32_t record, uint32_t lut_lane, uint32_t c1, uint32_t c2, uint32_t (&out)[4]) {
    uint32_t R[4], Q[4];
    expand_bases<WB, ADD>(w, record, lut_lane, R, Q);
#pragma unroll
    for (int q = 0; q < 4; ++q) out[q] = hfma2(c2, Q[q], hmul2(c1, R[q]));
}

// The record table in shared memory (8 KiB aligned), eight bank-disjoint copies; W4 in record order.
template <int WB>
__device__ __forceinline__ void fill_lut(unsigned char* lut, int tid, int n_threads) {
    for (int i = tid; i < 64 * kLutCopies; i += n_threads) {
        uint32_t slot = (uint32_t)(i / kLutCopies);
        if constexpr (WB == 4) {
            uint32_t spread = 0;
            for (int b = 0; b < 6; ++b) spread |= ((slot >> b) & 1u) << (4 * b + 3);
            slot = (spread * kHashMul) >> 26;
        }
        const uint32_t* e = c_lut.v[slot];
        *reinterpret_cast<uint4*>(lut + (size_t)i * 16) = make_uint4(e[0], e[1], e[2], e[3]);
    }
}

// host side, defined in goq_gemm_tc.cu
cudaError_t encode_x_map(CUtensorMap* map, void* xh, int k_in, int m, int rows);
cudaError_t encode_i8_map(CUtensorMap* map, const void* x, int k_in, int m, int rows);
cudaError_t encode_f32_map(CUtensorMap* map, const float* w, int cols, int rows, int bc, int br);
// packed records as boxes of one k-block x `row_tiles` row tiles (8-byte elements; rows past the end read as zeros). A record is one
// piece, or two where it has more elements than a box row may (W4 in groups of 8: 288).
inline int packed_pieces(const Geometry& g) { return g.unit_bytes / 8 > 256 ? 2 : 1; }
bool packed_map_supported(const Geometry& g);
cudaError_t encode_packed_map(CUtensorMap* map, const void* packed, const Geometry& g, int row_tiles);
cudaError_t launch_x_to_f16(const void* x, int k_in, int m, uint16_t* xh, float* inv_scale, cudaStream_t st);
// ... and, with `row_tiles` CTAs more, the channel scales
cudaError_t launch_pre_pass(const void* x, int k_in, int m, int row_tiles, uint16_t* xh, float* inv_scale, const void* packed,
                            int unit_bytes, int k_blocks, int gpb, uint32_t* row_scale, float* row_inv, cudaStream_t st);

}  // namespace tc
}  // namespace goq
