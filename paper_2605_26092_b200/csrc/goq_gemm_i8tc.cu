// Integer-activation layer (Eq. 4 with integer X~ and c~) on tcgen05 int8 tensor cores, exact in int32.
//
//   ACC_b[m,n] = sum_j c~_b[n,j] sum_{k in j} x~[m,k] v_b[n,k],   v_b = 2^emax b_b in {0, +-1, .. +-2^emax}
//
// The coefficient changes every macro-block while a tensor-core accumulator does not, so it goes into the operand: c~ v needs 11 bits
// (W3), two int8 digits: c~ v = B h + l, B = 16 (W2, W3) or 192 (W4), ACC = B sum x h + sum x l. All integers, summed modulo 2^32;
// the result is below 2^31 by the host's bound, so it is the same bits in any order. Four digit planes (two bases x two digits) of
// 64 channels make one N = 256 operand; a CTA's tile is 256 tokens (two M = 128 halves) x 64 channels, its accumulators all of tensor
// memory.
// Against per-macro-block sums in registers (mma.sync) this doubles the multiply-adds and takes the coefficient stage, eight
// integer multiply-adds per four MMAs, out of the loop.
//
// Digits come from byte tables: 256 entries, one per value of c~, of the digits of c~ v for every code, looked up per row and
// macro-block (16 bytes: h and l of eight codes); a weight is then two byte permutes. b2 = the same lookup routed by the exchange
// record; its pair signs negate bytes. For B = 16 both digits are chosen non-zero, so a byte's negation is (~q) + 1 without a
// carry into the next byte; for B = 192 the addition masks the top bits.
//
// Roles (27 warps, persistent CTAs): 0-7 epilogue (a thread is a token: ACC or y, eight channels a store), 8 packed records (one TMA
// copy per 64 channels x 128 k), 9 activation tiles (TMA), 10 MMA issue, 11-26 decode: two groups of eight alternate k-blocks, warp (e, v)
// of a group takes rows 8 v .. of record e. Bound: shared-memory bandwidth (per 64 x 256 x 128: operand reads of the MMAs ~770 clocks, digit
// stores, lookups and copies ~900). With 128 x 128 tiles the second part was twice that and the kernel ran at its sum (98 %).
// Every mbarrier wait is bounded; a CTA that gives up leaves its outputs unwritten, reports GOQ_ERR_TIMEOUT where it is given a
// status word, and makes every token's largest magnitude NaN where those are recorded (the caller without scratch sees that).
#include "goq_tc_core.cuh"
#include "goq_internal.h"

namespace goq {
namespace i8tc {

using namespace tc;

constexpr int kEpiWarps = 8, kPkWarp = 8, kXWarp = 9, kMmaWarp = 10, kDec0 = 11, kDecWarps = 16;
constexpr int kDecGroups = 2;   // decoding groups: group i takes the k-blocks u with u % 2 == i
constexpr int kThreads = (kDec0 + kDecWarps) * 32;
constexpr int kTokens = 128, kChannels = 64, kStages = 3, kMaxPk = 4;
constexpr int kABytes = kTokens * 128, kBBytes = 256 * 128, kStageBytes = kBBytes + 2 * kABytes;
constexpr int kLut8Bytes = 64 * 16 * 8;   // record table: 8-byte entries, 16 copies

struct Params {
    const uint8_t* packed;
    const int8_t* cq;
    const float *sx, *sc;
    void* y;
    int32_t* acc;
    float* amax;
    int* status;
    int unit_bytes, meta_off, k_blocks, groups_in, n_out, m, y_dtype, tiles_x, tiles, n_pk;
    int tt;   // M = 128 operands per tile: 1 or 2
    int spin;   // bound of every wait, in polls
};

// kind::i8: s8 x s8 -> s32, both K-major, M = 128, N = 256
constexpr uint32_t kIdesc = (2u << 4) | (1u << 7) | (1u << 10) | ((256u >> 3) << 17) | ((128u >> 4) << 24);
__device__ __forceinline__ void umma_i8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(kIdesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, int (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(taddr) : "memory");
}
// 32 bytes a thread: a whole sector, and half the address-divergent requests of two 16-byte stores
__device__ __forceinline__ void st_global_v8(float* d, const float (&v)[8]) {
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(d), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]),
                 "f"(v[6]), "f"(v[7]) : "memory");
}
__device__ __forceinline__ uint2 lds64(uint32_t addr) {
    uint2 v;
    asm("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts64(uint32_t addr, uint32_t a, uint32_t b) {
    asm volatile("st.shared.v2.u32 [%0], {%1,%2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}

// Slots of the packed-record ring: as many as fit. A multiple of the decoding groups, so that a slot always comes round to the same
// group: a barrier has one phase bit, and a group that does not wait for every phase of a slot may find the one before the last
// completed, take it for its own and decode the records it left.
constexpr int kSmemBytes = 227 * 1024 - 2 * 1024;   // the static variables take less than 2 KiB
constexpr int fixed_bytes(int lut_entry) { return 1024 + kStages * kStageBytes + kLut8Bytes + 256 * lut_entry; }
constexpr int ring_slots(int unit_bytes, int lut_entry) {
    const int n = (kSmemBytes - fixed_bytes(lut_entry)) / (4 * unit_bytes);
    return (n < kMaxPk ? n : kMaxPk) / kDecGroups * kDecGroups;
}

// W4: |c~ v| <= 2^14 = 85.3 * 192, and |l| <= 96: both digits and their negatives are int8 for every c~, -128 included
template <int WB> struct Digits { static constexpr int base = WB == 4 ? 192 : 16, entry = WB == 4 ? 32 : 16; };
// integer of code c (W4: sign << 3 | e): +-2^(emax - e)
template <int WB>
__device__ __forceinline__ int code_int(int c) {
    constexpr int emax = (1 << (WB - 1)) - 1;
    const int sg = c >> (WB - 1), e = c & emax;
    if (!sg && e == emax) return 0;
    return sg ? -(1 << (emax - e)) : 1 << (emax - e);
}
template <int WB>
__device__ __forceinline__ void split_digits(int v, int& h, int& l) {
    constexpr int B = Digits<WB>::base;
    h = (v + B / 2 + 256 * B) / B - 256;   // floor
    l = v - B * h;
    if constexpr (WB <= 3) {   // both non-zero
        if (l == 0) { h += 1; l = -B; }
        if (h == 0) {          // |v| < 8, or 16 - 16
            const int up = l < 0 ? -1 : 1;
            h = up; l -= up * B;
            if (l == 0) { h += up; l -= up * B; }
        }
    }
}

template <int WB, int GPB>
__global__ void __launch_bounds__(kThreads, 1)
gemm_i8tc_kernel(const Params p, const __grid_constant__ CUtensorMap x_map, const __grid_constant__ CUtensorMap packed_map) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* stages = smem_raw + ((1024u - (s32(smem_raw) & 1023u)) & 1023u);
    unsigned char* lut = stages + kStages * kStageBytes;
    unsigned char* ctab = lut + kLut8Bytes;                              // [c~ as a byte][h of 8 codes, l of 8 codes (W4: +, - of each)]
    unsigned char* pk_ring = ctab + 256 * Digits<WB>::entry;
    const int pk_bytes = 4 * p.unit_bytes;
    __shared__ uint64_t full[kStages], empty[kStages], pk_full[kMaxPk], pk_empty[kMaxPk], tm_full[2], tm_empty[2];
    // Per-channel scales of the current tile and its neighbours. Both token halves write a tile's (the same values); a half that
    // has finished tile i + 2 knows the other to be past tile i, whose buffer tile i + 3 takes.
    __shared__ float2 sc_s[3][kChannels];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
    const int my_tiles = (p.tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x, units = my_tiles * p.k_blocks;

    // packed records of the CTA's tiles, k-block by k-block
    struct { int tile, kb, slot, round, issued; } pk = {(int)blockIdx.x, 0, 0, 0, 0};
    auto pk_issue = [&]() {
        mbar_expect_tx(&pk_full[pk.slot], (uint32_t)pk_bytes);   // (rows past the last tile arrive as zeros)
        tma_load_3d(pk_ring + pk.slot * pk_bytes, &packed_map, 0, pk.kb, (pk.tile % p.tiles_x) * 4, &pk_full[pk.slot]);   // (groups of 32 or more: one piece a record)
        if (++pk.kb == p.k_blocks) { pk.kb = 0; pk.tile += (int)gridDim.x; }
        ++pk.issued;
        if (++pk.slot == p.n_pk) { pk.slot = 0; ++pk.round; }
    };
    if (warp == kPkWarp && lane == 0) {
        for (int i = 0; i < kMaxPk; ++i) { mbar_init(&pk_full[i], 1); mbar_init(&pk_empty[i], 8); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid == 0) {
        abort_flag = 0;
        for (int i = 0; i < kStages; ++i) { mbar_init(&full[i], 8 + 1); mbar_init(&empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&tm_full[i], 1); mbar_init(&tm_empty[i], kEpiWarps / 2); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // record table: byte selector of b2's first half (the second half's is this XOR 0x4444) and the flips of both halves, bit 7 and bit 6
    for (int i = tid; i < 64 * 16; i += kThreads) {
        uint32_t slot = (uint32_t)(i >> 4);
        if constexpr (WB == 4) {
            uint32_t spread = 0;
            for (int b = 0; b < 6; ++b) spread |= ((slot >> b) & 1u) << (4 * b + 3);
            slot = (spread * kHashMul) >> 26;
        }
        const uint32_t* e = c_lut.v[slot];
        *reinterpret_cast<uint2*>(lut + (size_t)i * 8) = make_uint2(e[0], e[2] | (e[3] >> 1));
    }
    for (int i = tid; i < 256 * (WB == 2 ? 4 : WB == 3 ? 8 : 16); i += kThreads) {
        constexpr int NC = WB == 2 ? 4 : WB == 3 ? 8 : 16;
        const int c = (int)(int8_t)(i / NC), code = i % NC;
        int h, l;
        split_digits<WB>(c * code_int<WB>(code), h, l);
        // W <= 3: h at bytes 0..7, l at 8..15.  W4: h of + (by e) 0..7, h of - 8..15, l of + 16..23, l of - 24..31
        unsigned char* d = ctab + (i / NC) * Digits<WB>::entry + code;
        d[0] = (unsigned char)(int8_t)h;
        d[Digits<WB>::entry / 2] = (unsigned char)(int8_t)l;
        if constexpr (WB == 2) { d[4] = 0; d[12] = 0; }   // codes 4..7 do not occur
    }
    if (warp == kMmaWarp) tmem_alloc<512>(&tmem_slot);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the packed weights, like everything else, only after earlier kernels
    const uint32_t tmem_base = tmem_slot;

    if (warp == kPkWarp) {
        if (lane == 0) {
            bool ok = true;
            while (pk.issued < units && ok) {
                if (pk.round > 0) ok = mbar_wait(&pk_empty[pk.slot], (pk.round - 1) & 1, &abort_flag, p.spin);
                if (ok) pk_issue();
            }
        }
    } else if (warp == kXWarp) {
        if (lane == 0) {
            bool ok = true;
            int u = 0;
            for (int tile = blockIdx.x; tile < p.tiles && ok; tile += gridDim.x)
                for (int kb = 0; kb < p.k_blocks; ++kb, ++u) {
                    const int s = u % kStages;
                    if (u >= kStages) ok = mbar_wait(&empty[s], ((u / kStages) - 1) & 1, &abort_flag, p.spin);
                    if (!ok) break;
                    mbar_expect_tx(&full[s], (uint32_t)(p.tt * kABytes));
                    for (int i = 0; i < p.tt; ++i)
                        tma_load_2d(stages + s * kStageBytes + kBBytes + i * kABytes, &x_map, kb * kBlockK, ((tile / p.tiles_x) * p.tt + i) * kTokens, &full[s]);
                }
        }
    } else if (warp == kMmaWarp) {
        const uint64_t bdesc0 = smem_desc_sw128(s32(stages)), adesc0 = smem_desc_sw128(s32(stages + kBBytes));
        const bool leader = elect_one();
        bool ok = true, ready = false;
        int s = 0;
        uint32_t par = 0;
        for (int i = 0; i < my_tiles && ok; ++i) {
            for (int kb = 0; kb < p.k_blocks; ++kb) {
                if (!ready) ok = mbar_wait(&full[s], par, &abort_flag, p.spin);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                const int s_next = s + 1 == kStages ? 0 : s + 1;
                const uint32_t par_next = s_next == 0 ? par ^ 1u : par;
                ready = mbar_test(&full[s_next], par_next);
                const uint64_t ad = adesc0 + (uint32_t)(s * (kStageBytes >> 4)), bd = bdesc0 + (uint32_t)(s * (kStageBytes >> 4));
                for (int h = 0; h < p.tt; ++h) {   // 128 tokens each
                    if (kb == 0 && i > 0) {
                        ok = __all_sync(0xFFFFFFFFu, mbar_wait(&tm_empty[h], (i - 1) & 1, &abort_flag, p.spin));
                        if (!ok) break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    if (leader) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            umma_i8(tmem_base + h * 256, ad + h * (kABytes >> 4) + 2 * ks, bd + 2 * ks, (kb > 0 || ks > 0) ? 1u : 0u);
                        if (kb == p.k_blocks - 1) umma_commit(&tm_full[h]);
                    }
                }
                if (!ok) break;
                if (leader) umma_commit(&empty[s]);   // (the last one arrives with the accumulators', a tile's epilogue before the CTA leaves)
                __syncwarp();
                s = s_next; par = par_next;
            }
        }
    } else if (warp >= kDec0) {
        // ------------------------------ decode: packed records -> digit planes ------------------------------
        const int group = (warp - kDec0) >> 3, e = ((warp - kDec0) >> 1) & 3, v = (warp - kDec0) & 1, g = lane >> 2, t = lane & 3;
        const uint32_t lut_lane = s32(lut) + (uint32_t)(lane & 15) * 8, ctab_a = s32(ctab);
        // Row r of a plane: 128 bytes, 16-byte piece j at j ^ (r & 7). Odd rows take their words in the order c ^ 2: the four rows of a
        // half warp's store then cover all eight pieces.
        const int flip = (g & 1) * 2;
        uint32_t off[4];
#pragma unroll
        for (int ci = 0; ci < 4; ++ci)
            off[ci] = (uint32_t)((e * 16 + v * 8 + g) * 128 + (((2 * (ci ^ flip) + (t >> 1)) ^ g) << 4) + (t & 1) * 8);
        int tile = blockIdx.x, kb = 0;
        auto step = [&]() { if (++kb == p.k_blocks) { kb = 0; tile += gridDim.x; } };
        if (group) step();
        uint32_t next_c[GPB];
        auto fetch = [&]() {   // (c~_1, c~_2) of this lane's row, the k-block's macro-blocks; then step on
            const int row = (tile % p.tiles_x) * kChannels + e * 16 + v * 8 + g;
#pragma unroll
            for (int jj = 0; jj < GPB; ++jj) {
                const int j = kb * GPB + jj;
                next_c[jj] = (row < p.n_out && j < p.groups_in) ? (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(p.cq) + (size_t)row * p.groups_in + j) : 0u;
            }
            step(); step();
        };
        if (group < units) fetch();
        bool ok = true;
        int slot = group, s = group;   // n_pk is even: a slot belongs to one group
        uint32_t pk_par = 0, st_par = 1;   // st_par: parity of the stage's previous release (the first round passes at once)
        for (int u = group; u < units; u += 2) {
            uint32_t cc[GPB];
#pragma unroll
            for (int jj = 0; jj < GPB; ++jj) cc[jj] = next_c[jj];
            if (u + 2 < units) fetch();
            ok = __all_sync(0xFFFFFFFFu, mbar_wait(&pk_full[slot], pk_par, &abort_flag, p.spin));
            if (!ok) break;
            const uint32_t unit = after_wait(s32(pk_ring) + slot * pk_bytes + e * p.unit_bytes);
            const uint4 wv = lds128(unit + v * 512 + lane * 16);
            uint32_t mv = 0u;
            if constexpr (WB == 4) mv = lds32(unit + p.meta_off + v * 128 + lane * 4);
            const bool odd = flip != 0;
            const uint32_t w[4] = {odd ? wv.z : wv.x, odd ? wv.w : wv.y, odd ? wv.x : wv.z, odd ? wv.y : wv.w};
            if constexpr (WB == 4) mv = odd ? __funnelshift_l(mv, mv, 16) : mv;
            ok = __all_sync(0xFFFFFFFFu, mbar_wait(&empty[s], st_par, &abort_flag, p.spin));
            if (!ok) break;
            const uint32_t at = s32(stages) + (uint32_t)(s * kStageBytes);
#pragma unroll
            for (int ci = 0; ci < 4; ++ci) {
                // macro-block of chunk ci ^ flip: with four, odd rows go through them in the other order; with two, likewise by halves
                const uint32_t c12 = GPB == 1 ? cc[0] : GPB == 2 ? (odd ? cc[(ci >> 1) ^ 1] : cc[ci >> 1]) : (odd ? cc[(ci ^ 2) & (GPB - 1)] : cc[ci & (GPB - 1)]);
                const uint32_t m = w[ci] & 0x77777777u, mh = m >> 16;
                const uint32_t slot_off = WB <= 3 ? (((w[ci] - m) * kHashMul) >> 19) & 0x1F80u : ((mv >> (8 * ci)) & 63u) << 7;
                const uint2 ex = lds64(slot_off + lut_lane);
                uint32_t b1[4], b2[4];   // h of weights 0..3, 4..7; l likewise
                if constexpr (WB <= 3) {
                    const uint4 t1 = lds128(ctab_a + (c12 & 255u) * 16u), t2 = lds128(ctab_a + (c12 >> 8) * 16u);
                    b1[0] = prmt(t1.x, t1.y, m); b1[1] = prmt(t1.x, t1.y, mh); b1[2] = prmt(t1.z, t1.w, m); b1[3] = prmt(t1.z, t1.w, mh);
                    b2[0] = prmt(t2.x, t2.y, m); b2[1] = prmt(t2.x, t2.y, mh); b2[2] = prmt(t2.z, t2.w, m); b2[3] = prmt(t2.z, t2.w, mh);
                } else {   // sign bits -> byte masks (prmt's sign-replicate mode), positive or negative table per weight
                    const uint32_t s_odd = prmt(w[ci], 0u, 0xBA98u), s_even = prmt(w[ci] << 4, 0u, 0xBA98u);
                    const uint32_t ma = prmt(s_even, s_odd, 0x5140u), mb = prmt(s_even, s_odd, 0x7362u);
                    auto pick = [&](uint32_t entry, uint32_t (&b)[4]) {
                        const uint4 th = lds128(entry), tl = lds128(entry + 16);
                        b[0] = (prmt(th.x, th.y, m) & ~ma) | (prmt(th.z, th.w, m) & ma);
                        b[1] = (prmt(th.x, th.y, mh) & ~mb) | (prmt(th.z, th.w, mh) & mb);
                        b[2] = (prmt(tl.x, tl.y, m) & ~ma) | (prmt(tl.z, tl.w, m) & ma);
                        b[3] = (prmt(tl.x, tl.y, mh) & ~mb) | (prmt(tl.z, tl.w, mh) & mb);
                    };
                    pick(ctab_a + (c12 & 255u) * 32u, b1);
                    pick(ctab_a + (c12 >> 8) * 32u, b2);
                }
                const uint32_t dst = at + off[ci];
                sts64(dst, b1[0], b1[1]);
                sts64(dst + 64 * 128, b1[2], b1[3]);
                // b2: routed, then negated where the pair sign says so
                const uint32_t sel2 = ex.x ^ 0x4444u, fa = prmt(ex.y, 0u, 0xBA98u), fb = prmt(ex.y << 1, 0u, 0xBA98u);
                uint32_t q[4] = {prmt(b2[0], b2[1], ex.x), prmt(b2[0], b2[1], sel2), prmt(b2[2], b2[3], ex.x), prmt(b2[2], b2[3], sel2)};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t f = (i & 1) ? fb : fa, x = q[i] ^ f, one = f & 0x01010101u;
                    if constexpr (WB <= 3) q[i] = x + one;   // no byte is zero: no carry
                    else q[i] = ((x & 0x7F7F7F7Fu) + one) ^ (x & 0x80808080u);
                }
                sts64(dst + 128 * 128, q[0], q[1]);
                sts64(dst + 192 * 128, q[2], q[3]);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> tensor-core reads
            __syncwarp();
            if (lane == 0) { mbar_arrive(&full[s]); mbar_arrive(&pk_empty[slot]); }
            slot += 2;
            if (slot >= p.n_pk) { slot -= p.n_pk; pk_par ^= 1u; }
            s += 2;
            if (s >= kStages) { s -= kStages; st_par ^= 1u; }
        }
    } else {
        // ------------------------------ epilogue: a thread is a token, a warp 32 tokens x 64 channels ------------------------------
        const int quarter = warp & 3, h2 = warp >> 2;
        constexpr float kInvScale = 1.0f / (float)(1u << ((1u << (WB - 1)) - 1u));
        constexpr uint32_t kB = Digits<WB>::base;
        bool ok = true;
        int tile = blockIdx.x;
        if (h2 < p.tt)
        for (int i = 0; i < my_tiles; ++i, tile += gridDim.x) {
            const int ch0 = (tile % p.tiles_x) * kChannels, tok = ((tile / p.tiles_x) * p.tt + h2) * kTokens + quarter * 32 + lane;
            float2* sc = sc_s[i % 3];
            if (p.y) {
                for (int c = lane; c < 64; c += 32) {
                    const float* src = p.sc + (size_t)(ch0 + c) * 2;   // 4-byte aligned is all that the caller promises
                    sc[c] = ch0 + c < p.n_out ? make_float2(src[0], src[1]) : make_float2(0.f, 0.f);
                }
            }
            __syncwarp();
            const float sxk = (p.sx && tok < p.m ? p.sx[tok] : 1.f) * kInvScale;
            ok = __all_sync(0xFFFFFFFFu, mbar_wait(&tm_full[h2], i & 1, &abort_flag, p.spin));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t ta = tmem_base + ((uint32_t)(quarter * 32) << 16) + h2 * 256;
            const bool f32 = p.y_dtype == GOQ_F32;
            float vmax = 0.f;
#pragma unroll 1
            for (int c0 = 0; c0 < 64; c0 += 8) {
                int h[8], l[8], a1[8], a2[8];
                __syncwarp();   // lanes without a token skip the stores: the warp reads tensor memory as one
                tmem_ld8(ta + c0, h); tmem_ld8(ta + 64 + c0, l);
                tmem_ld8(ta + 128 + c0, a1); tmem_ld8(ta + 192 + c0, a2);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    a2[j] = (int)((uint32_t)a1[j] * kB + (uint32_t)a2[j]);
                    a1[j] = (int)((uint32_t)h[j] * kB + (uint32_t)l[j]);
                }
                if (tok >= p.m || ch0 + c0 >= p.n_out) continue;
                const size_t o = (size_t)tok * p.n_out + ch0 + c0;
                const bool all8 = ch0 + c0 + 8 <= p.n_out && (p.n_out & 7) == 0;
                if (p.acc) {
                    int32_t *d1 = p.acc + o, *d2 = p.acc + (size_t)p.m * p.n_out + o;
                    if (all8 && (reinterpret_cast<uintptr_t>(p.acc) & 15u) == 0) {
#pragma unroll
                        for (int j = 0; j < 8; j += 4) {
                            *reinterpret_cast<int4*>(d1 + j) = make_int4(a1[j], a1[j + 1], a1[j + 2], a1[j + 3]);
                            *reinterpret_cast<int4*>(d2 + j) = make_int4(a2[j], a2[j + 1], a2[j + 2], a2[j + 3]);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (ch0 + c0 + j < p.n_out) { d1[j] = a1[j]; d2[j] = a2[j]; }
                    }
                }
                if (p.y) {
                    float y[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float2 s2 = sc[c0 + j];
                        y[j] = sxk * (s2.x * (float)a1[j] + s2.y * (float)a2[j]);
                        if (ch0 + c0 + j < p.n_out) vmax = fmaxf(vmax, fabsf(y[j]));
                    }
                    if (f32) {
                        float* d = reinterpret_cast<float*>(p.y) + o;
                        if (all8 && (reinterpret_cast<uintptr_t>(p.y) & 31u) == 0) {
                            st_global_v8(d, y);
                        } else {
#pragma unroll
                            for (int j = 0; j < 8; ++j) if (ch0 + c0 + j < p.n_out) d[j] = y[j];
                        }
                    } else {
                        uint16_t* d = reinterpret_cast<uint16_t*>(p.y) + o;
                        const uint32_t b[4] = {pack_bf16x2(y[0], y[1]), pack_bf16x2(y[2], y[3]), pack_bf16x2(y[4], y[5]), pack_bf16x2(y[6], y[7])};
                        if (all8 && (reinterpret_cast<uintptr_t>(p.y) & 15u) == 0) *reinterpret_cast<uint4*>(d) = make_uint4(b[0], b[1], b[2], b[3]);
                        else {
#pragma unroll
                            for (int j = 0; j < 8; ++j) if (ch0 + c0 + j < p.n_out) d[j] = (uint16_t)(b[j >> 1] >> (16 * (j & 1)));
                        }
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&tm_empty[h2]);
            // requantising epilogue (Section 3.5): the token's largest output magnitude; non-negative floats order like their bits
            if (p.amax && p.y && tok < p.m) atomicMax(reinterpret_cast<int*>(p.amax) + tok, __float_as_int(vmax));
        }
    }
    __syncthreads();
    if (abort_flag) {
        settle_after_give_up();
        if (tid == 0 && p.status) atomicExch(p.status, (int)GOQ_ERR_TIMEOUT);
        if (p.amax)   // NaN is the largest of the non-negative floats' bit patterns: it stays, and the quantizer behind passes it on
            for (int tok = tid; tok < p.m; tok += kThreads) atomicMax(reinterpret_cast<int*>(p.amax) + tok, 0x7FC00000);
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_dealloc<512>(tmem_base);
    }
}

template <int WB, int GPB>
static cudaError_t launch(const Geometry& g, Params& p, const CUtensorMap& x_map, const CUtensorMap& packed_map, cudaStream_t st) {
    constexpr int kUnitBytes = kCodeBytesPerUnit + 64 * GPB + (WB == 4 ? kWordsPerBlock : 0), kSlots = ring_slots(kUnitBytes, Digits<WB>::entry);
    static_assert(kSlots >= kDecGroups && kSlots % kDecGroups == 0, "a slot must belong to one decoding group");
    if (g.unit_bytes != kUnitBytes) return cudaErrorInvalidValue;
    p.n_pk = kSlots;
    const size_t smem = fixed_bytes(Digits<WB>::entry) + (size_t)kSlots * 4 * kUnitBytes;
    static SmemAttrCache smem_attr;
    if (cudaError_t e = ensure_dynamic_smem(gemm_i8tc_kernel<WB, GPB>, smem, smem_attr)) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.tiles < sm_count() ? p.tiles : sm_count());
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gemm_i8tc_kernel<WB, GPB>, p, x_map, packed_map);
}

}  // namespace i8tc

bool gemm_i8tc_supported(const Geometry& g, int m) { return g.group >= 32 && g.k_in % 16 == 0 && tc::packed_map_supported(g) && m >= 1; }

cudaError_t launch_gemm_i8tc(const Geometry& g, const void* packed, const int8_t* x, int m, const float* sx, const int8_t* cq, const float* sc,
                             void* y, int y_dtype, int32_t* acc, float* amax, int* status, int spin_limit, cudaStream_t st) {
    CUtensorMap xm, pm;
    if (cudaError_t e = tc::encode_i8_map(&xm, x, g.k_in, m, i8tc::kTokens)) return e;
    if (cudaError_t e = tc::encode_packed_map(&pm, packed, g, 4)) return e;
    i8tc::Params p;
    p.packed = (const uint8_t*)packed; p.cq = cq; p.sx = sx; p.sc = sc; p.y = y; p.acc = acc; p.amax = amax;
    p.unit_bytes = g.unit_bytes; p.meta_off = g.meta_off; p.k_blocks = g.k_blocks; p.groups_in = g.k_in / g.group; p.n_out = g.n_out;
    p.m = m; p.y_dtype = y_dtype;
    p.tiles_x = (g.n_pad + i8tc::kChannels - 1) / i8tc::kChannels;
    const int half_tiles = (m + i8tc::kTokens - 1) / i8tc::kTokens;
    // 256 tokens a tile halve the decode; 128 where that would leave SMs without a tile, or where there are no more (the second half's
    // MMAs would be padding: 16000 x 512 at 64 tokens 11.9 us)
    p.tt = half_tiles > 1 && p.tiles_x * ((half_tiles + 1) / 2) >= sm_count() ? 2 : 1;
    p.tiles = p.tiles_x * ((half_tiles + p.tt - 1) / p.tt);
    p.status = status;
    p.spin = spin_limit > 0 ? spin_limit : tc::kSpin;
#define GOQ_I8TC(WB_)                                                                                                       \
    (g.groups_per_block == 1 ? i8tc::launch<WB_, 1>(g, p, xm, pm, st) : g.groups_per_block == 2 ? i8tc::launch<WB_, 2>(g, p, xm, pm, st) \
                                                                                               : i8tc::launch<WB_, 4>(g, p, xm, pm, st))
    return g.wbits == 4 ? GOQ_I8TC(4) : g.wbits == 3 ? GOQ_I8TC(3) : GOQ_I8TC(2);
#undef GOQ_I8TC
}

}  // namespace goq
