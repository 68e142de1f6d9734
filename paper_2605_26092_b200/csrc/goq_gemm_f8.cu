// Float-activation layer for a few tokens up to 128 on the 5th-generation tensor cores, both bases as exact 8-bit operands; groups of 32 and more.
//
//   y[m,n] = sum_j ( c1[n,j] sum_{k in j} b1[n,k] x[m,k]  +  c2[n,j] sum_{k in j} b2[n,k] x[m,k] )      (Eq. 4 read per macro-block)
//
// The inner sums have PoT operands only, and a PoT state is an e4m3 number: one byte a weight, found by the byte permutes of the decode alone
// (b1: a table lookup per four weights; b2: the same bytes routed by the exchange record, sign bits flipped), with no coefficient in the inner
// loop. The activations are two e4m3 slices, hi + 2^-5 lo, of four significant bits each, which hold a bf16 number exactly if it is at least 2^-14 of its
// token's largest magnitude (every token is scaled by a power of two). What is smaller goes, times 2^15, into two slices of its own, as if it were another
// token; a macro-block's two sums are added as they are read back, and the coefficients multiply them in fp32. Exact down to 2^-29 of the largest, and below
// that off by at most 2^-37 of it: for a few elements of an ordinary token (0.5 to 0.9 % of the tokens that silu(gate) up makes have one) that is nothing to
// any sum. A token with more of them, or with an infinity or a NaN, is marked by the pre-pass, and its outputs are computed from the bf16 elements themselves
// by the summing kernel (goq_gemm_f8_finish.cu). (With one pair of slices an element 2^13 times the others left errors of
// 8e-4 in the channels whose code is zero there.) The fp16 form (w_hat = c1 b1 + c2 b2 rounded once, goq_gemm_mid.cu) has 19 operations on the integer pipe
// and 8 on the other per 8 weights; this has 13, and no rounding of the weights.
//
// Work split: units of 128 channels x one 128-wide k-block spread evenly over the SMs, as in goq_streamk.cuh; a token tile is 16 to 64 rows of activations, two
// rows a token ("tokens" of a tile or column below are these rows).
// Roles: four warps (eight above 32 tokens) read the group sums back (a thread is a channel) and hold y in registers until the part ends, sixteen
// decode (two groups of eight alternate k-blocks; warp = one 16-row record), one each packed records (TMA), activations (TMA) and MMA issue. The decoded
// operand goes straight to tensor memory (tcgen05.st 16x256b: its element map is the packed words' ownership), so that shared memory serves
// only the packed records, the record table and the activations. Tensor memory: four operand stages of 64 columns, and a ring of group sums
// (2 x tokens columns a basis) in the other half.
// Bound: the chain of waits between decode, MMA and read-back; no pipe is above 41 % (integer 41, 39 and 35 % at 16, 32 and 64 rows, tensor
// 11, 21 and 34 %, issue 55 to 60 %).
// Measured, W3 g128, us, goq_gemm otherwise (mid-batch kernel or decode launches) -> this: 28672 x 8192 at 24 / 32 tokens 97 / 98 -> 71 / 77; 8192 x 8192 36 / 37 -> 28 / 30.5;
// 4096 x 4096 16 / 17 -> 15.3 / 16.1; 2048 x 4096 at 64 18.4 -> 16.0; W4 28672 x 8192 at 32 tokens 98 -> 83. As goq_gemv (gemv_mma_kernel otherwise): 28672 x 8192 at 8 / 16
// tokens 66 / 83 -> 55 / 60, W4 at 1 to 8 tokens 81 -> 59. A unit takes 0.46 us with 16 rows, 0.54 with 32, 0.70 with 64. Normwise error 5.1e-8 to 1.0e-7, no larger than the
// fragment kernel's at any of 60 sizes (w_hat rounded to fp16: 2.1e-4).
// Not kept: three decoding groups (28672 x 8192 at 16 rows 55.2 -> 56.5), records copied one by one (71.5) or four k-blocks at a time (55.6).
// Every mbarrier wait is bounded; on expiry the CTA raises an abort flag, runs out its control flow, waits for what it has in flight,
// frees its tensor memory and records GOQ_ERR_TIMEOUT in the status word.
#include "goq_streamk.cuh"
#include "goq_internal.h"

namespace goq {
namespace f8 {

using namespace tc;
using namespace streamk;

// Warps by tokens of a tile / 16: reading warps, then 16 that decode, then packed records, activations, MMA issue
template <int NB8> struct Roles {
    static constexpr bool kPair = NB8 <= 2;   // both bases' sums of a macro-block are read at once (wider ones are two steps, or nothing would overlap)
    static constexpr int kDrain = kPair ? 4 : 8, kDec0 = kDrain, kPk = kDec0 + 16, kX = kPk + 1, kMma = kPk + 2, kThreads = (kPk + 3) * 32;
};
constexpr int kStages = 4, kMaxX = 8, kMaxPk = 8, kMaxSums = 8, kCoefSlots = 8;
constexpr int kMaxTokens = 64;             // rows of a tile: two a token, its larger and its smaller elements
constexpr float kSmall = 1.f / 32768.f;    // what undoes the smaller elements' factor
// Rows of activations: four tokens' larger elements, the same tokens' smaller ones, the next four's larger ones, ...
__host__ __device__ constexpr int rows_of(int m) { return (m + 3) / 4 * 8; }

struct Params {
    const uint8_t* packed;
    void* y;
    const float* inv_scale;   // [m] 2^-s of each token
    int* status;
    float* partial;           // [CTA][2][tokens][128]
    int unit_bytes, meta_off, k_blocks, n_tiles, n_out, m, rows, y_dtype;   // rows: of activations
    int tiles_x, units, n_x, n_pk;   // channel tiles; units; ring depths: activation tiles, packed units
    int run;    // units added up in one chain: about sqrt(k-blocks / macro-blocks of one), where its roundings and those of the sum over the runs are as large
    int spin;
};

// kind::f8f6f4: e4m3 x e4m3 -> fp32, both K-major, M = 128
__host__ __device__ constexpr uint32_t idesc_f8(uint32_t n) { return (1u << 4) | ((n >> 3) << 17) | ((128u >> 4) << 24); }
// the weight operand in tensor memory
__device__ __forceinline__ void umma_f8(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// 16 rows x 128 bytes: registers 4 c .. 4 c + 3 of lane (g, t) are bytes 32 c + 8 t .. + 7 of row g and of row g + 8
__device__ __forceinline__ void tmem_st_record(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile("tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
                 "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]),
                 "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {   // not waited for
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(taddr) : "memory");
}
// the loaded values pass through the wait: none is used in front of it
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&a)[8], uint32_t (&b)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]), "+r"(b[0]), "+r"(b[1]), "+r"(b[2]),
                   "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7])::"memory");
}
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&a)[8], uint32_t (&b)[8], uint32_t (&c)[8], uint32_t (&d)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]), "+r"(b[0]), "+r"(b[1]), "+r"(b[2]),
                   "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7]), "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(c[4]), "+r"(c[5]),
                   "+r"(c[6]), "+r"(c[7]), "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(d[4]), "+r"(d[5]), "+r"(d[6]), "+r"(d[7])::"memory");
}
__device__ __forceinline__ uint32_t lds32v(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
// (a0, a1) = (b0, b1) * (c0, c1) + (d0, d1)
__device__ __forceinline__ void fma2(float& a0, float& a1, float b0, float b1, float c, float d0, float d1) {
    asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %4};\n\tmov.b64 z, {%5, %6};\n\tfma.rn.f32x2 x, x, y, z;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "=f"(a0), "=f"(a1) : "f"(b0), "f"(b1), "f"(c), "f"(d0), "f"(d1));
}
// Waits for three barriers. A wait takes a trip through the shared-memory pipe even where it holds already: the three are probed at once.
// Every lane of the warp polls the same barriers and leaves with the same answer: what follows are warp-wide (.aligned) tcgen05 instructions and loop state in
// uniform registers, so a barrier per lane or one lane that polls for the others has no place here.
__device__ __forceinline__ bool wait_all(uint64_t* a, uint32_t pa, uint64_t* b, uint32_t pb, uint64_t* c, uint32_t pc, volatile int* abort_flag, int limit) {
    const bool ra = mbar_test(a, pa), rb = mbar_test(b, pb), rc = mbar_test(c, pc);
    return (ra || mbar_wait(a, pa, abort_flag, limit)) && (rb || mbar_wait(b, pb, abort_flag, limit)) && (rc || mbar_wait(c, pc, abort_flag, limit));
}
// e4m3 bytes of the PoT states, by code
template <int WB> struct PotE4m3;
template <> struct PotE4m3<3> { static constexpr uint32_t P0 = 0x00283038u, P1 = 0xA0A8B0B8u; };   // +1 +.5 +.25 0 -1 -.5 -.25 -.125
template <> struct PotE4m3<2> { static constexpr uint32_t P0 = 0xB0B80038u, P1 = 0u; };            // +1 0 -1 -.5
struct PotE4m3W4 { static constexpr uint32_t P0 = 0x20283038u, P1 = 0x00081018u, N0 = 0xA0A8B0B8u, N1 = 0x84889098u; };   // by e; +: e = 7 is the zero, -: -2^-7 is subnormal

// One micro-block word -> the bytes of b1 (r[0], r[1]) and b2 (q[0], q[1]). `record`: W4 only.
template <int WB>
__device__ __forceinline__ void expand_bytes(uint32_t w, uint32_t record, uint32_t lut_lane, uint32_t* r, uint32_t* q) {
    const uint32_t m = w & 0x77777777u, mh = m >> 16;
    uint32_t slot_off;
    if constexpr (WB <= 3) {
        r[0] = prmt(PotE4m3<WB>::P0, PotE4m3<WB>::P1, m);
        r[1] = prmt(PotE4m3<WB>::P0, PotE4m3<WB>::P1, mh);
        slot_off = (((w - m) * kHashMul) >> 19) & 0x1F80u;
    } else {   // a byte mask of the sign bits (prmt's sign-replicate mode; even weights' signs are the top bits of w << 4) chooses the table
        const uint32_t w4 = w << 4, ma = prmt(w4, w, 0xD9C8u), mb = prmt(w4, w, 0xFBEAu);
        r[0] = (prmt(PotE4m3W4::P0, PotE4m3W4::P1, m) & ~ma) | (prmt(PotE4m3W4::N0, PotE4m3W4::N1, m) & ma);
        r[1] = (prmt(PotE4m3W4::P0, PotE4m3W4::P1, mh) & ~mb) | (prmt(PotE4m3W4::N0, PotE4m3W4::N1, mh) & mb);
        slot_off = (record & 63u) << 7;
    }
    const uint4 e = lds128(slot_off | lut_lane);
    q[0] = prmt(r[0], r[1], e.x) ^ e.z;
    q[1] = prmt(r[0], r[1], e.y) ^ e.w;
}

// GPB: macro-blocks per k-block (1, 2, 4). NB8: tokens of a tile / 16 (a reading warp holds 8 NB8 of them)
template <int WB, int GPB, int NB8>
__global__ void __launch_bounds__(Roles<NB8>::kThreads, 1) gemm_f8_kernel(const Params p, const __grid_constant__ CUtensorMap x_map, const __grid_constant__ CUtensorMap packed_map) {
    using R = Roles<NB8>;
    constexpr int kThreads = R::kThreads, kDrainWarps = R::kDrain, kDec0 = R::kDec0, kPkWarp = R::kPk, kXWarp = R::kX, kMmaWarp = R::kMma;
    constexpr int kTok = 16 * NB8, kN = 2 * kTok, kXBytes = kN * 128;   // columns of a basis: hi and lo slice of every token
    constexpr int kBases = R::kPair ? 2 : 1, kSteps = 2 * GPB / kBases, kStepCols = kBases * kN, kSums = 256 / kStepCols;   // of a step: what is read back at once
    static_assert(kSums >= 2 && kSums <= kMaxSums, "sums");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* lut = smem_raw + ((8192u - (s32(smem_raw) & 8191u)) & 8191u);   // 8 KiB boundary: table offsets are OR-ed in
    unsigned char* x_tiles = lut + kLutBytes;
    uint32_t* coef = reinterpret_cast<uint32_t*>(x_tiles + p.n_x * kXBytes);   // [slot][macro-block][128]: the pairs of a unit, for the reading warps
    unsigned char* pk_ring = reinterpret_cast<unsigned char*>(coef + kCoefSlots * GPB * kTileN);
    const int pk_bytes = 8 * p.unit_bytes;
    __shared__ uint64_t a_full[kStages], a_empty[kStages], x_full[kMaxX], x_empty[kMaxX], pk_full[kMaxPk], pk_empty[kMaxPk], d_full[kMaxSums], d_empty[kMaxSums];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
    const int cta = blockIdx.x;
    const int u0 = range_begin(cta, p.units, gridDim.x), u1 = range_begin(cta + 1, p.units, gridDim.x);

    struct PkState { int u, tile, kb, slot, round; } pk = {u0, 0, -1, 0, 0};
    auto pk_issue = [&]() {   // next unit into its slot (which must be free)
        if (pk.kb < 0) { pk.tile = pk.u / p.k_blocks; pk.kb = pk.u - pk.tile * p.k_blocks; }
        mbar_expect_tx(&pk_full[pk.slot], (uint32_t)pk_bytes);   // (rows past the last tile arrive as zeros)
        tma_load_3d(pk_ring + pk.slot * pk_bytes, &packed_map, 0, pk.kb, (pk.tile % p.tiles_x) * 8, &pk_full[pk.slot]);   // (groups of 32 or more: one piece a record)
        if (++pk.kb == p.k_blocks) { pk.kb = 0; ++pk.tile; }
        ++pk.u;
        if (++pk.slot == p.n_pk) { pk.slot = 0; ++pk.round; }
    };
    if (warp == kPkWarp && lane == 0) {
        for (int i = 0; i < kMaxPk; ++i) { mbar_init(&pk_full[i], 1); mbar_init(&pk_empty[i], 8); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        while (pk.u < u1 && pk.round == 0) pk_issue();
    }
    if (tid == 0) {
        abort_flag = 0;
        for (int i = 0; i < kStages; ++i) { mbar_init(&a_full[i], 8); mbar_init(&a_empty[i], 1); }
        for (int i = 0; i < kMaxX; ++i) { mbar_init(&x_full[i], 1); mbar_init(&x_empty[i], 1); }
        for (int i = 0; i < kMaxSums; ++i) { mbar_init(&d_full[i], 1); mbar_init(&d_empty[i], kDrainWarps); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fill_lut<WB>(lut, tid, kThreads);
    if (warp == kMmaWarp) tmem_alloc<512>(&tmem_slot);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t tmem_sums = tmem_slot, tmem_a = tmem_slot + 256;

    if (warp == kPkWarp) {
        if (lane == 0) {
            bool ok = true;
            while (pk.u < u1 && ok) {
                ok = mbar_wait(&pk_empty[pk.slot], (pk.round - 1) & 1, &abort_flag, p.spin);
                if (ok) pk_issue();
            }
        }
    } else if (warp == kXWarp) {
        if (lane == 0) {
            asm volatile("griddepcontrol.wait;" ::: "memory");   // the pre-pass has written the slices
            int s = 0, round = 0, tile = u0 / p.k_blocks, kb = u0 - tile * p.k_blocks;
            for (int u = u0; u < u1; ++u) {
                if (round > 0 && !mbar_wait(&x_empty[s], (round - 1) & 1, &abort_flag, p.spin)) break;
                const int tok0 = (tile / p.tiles_x) * kTok;
                mbar_expect_tx(&x_full[s], kXBytes);   // (rows past the end arrive as zeros; tokens past the last read the other slice: columns of their own)
                tma_load_2d(x_tiles + s * kXBytes, &x_map, kb * kBlockK, tok0, &x_full[s]);
                tma_load_2d(x_tiles + s * kXBytes + kTok * 128, &x_map, kb * kBlockK, p.rows + tok0, &x_full[s]);
                if (++s == p.n_x) { s = 0; ++round; }
                if (++kb == p.k_blocks) { kb = 0; ++tile; }
            }
        }
    } else if (warp == kMmaWarp) {
        // The whole warp runs the loop and one elected lane issues.
        const uint64_t bdesc0 = smem_desc_sw128(s32(x_tiles));
        const bool leader = elect_one();
        bool ok = true;
        int xs = 0, st = 0, d = 0;
        uint32_t x_par = 0, st_par = 0, d_par = 1;   // d_par: parity of the sums' previous release (the first round passes at once)
        for (int u = u0; u < u1 && ok; ++u) {
#pragma unroll
            for (int j = 0; j < kSteps; ++j) {
                if (j == 0) ok = wait_all(&x_full[xs], x_par, &a_full[st], st_par, &d_empty[d], d_par, &abort_flag, p.spin);
                else ok = mbar_wait(&d_empty[d], d_par, &abort_flag, p.spin);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (leader) {
                    const uint64_t b = bdesc0 + (uint32_t)(xs * (kXBytes >> 4));
#pragma unroll
                    for (int i = 0; i < kBases; ++i) {
                        const int jj = j * kBases + i;   // macro-block jj / 2, basis jj % 2
                        const uint32_t a = tmem_a + (uint32_t)(st * 64 + (jj & 1) * 32), out = tmem_sums + (uint32_t)(d * kStepCols + i * kN);
#pragma unroll
                        for (int ks = 0; ks < 4 / GPB; ++ks) {
                            const int k32 = (jj >> 1) * (4 / GPB) + ks;
                            umma_f8(out, a + k32 * 8, b + 2 * k32, idesc_f8(kN), ks > 0 ? 1u : 0u);
                        }
                    }
                    umma_commit(&d_full[d]);
                    if (j == kSteps - 1) { umma_commit(&a_empty[st]); umma_commit(&x_empty[xs]); }
                }
                __syncwarp();
                if (++d == kSums) { d = 0; d_par ^= 1u; }
            }
            if (++xs == p.n_x) { xs = 0; x_par ^= 1u; }
            if (++st == kStages) { st = 0; st_par ^= 1u; }
        }
        // the last unit's releases have no reader: they must have arrived before the CTA lets go of its shared memory
        if (ok) {
            const int last_x = xs == 0 ? p.n_x - 1 : xs - 1;
            mbar_wait(&x_empty[last_x], x_par ^ (xs == 0 ? 1u : 0u), &abort_flag, p.spin);
        }
    } else if (warp >= kDec0) {
        // ------------------------------ decode: packed records -> operand bytes in tensor memory ------------------------------
        // A warp reaches the 32 tensor-memory lanes of its number mod 4: rows 32 (warp mod 4) .., of which it takes 16.
        const int dw = warp - kDec0, group = dw >> 3, e = 2 * (warp & 3) + ((dw >> 2) & 1);
        const uint32_t lut_lane = s32(lut) + (uint32_t)(lane & (kLutCopies - 1)) * 16;
        const uint32_t a_row = tmem_a + ((uint32_t)(e * 16) << 16);
        int slot = group, st = group, cs = group;
        uint32_t pk_par = 0, st_par = 1;
        bool ok = true;
        for (int u = u0 + group; u < u1; u += 2) {
            ok = __all_sync(0xFFFFFFFFu, wait_all(&pk_full[slot], pk_par, &a_empty[st], st_par, &a_empty[st], st_par, &abort_flag, p.spin));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t unit = after_wait(s32(pk_ring) + slot * pk_bytes + e * p.unit_bytes);
            const uint4 wv0 = lds128(unit + lane * 16), wv1 = lds128(unit + 512 + lane * 16);
            uint32_t mv0 = 0u, mv1 = 0u;
            if constexpr (WB == 4) { mv0 = lds32(unit + p.meta_off + lane * 4); mv1 = lds32(unit + p.meta_off + 128 + lane * 4); }
            uint32_t cf[(GPB * 16 + 31) / 32];
#pragma unroll
            for (int i = 0; i < (GPB * 16 + 31) / 32; ++i) cf[i] = lds32(unit + kCodeBytesPerUnit + ((i * 32 + lane) & (GPB * 16 - 1)) * 4);
            // the coefficient pairs of eight units ago: their sums were read before the ones behind which this stage was released
#pragma unroll
            for (int i = 0; i < (GPB * 16 + 31) / 32; ++i) {
                const int at = i * 32 + lane;
                if (at < GPB * 16) coef[(cs * GPB + (at >> 4)) * kTileN + e * 16 + (at & 15)] = cf[i];
            }
            const uint32_t w0[4] = {wv0.x, wv0.y, wv0.z, wv0.w}, w1[4] = {wv1.x, wv1.y, wv1.z, wv1.w};
            uint32_t r[16], q[16];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                expand_bytes<WB>(w0[c], mv0 >> (8 * c), lut_lane, r + 4 * c, q + 4 * c);
                expand_bytes<WB>(w1[c], mv1 >> (8 * c), lut_lane, r + 4 * c + 2, q + 4 * c + 2);
            }
            const uint32_t at = a_row + (uint32_t)(st * 64);
            tmem_st_record(at, r);
            tmem_st_record(at + 32, q);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) { mbar_arrive(&a_full[st]); mbar_arrive(&pk_empty[slot]); }
            slot += 2;
            if (slot >= p.n_pk) { slot -= p.n_pk; pk_par ^= 1u; }
            st += 2;
            if (st >= kStages) { st -= kStages; st_par ^= 1u; }
            cs = (cs + 2) & (kCoefSlots - 1);
        }
    } else {
        // ------------------------------ group sums -> y ------------------------------
        // Warp (h, quarter): channels 32 quarter + lane, rows kMine h .. of the tile: kMine / 2 tokens
        constexpr int kMine = kTok * 4 / kDrainWarps;
        const int quarter = warp & 3, h = warp >> 2, row = quarter * 32 + lane;
        const uint32_t taddr = tmem_sums + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(h * kMine), coef_a = s32(coef) + (uint32_t)row * 4;
        const Output out = {p.y, p.y_dtype, p.n_out};
        constexpr size_t kPark = (size_t)(kTok / 2) * kTileN;
        asm volatile("griddepcontrol.wait;" ::: "memory");   // outputs, parked parts and the token scales: only after earlier kernels
        bool ok = true;
        int d = 0, cs = 0, q = 0;
        uint32_t d_par = 0;
        for (int u = u0; u < u1 && ok; ++q) {
            const Part part = part_at(u, u1, p.k_blocks);
            // sums of a run of units, and of the runs before: one chain of fp32 additions over a part doubled the error (28672 x 8192: 1.8e-7, in runs 8.5e-8)
            float acc[kMine / 2], tot[kMine / 2];
#pragma unroll
            for (int i = 0; i < kMine / 2; ++i) acc[i] = tot[i] = 0.f;
            int run = 0;
            for (int k = 0; k < part.n && ok; ++k) {
#pragma unroll
                for (int j = 0; j < kSteps; ++j) {
                    ok = __all_sync(0xFFFFFFFFu, mbar_wait(&d_full[d], d_par, &abort_flag, p.spin));
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t pair = lds32v(coef_a + (uint32_t)((cs * GPB + j * kBases / 2) * kTileN * 4));
                    const float2 c = __half22float2(*reinterpret_cast<const __half2*>(&pair));
                    const uint32_t at = taddr + (uint32_t)(d * kStepCols);
                    __syncwarp();   // stores and arrivals may have diverged: the warp reads tensor memory as one
                    // 32 columns at a time: eight rows of both bases, or sixteen of one (24 rows: eight). Nothing but the wait follows a load
                    // that is on its way: its registers are not the compiler's to move or use until then.
                    constexpr int kPer = kBases == 2 || kMine % 16 != 0 ? 8 : 16, kLoads = kBases * kPer / 8;
#pragma unroll
                    for (int b = 0; b < kMine; b += kPer) {
                        uint32_t v[2 * kLoads][8];
#pragma unroll
                        for (int i = 0; i < kLoads; ++i) {
                            const uint32_t from = at + (uint32_t)(b + (kBases == 2 ? i * kN : i * 8));
                            tmem_ld8(from, v[2 * i]); tmem_ld8(from + kTok, v[2 * i + 1]);
                        }
                        if constexpr (kLoads == 2) tmem_ld_wait(v[0], v[1], v[2], v[3]);
                        else tmem_ld_wait(v[0], v[1]);
                        float both[4] = {0.f, 0.f, 0.f, 0.f};   // (both bases at once: c1 S1 + c2 S2 is one addition)
#pragma unroll
                        for (int i = 0; i < kLoads; ++i) {
                            const float cc = kBases == 2 ? (i ? c.y : c.x) : ((j & 1) ? c.y : c.x);
                            float* to = acc + (b + (kBases == 2 ? 0 : i * 8)) / 2;
                            float f[8];   // hi + 2^-5 lo of four tokens' larger elements, and of their smaller ones
#pragma unroll
                            for (int e = 0; e < 8; e += 2)
                                fma2(f[e], f[e + 1], __uint_as_float(v[2 * i + 1][e]), __uint_as_float(v[2 * i + 1][e + 1]), 0.03125f, __uint_as_float(v[2 * i][e]),
                                     __uint_as_float(v[2 * i][e + 1]));
#pragma unroll
                            for (int e = 0; e < 4; e += 2) {
                                float s0, s1;
                                fma2(s0, s1, f[4 + e], f[5 + e], kSmall, f[e], f[e + 1]);
                                if constexpr (kBases == 2) {
                                    fma2(both[e], both[e + 1], s0, s1, cc, both[e], both[e + 1]);
                                    if (i == 1) { to[e] += both[e]; to[e + 1] += both[e + 1]; }
                                } else {
                                    fma2(to[e], to[e + 1], s0, s1, cc, to[e], to[e + 1]);
                                }
                            }
                        }
                    }
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&d_empty[d]);
                    if (++d == kSums) { d = 0; d_par ^= 1u; }
                }
                cs = (cs + 1) & (kCoefSlots - 1);
                if (++run == p.run || k + 1 == part.n) {
                    run = 0;
#pragma unroll
                    for (int i = 0; i < kMine / 2; ++i) { tot[i] += acc[i]; acc[i] = 0.f; }
                }
            }
            if (!ok) break;
            const int t0 = (part.tile / p.tiles_x) * (kTok / 2), first = h * (kMine / 2), cols = min(kTok / 2, p.m - t0);
            const int ch = (part.tile % p.tiles_x) * kTileN + row;
            if (part.n < p.k_blocks) {
                float* park = p.partial + ((size_t)cta * 2 + (q == 0 ? 0 : 1)) * kPark + row;
#pragma unroll
                for (int i = 0; i < kMine / 2; ++i)
                    if (first + i < cols) __stcg(park + (size_t)(first + i) * kTileN, tot[i]);
            } else {
#pragma unroll
                for (int b = 0; b < kMine / 8; ++b) {   // (four factors at once; the array ends 16 behind the last token)
                    const int c0 = first + b * 4;
                    if (c0 >= cols) break;
                    const float4 s0 = __ldcg(reinterpret_cast<const float4*>(p.inv_scale + t0 + c0));
                    const float sc[4] = {s0.x, s0.y, s0.z, s0.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (c0 + i < cols && ch < p.n_out) out.store1(t0 + c0 + i, ch, tot[b * 4 + i] * sc[i]);
                }
            }
            u += part.n;
        }
    }
    __syncthreads();
    if (abort_flag) {
        settle_after_give_up();
        if (tid == 0) atomicExch(p.status, (int)GOQ_ERR_TIMEOUT);
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_dealloc<512>(tmem_slot);
    }
}

// ---- activation pre-pass: bf16 -> e4m3 slices, one CTA per token ------------------------------------
// v = x 2^s with the token's largest magnitude in [2^7, 2^8). Its first row holds the elements of 2^-7 and more (hi = e4m3(v), lo = e4m3((v - hi) 2^5): exact),
// its second one, four rows on, the others, times 2^15; zeros past k_in. What these do not give back is below 2^-22 and off by at most 2^-30. Where at most one
// element in 1024 of the first row's number is such a one, the error is below 2^-28 of what a channel sees of the first row (2^-30 / 2^-7 / sqrt(1024) at the
// worst, under fp32's own roundings). Else, and with an infinity or a NaN, the token is marked.
constexpr int kPrepThreads = 256;
constexpr int kPrepHold = 6;   // 16-byte vectors a thread keeps: rows up to 12288
__device__ __forceinline__ uint32_t e4m3x2(float a, float b) {   // a in the low byte
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(b), "f"(a));
    return r;
}
__device__ __forceinline__ float2 from_e4m3x2(uint32_t v) {
    uint32_t h;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h) : "h"((uint16_t)v));
    return __half22float2(*reinterpret_cast<__half2*>(&h));
}
__global__ void __launch_bounds__(kPrepThreads) x_to_f8_kernel(const uint16_t* __restrict__ x, int k_in, int k_pad, uint8_t* __restrict__ x8,
                                                               float* __restrict__ inv_scale, int* __restrict__ inexact, int m) {
    // its own dependents only when everything before it is complete: they read the packed weights at once, in stream order
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int tok = blockIdx.x, tid = threadIdx.x;
    const uint4* row = reinterpret_cast<const uint4*>(x + (size_t)tok * k_in);
    const int first_row = (tok >> 2) * 8 + (tok & 3);
    uint8_t *hi_out = x8 + (size_t)first_row * k_pad, *lo_out = x8 + (size_t)(rows_of(m) + first_row) * k_pad;
    const int n_vec = k_in / 8, n_pad = k_pad / 8;
    __shared__ uint32_t warp_max[kPrepThreads / 32];
    __shared__ int2 warp_count[kPrepThreads / 32];
    uint32_t amax = 0;
    auto largest = [&](const uint4& v) {
        const uint32_t in32[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) amax = max(amax, max(in32[j] & 0x7FFFu, (in32[j] >> 16) & 0x7FFFu));
    };
    uint4 held[kPrepHold];
#pragma unroll
    for (int h = 0; h < kPrepHold; ++h) {
        const int i = tid + h * kPrepThreads;
        held[h] = i < n_vec ? __ldg(&row[i]) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int h = 0; h < kPrepHold; ++h) largest(held[h]);
    for (int i = tid + kPrepHold * kPrepThreads; i < n_vec; i += kPrepThreads) largest(__ldg(&row[i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = max(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, o));
    if ((tid & 31) == 0) warp_max[tid >> 5] = amax;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kPrepThreads / 32; ++w) amax = max(amax, warp_max[w]);
    int sfield = 261 - (int)(amax >> 7);   // exponent field of 2^s
    sfield = sfield < 1 ? 1 : (sfield > 253 ? 253 : sfield);
    const float mult = __uint_as_float((uint32_t)sfield << 23);
    int lost = 0, large = 0;   // elements that the slices do not hold; elements of the first row
    auto convert = [&](int i, const uint4& v) {
        const uint32_t in32[4] = {v.x, v.y, v.z, v.w};
        uint32_t hi[2][2] = {{0u, 0u}, {0u, 0u}}, lo[2][2] = {{0u, 0u}, {0u, 0u}};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float a = __uint_as_float(in32[j] << 16) * mult, b = __uint_as_float(in32[j] & 0xFFFF0000u) * mult;
            const bool big_a = !(fabsf(a) < 0.0078125f), big_b = !(fabsf(b) < 0.0078125f);
            large += (int)big_a + (int)big_b;
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                const float pa = big_a == (part == 0) ? (part ? a * 32768.f : a) : 0.f, pb = big_b == (part == 0) ? (part ? b * 32768.f : b) : 0.f;
                const uint32_t h = e4m3x2(pa, pb);
                const float2 back = from_e4m3x2(h);
                const float ra = pa - back.x, rb = pb - back.y;   // exact
                const uint32_t l = e4m3x2(ra * 32.f, rb * 32.f);
                const float2 rest = from_e4m3x2(l);
                lost += (int)!(rest.x == ra * 32.f) + (int)!(rest.y == rb * 32.f);
                hi[part][j >> 1] |= h << (16 * (j & 1));
                lo[part][j >> 1] |= l << (16 * (j & 1));
            }
        }
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            *reinterpret_cast<uint2*>(hi_out + (size_t)(4 * part) * k_pad + (size_t)i * 8) = make_uint2(hi[part][0], hi[part][1]);
            *reinterpret_cast<uint2*>(lo_out + (size_t)(4 * part) * k_pad + (size_t)i * 8) = make_uint2(lo[part][0], lo[part][1]);
        }
    };
#pragma unroll
    for (int h = 0; h < kPrepHold; ++h)
        if (tid + h * kPrepThreads < n_pad) convert(tid + h * kPrepThreads, held[h]);
    for (int i = tid + kPrepHold * kPrepThreads; i < n_pad; i += kPrepThreads) convert(i, i < n_vec ? __ldg(&row[i]) : make_uint4(0u, 0u, 0u, 0u));
    lost = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)lost);
    large = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)large);
    if ((tid & 31) == 0) warp_count[tid >> 5] = make_int2(lost, large);
    __syncthreads();
    if (tid == 0) {
        int2 n = make_int2(0, 0);
        for (int w = 0; w < kPrepThreads / 32; ++w) { n.x += warp_count[w].x; n.y += warp_count[w].y; }
        inv_scale[tok] = __uint_as_float((uint32_t)(254 - sfield) << 23);
        inexact[tok] = amax >= 0x7F80u || n.x > n.y / 1024;
    }
}

// ---- host side ------------------------------------------------------------------------------------
static size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

struct Plan {
    int tokens, t_tiles, tiles_x, units, grid, n_x, n_pk;   // tokens: rows of a tile
    size_t smem, inv_off, mark_off, x8_off, partial_off, total;
};
static bool make_plan(const Geometry& g, int m, Plan* p) {
    const int rows = rows_of(m);
    p->t_tiles = (rows + kMaxTokens - 1) / kMaxTokens;
    p->tokens = ((rows + p->t_tiles - 1) / p->t_tiles + 15) & ~15;   // equal token tiles
    p->tiles_x = (g.n_pad + kTileN - 1) / kTileN;
    const long long units = (long long)p->t_tiles * p->tiles_x * g.k_blocks;
    if (units >= (1ll << 30)) return false;
    p->units = (int)units;
    p->grid = (int)(units < sm_count() ? units : sm_count());
    const size_t budget = 227 * 1024 - 2 * 1024 - 8192 - kLutBytes - (size_t)kCoefSlots * g.groups_per_block * kTileN * 4, pk = (size_t)8 * g.unit_bytes,
                 x = (size_t)2 * p->tokens * 128;
    p->n_x = p->tokens > 32 ? 4 : kMaxX;
    p->n_pk = (int)((budget - p->n_x * x) / pk) / 2 * 2;   // even: a slot comes round to the same group of decoding warps
    if (p->n_pk > kMaxPk) p->n_pk = kMaxPk;
    if (p->n_pk < 2) return false;
    p->smem = 8192 + kLutBytes + (size_t)kCoefSlots * g.groups_per_block * kTileN * 4 + p->n_x * x + p->n_pk * pk;
    p->inv_off = kWsScratchOff;
    p->mark_off = p->inv_off + align256((size_t)(m + 16) * sizeof(float));
    p->x8_off = p->mark_off + align256((size_t)m * sizeof(int));
    p->partial_off = align256(p->x8_off + (size_t)2 * rows * g.k_pad);
    p->total = p->partial_off + (size_t)p->grid * p->tokens * kTileN * sizeof(float);   // (two parts a CTA, two rows a token)
    return true;
}

template <int WB, int GPB, int NB8>
static cudaError_t launch(const Geometry& g, const Plan& pl, const void* packed, const void* x, int m, void* y, int y_dtype, uint8_t* ws, int spin_limit, cudaStream_t st) {
    CUtensorMap map, pmap;
    if (cudaError_t e = encode_packed_map(&pmap, packed, g, 8)) return e;
    if (cudaError_t e = encode_i8_map(&map, ws + pl.x8_off, g.k_pad, 2 * rows_of(m), pl.tokens)) return e;
    Params p;
    p.packed = (const uint8_t*)packed;
    p.y = y;
    p.inv_scale = (const float*)(ws + pl.inv_off);
    p.status = (int*)ws;
    p.partial = (float*)(ws + pl.partial_off);
    p.unit_bytes = g.unit_bytes; p.meta_off = g.meta_off; p.k_blocks = g.k_blocks; p.n_tiles = g.n_tiles; p.n_out = g.n_out;
    p.m = m; p.rows = rows_of(m); p.y_dtype = y_dtype; p.tiles_x = pl.tiles_x; p.units = pl.units; p.n_x = pl.n_x; p.n_pk = pl.n_pk;
    p.run = 1;
    while (p.run * (p.run + 1) * g.groups_per_block <= g.k_blocks) ++p.run;
    p.spin = spin_limit > 0 ? spin_limit : kSpin;
    static SmemAttrCache smem_attr;
    if (cudaError_t e = ensure_dynamic_smem(gemm_f8_kernel<WB, GPB, NB8>, pl.smem, smem_attr)) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pl.grid);
    cfg.blockDim = dim3(Roles<NB8>::kThreads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaError_t e = cudaLaunchKernelEx(&cfg, gemm_f8_kernel<WB, GPB, NB8>, p, map, pmap)) return e;
    return launch_f8_finish(g, packed, x, m, y, y_dtype, p.partial, p.inv_scale, (const int*)(ws + pl.mark_off), pl.tokens / 2, pl.tiles_x, pl.t_tiles, pl.units, pl.grid, st);
}
template <int WB, int GPB>
static cudaError_t launch_tokens(const Geometry& g, const Plan& pl, const void* packed, const void* x, int m, void* y, int y_dtype, uint8_t* ws, int spin_limit, cudaStream_t st) {
    switch (pl.tokens / 16) {
        case 1: return launch<WB, GPB, 1>(g, pl, packed, x, m, y, y_dtype, ws, spin_limit, st);
        case 2: return launch<WB, GPB, 2>(g, pl, packed, x, m, y, y_dtype, ws, spin_limit, st);
        case 3: return launch<WB, GPB, 3>(g, pl, packed, x, m, y, y_dtype, ws, spin_limit, st);
        default: return launch<WB, GPB, 4>(g, pl, packed, x, m, y, y_dtype, ws, spin_limit, st);
    }
}

}  // namespace f8

bool gemm_f8_supported(const Geometry& g, int m) {
    f8::Plan p;
    return g.group >= 32 && g.k_in % 8 == 0 && tc::packed_map_supported(g) && m >= 1 && f8::make_plan(g, m, &p);
}
size_t gemm_f8_workspace(const Geometry& g, int m) {
    f8::Plan p;
    return f8::make_plan(g, m, &p) ? p.total : 0;
}
// Estimated time: waves of units, a unit by its tokens and the steps its sums are read back in, and pre-pass, start and the sum of shared tiles
// (us; within 10 % of the measured times from 4096 x 4096 to 28672 x 8192, 1 to 32 tokens; up to 19 % above them where an SM has a few units, 8 % below at k = 28672).
float gemm_f8_us(const Geometry& g, int m) {
    f8::Plan p;
    if (!f8::make_plan(g, m, &p)) return 1e30f;
    const float t = (float)p.tokens, parts = (float)p.grid / (float)(p.tiles_x * p.t_tiles);
    const float unit = (g.groups_per_block == 1 ? 0.385f + 0.0049f * t : g.groups_per_block == 2 ? 0.36f + 0.0117f * t : 0.5f + 0.0207f * t) + (g.wbits == 4 ? 0.045f : 0.f);
    return 9.5f + 0.022f * t + 0.14f * parts + unit * (float)((p.units + p.grid - 1) / p.grid);
}
size_t gemm_f8_workspace_upto(const Geometry& g, int m) {   // enough for every call of up to m rows
    if (!gemm_f8_supported(g, 1)) return 0;
    const int rows = f8::rows_of(m);
    const long long units = (long long)((rows + f8::kMaxTokens - 1) / f8::kMaxTokens) * ((g.n_pad + f8::kTileN - 1) / f8::kTileN) * g.k_blocks;
    const size_t grid = units < sm_count() ? (size_t)units : (size_t)sm_count(), tokens = rows < f8::kMaxTokens ? (rows + 15) & ~15 : f8::kMaxTokens;
    return f8::align256(kWsScratchOff + f8::align256((size_t)(m + 16) * sizeof(float)) + f8::align256((size_t)m * sizeof(int)) + (size_t)2 * rows * g.k_pad) +
           grid * tokens * f8::kTileN * sizeof(float);
}
cudaError_t launch_gemm_f8(const Geometry& g, const void* packed, const void* x, int m, void* y, int y_dtype, void* ws, int spin_limit, cudaStream_t st) {
    f8::Plan p;
    if (!f8::make_plan(g, m, &p)) return cudaErrorInvalidValue;
    uint8_t* b = (uint8_t*)ws;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(m);
    cfg.blockDim = dim3(f8::kPrepThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaError_t e = cudaLaunchKernelEx(&cfg, f8::x_to_f8_kernel, (const uint16_t*)x, g.k_in, g.k_pad, b + p.x8_off, (float*)(b + p.inv_off),
                                           (int*)(b + p.mark_off), m)) return e;
#define GOQ_F8(WB_)                                                                                                       \
    (g.groups_per_block == 1 ? f8::launch_tokens<WB_, 1>(g, p, packed, x, m, y, y_dtype, b, spin_limit, st)                  \
     : g.groups_per_block == 2 ? f8::launch_tokens<WB_, 2>(g, p, packed, x, m, y, y_dtype, b, spin_limit, st)                \
                               : f8::launch_tokens<WB_, 4>(g, p, packed, x, m, y, y_dtype, b, spin_limit, st))
    return g.wbits == 4 ? GOQ_F8(4) : g.wbits == 3 ? GOQ_F8(3) : GOQ_F8(2);
#undef GOQ_F8
}

}  // namespace goq
