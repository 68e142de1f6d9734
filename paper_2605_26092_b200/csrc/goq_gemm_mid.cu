// Float-activation layer for a batch between decode and prefill (a few to a few hundred tokens) on the 5th-generation tensor
// cores. Few tokens make the packed weights and their decode the work and the tensor cores nearly free, so everything here
// keeps the decode running: deep rings, sixteen decoding warps, and the same number of records for every SM.
//
//   y[m,n] = sum_k x[m,k] ( c1[n,j] b1[n,k] + c2[n,j] b2[n,k] )        (Section 3.1, Eq. 4)
//
// Work split. A unit is 128 output channels x one 128-wide k-block (eight unit records). The units of a call are numbered
// token tile by token tile, channel tile by channel tile, k-block by k-block; CTA c of G takes [U c / G, U (c+1) / G): equal
// work for every SM whatever the shape (8192 x 8192: 4096 units on 148 SMs). Every CTA parks its fp32 part of a channel tile that it
// shares with others; a small second kernel adds the parts in CTA order (deterministic). A range's last part is drained by all
// warps.
//
// Roles (23 warps). Warps 0-3: coefficient scales ahead of each tile, then the epilogue (tensor memory -> y or the parked part).
// Warp 4: packed records into a ring (one TMA copy per unit). Warp 5: activation tiles (2-D TMA, 128-byte swizzle). Warp 6:
// tcgen05.mma issue. Warps 7-22: two groups of eight decode alternate k-blocks, warp e of a group record e, and write fp16
// operand tiles of 64 k. The accumulator is double-buffered in tensor memory, so a tile's epilogue overlaps the next tile.
//
// Operands. fp16 with fp32 accumulation, activations scaled per token by a power of two (pre-pass), coefficients per channel
// by a power of two (found by warps 0-3 in the coefficients of this CTA's own k-range, undone in the epilogue).
//   TWO = false: one operand w_hat = c1 b1 + c2 b2, rounded once to fp16 (2^-12 per weight), as in the prefill GEMM.
//   TWO = true:  two operands, c1 b1 and c2 b2, each exact in fp16 (a power of two times an fp16 number): no rounding before the
//                fp32 sums. For the calls whose results carry fp32 accuracy (few tokens).
//
// Every mbarrier wait is bounded; on expiry the CTA raises an abort flag, runs out its control flow, waits for what it has in flight,
// frees its tensor memory and records GOQ_ERR_TIMEOUT in the status word.
#include "goq_streamk.cuh"
#include "goq_internal.h"

namespace goq {
namespace mid {

using namespace tc;
using namespace streamk;

constexpr int kChunkBytes = kTileN * 128;   // one operand tile: 128 channels x 64 k fp16
constexpr int kEpiWarps = 4, kPkWarp = 4, kXWarp = 5, kMmaWarp = 6, kExp0 = 7, kExpWarps = 16;
constexpr int kThreads = (kExp0 + kExpWarps) * 32;
constexpr int kMaxStages = 8, kMaxPk = 8;
constexpr int kTmemCols = 512;

struct Params {
    const uint8_t* packed;
    void* y;
    const float* inv_scale;   // [m] 2^-s of each token
    int* status;
    float* partial;           // [CTA][2][n_cols][128]
    int unit_bytes, meta_off, k_blocks, n_tiles, n_out, m, y_dtype, group_log2;
    int n_cols;               // tokens per tile (MMA N): a multiple of 16, at most 256
    int tiles_x;              // channel tiles
    int units;                // token tiles x channel tiles x k-blocks
    int na;                   // accumulators of a part (1, 2, 4; TWO: 8), 256 / na tensor-memory columns apart: short sums
    int n_stages, n_pk;       // ring depths: operand stages (64 k), packed k-blocks
    int pk_pieces;            // pieces of a record in its tensor map
    int spin;                 // bound of the waits for a finished accumulator, in polls (of all of them it cost 2 %)
};

// 16 accumulator columns of this warp's 32 lanes
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}
// ... summed over the `na` accumulators of a part, `step` columns apart, in order
__device__ __forceinline__ void tmem_sum16(uint32_t taddr, int na, uint32_t step, float (&f)[16]) {
    uint32_t v[16], w[16];
    tmem_ld16(taddr, v);
    if (na > 1) tmem_ld16(taddr + step, w);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) f[j] = na > 1 ? __uint_as_float(v[j]) + __uint_as_float(w[j]) : __uint_as_float(v[j]);
    for (int a = 2; a < na; a += 2) {
        tmem_ld16(taddr + a * step, v);
        tmem_ld16(taddr + (a + 1) * step, w);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 16; ++j) f[j] += __uint_as_float(v[j]) + __uint_as_float(w[j]);
    }
}
// larger magnitude of a coefficient pair: fp16 magnitudes order like their bit patterns
__device__ __forceinline__ uint32_t coef_max(const uint8_t* pair) {
    const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(pair));
    return max(w & 0x7FFFu, (w >> 16) & 0x7FFFu);
}
// largest magnitude of a channel's pairs first, first + step, .. below n (pair i: macro-block i & (gpb - 1) of record i >> gpb_log2).
// BATCH loads in flight whatever n is (past the end the last pair again): left to the compiler, the remainder of an unrolled loop is
// one load after another, and with narrow groups and few k-blocks that was most of the kernel's time (W3, 28672 x 896 in groups of 8
// at 512 tokens 153 us).
template <int BATCH>
__device__ __forceinline__ uint32_t coef_max_of(const uint8_t* src, int first, int step, int n, int gpb_log2, int unit_bytes) {
    uint32_t mx = 0;
    for (int i0 = first; i0 < n; i0 += BATCH * step) {
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int i = min(i0 + u * step, n - 1);
            mx = max(mx, coef_max(src + (size_t)(i >> gpb_log2) * unit_bytes + (i & ((1 << gpb_log2) - 1)) * 64));
        }
    }
    return mx;
}

__device__ __forceinline__ __half2 u2h(uint32_t v) { return *reinterpret_cast<__half2*>(&v); }
__device__ __forceinline__ uint32_t h2u(__half2 v) { return *reinterpret_cast<uint32_t*>(&v); }

// GL: log2 of the group size where it is known at compile time (7: one coefficient pair per row and record), else 0
template <int WB, bool TWO, int GL>
__global__ void __launch_bounds__(kThreads, 1) gemm_mid_kernel(const Params p, const __grid_constant__ CUtensorMap x_map, const __grid_constant__ CUtensorMap packed_map) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    constexpr int kOperands = TWO ? 2 : 1, kABytes = kOperands * kChunkBytes;
    unsigned char* lut = smem_raw + ((8192u - (s32(smem_raw) & 8191u)) & 8191u);   // 8 KiB boundary: table offsets are OR-ed in
    unsigned char* a_tiles = lut + kLutBytes;
    const int b_bytes = p.n_cols * 128, pk_bytes = 8 * p.unit_bytes;
    unsigned char* b_tiles = a_tiles + p.n_stages * kABytes;
    unsigned char* pk_ring = b_tiles + p.n_stages * b_bytes;
    __shared__ uint64_t full[kMaxStages], empty[kMaxStages], pk_full[kMaxPk], pk_empty[kMaxPk], tm_full[2],
        tm_empty[2], sc_full[2];
    __shared__ uint32_t row_s[2][kTileN];   // per-channel coefficient scale (fp16 x 2) of the current and the next part
    __shared__ uint32_t row_max[kTileN];    // (start) largest |c| of the first part's channels, as fp16 bits
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
    const int G = gridDim.x, cta = blockIdx.x;
    const int u0 = range_begin(cta, p.units, G), u1 = range_begin(cta + 1, p.units, G);
    const int gpb_log2 = GL == 7 ? 0 : 7 - p.group_log2;   // macro-blocks per k-block

    // Packed records: unit by unit of the range, the eight records of a unit with one tiled copy (a copy a record, issued by one
    // thread, took ~1700 clocks a unit and was what bound this kernel). The ring is filled before anything else.
    struct PkState { int u, tile, kb, slot, round, issued; } pk = {u0, 0, -1, 0, 0, 0};
    auto pk_issue = [&]() {   // next unit into its slot (which must be free)
        if (pk.kb < 0) { pk.tile = pk.u / p.k_blocks; pk.kb = pk.u - pk.tile * p.k_blocks; }
        mbar_expect_tx(&pk_full[pk.slot], (uint32_t)pk_bytes);   // (rows past the last tile arrive as zeros)
        tma_load_3d(pk_ring + pk.slot * pk_bytes, &packed_map, 0, pk.kb * p.pk_pieces, (pk.tile % p.tiles_x) * 8, &pk_full[pk.slot]);
        if (++pk.kb == p.k_blocks) { pk.kb = 0; ++pk.tile; }
        ++pk.u; ++pk.issued;
        if (++pk.slot == p.n_pk) { pk.slot = 0; ++pk.round; }
    };
    if (warp == kPkWarp && lane == 0) {
        for (int i = 0; i < kMaxPk; ++i) { mbar_init(&pk_full[i], 1); mbar_init(&pk_empty[i], 8); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        while (pk.u < u1 && pk.round == 0) pk_issue();
    }
    if (tid < kTileN) row_max[tid] = 0u;
    if (tid == 0) {
        abort_flag = 0;
        for (int i = 0; i < kMaxStages; ++i) { mbar_init(&full[i], 8 + 1); mbar_init(&empty[i], 1); }   // eight decoding warps and the activation copy
        for (int i = 0; i < 2; ++i) { mbar_init(&tm_full[i], 1); mbar_init(&tm_empty[i], kEpiWarps); mbar_init(&sc_full[i], kEpiWarps); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fill_lut<WB>(lut, tid, kThreads);
    if (warp == kMmaWarp) tmem_alloc<kTmemCols>(&tmem_slot);
    __syncthreads();
    {   // coefficient maxima of the first part's channels, by five threads per channel (one round trip to memory)
        const Part part = part_at(u0, u1, p.k_blocks);
        const int row = tid & (kTileN - 1), sub = tid >> 7, T = (part.tile % p.tiles_x) * 8 + (row >> 4);
        if (sub < 5 && T < p.n_tiles) {
            const uint8_t* src = p.packed + unit_offset(T, part.kb, p.k_blocks, p.unit_bytes) + kCodeBytesPerUnit + (row & 15) * 4;
            atomicMax(&row_max[row], coef_max_of<8>(src, sub, 5, part.n << gpb_log2, gpb_log2, p.unit_bytes));
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t tmem_base = tmem_slot;

    const Output out = {p.y, p.y_dtype, p.n_out};
    const size_t park_floats = (size_t)p.n_cols * kTileN;   // a CTA parks at most two parts: its range's first and last tile

    // Accumulator columns first, first + step, ... (16 at a time) of a part's tile, channel quarter `quarter` (the tensor-memory
    // lanes a warp may read): to y if the part is the whole tile, else to this CTA's parked part.
    auto drain = [&](const Part& part, int q, int quarter, int first, int step, float inv_row) {
        const bool whole = part.n == p.k_blocks;
        const int tok0 = (part.tile / p.tiles_x) * p.n_cols, cols = min(p.n_cols, p.m - tok0);
        const int ch = (part.tile % p.tiles_x) * kTileN + quarter * 32 + lane;
        float* park = p.partial + ((size_t)cta * 2 + (q == 0 ? 0 : 1)) * park_floats + quarter * 32 + lane;
        const uint32_t taddr = tmem_base + (uint32_t)(q & 1) * 256u + ((uint32_t)(quarter * 32) << 16);
        for (int c0 = first; c0 < cols; c0 += step) {
            float v[16];
            __syncwarp();   // lanes without a channel skip the stores: the warp reads tensor memory as one
            tmem_sum16(taddr + c0, p.na, 256u / (uint32_t)p.na, v);
            if (!whole) {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (c0 + j < cols) __stcg(park + (size_t)(c0 + j) * kTileN, v[j] * inv_row);
            } else {
                // the tokens' factors at once: loaded one by one between the stores they made a tile's drain longer than its main
                // loop (16 of them are always there to read)
                float4 s[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) s[j] = __ldcg(reinterpret_cast<const float4*>(p.inv_scale + tok0 + c0) + j);
                const float sc[16] = {s[0].x, s[0].y, s[0].z, s[0].w, s[1].x, s[1].y, s[1].z, s[1].w,
                                      s[2].x, s[2].y, s[2].z, s[2].w, s[3].x, s[3].y, s[3].z, s[3].w};
                if (ch < p.n_out) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (c0 + j < cols) out.store1(tok0 + c0 + j, ch, v[j] * (sc[j] * inv_row));
                }
            }
        }
    };

    if (warp == kPkWarp) {
        // ------------------------------ packed records, after the first fill of the ring ------------------------------
        if (lane == 0) {
            bool ok = true;
            while (pk.u < u1 && ok) {
                ok = mbar_wait(&pk_empty[pk.slot], (pk.round - 1) & 1, &abort_flag);
                if (ok) pk_issue();
            }
        }
    } else if (warp == kXWarp) {
        // ------------------------------ activation tiles ------------------------------
        if (lane == 0) {
            asm volatile("griddepcontrol.wait;" ::: "memory");   // the pre-pass has written the fp16 activations
            bool ok = true;
            int s = 0, round = 0;
            for (int u = u0; u < u1 && ok;) {
                const Part part = part_at(u, u1, p.k_blocks);
                const int tok0 = (part.tile / p.tiles_x) * p.n_cols;
                for (int ck = 2 * part.kb; ck < 2 * (part.kb + part.n); ++ck) {
                    if (round > 0) ok = mbar_wait(&empty[s], (round - 1) & 1, &abort_flag);
                    if (!ok) break;
                    mbar_expect_tx(&full[s], (uint32_t)b_bytes);
                    tma_load_2d(b_tiles + s * b_bytes, &x_map, ck * 64, tok0, &full[s]);
                    if (++s == p.n_stages) { s = 0; ++round; }
                }
                u += part.n;
            }
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------ MMA issue ------------------------------
        // The whole warp runs the loop and one elected lane issues: descriptors stay in uniform registers. A wait that succeeds
        // still takes a trip through the (busy) shared-memory pipe, ~250 clocks, so the next stage is probed before this one's
        // MMAs are issued.
        const uint32_t idesc = idesc_f16((uint32_t)p.n_cols), acc_step = 256u / (uint32_t)p.na;
        const uint64_t adesc0 = smem_desc_sw128(s32(a_tiles)), bdesc0 = smem_desc_sw128(s32(b_tiles));
        const bool leader = elect_one();
        bool ok = true;
        int s = 0, q = 0;
        uint32_t par = 0;
        bool ready = false;
        for (int u = u0; u < u1 && ok; ++q) {
            const int n = min(p.k_blocks - u % p.k_blocks, u1 - u);
            const uint32_t d = tmem_base + (uint32_t)(q & 1) * 256u;
            if (q >= 2) ok = mbar_wait(&tm_empty[q & 1], ((q >> 1) - 1) & 1, &abort_flag);
            for (int ck = 0; ck < 2 * n && ok; ++ck) {
                if (!ready) ok = mbar_wait(&full[s], par, &abort_flag);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int s_next = s + 1 == p.n_stages ? 0 : s + 1;
                const uint32_t par_next = s_next == 0 ? par ^ 1u : par;
                ready = mbar_test(&full[s_next], par_next);
                // descriptor addresses count 16-byte units
                const uint64_t bdesc = bdesc0 + (uint32_t)(s * (b_bytes >> 4)), adesc = adesc0 + (uint32_t)(s * (kABytes >> 4));
                if (leader) {
#pragma unroll
                    for (int m = 0; m < 4 * kOperands; ++m)   // consecutive MMAs take turns on the accumulators
                        umma_f16(d + (uint32_t)(m & (p.na - 1)) * acc_step, adesc + (m >> 2) * (kChunkBytes >> 4) + 2 * (m & 3),
                                 bdesc + 2 * (m & 3), idesc, (ck > 0 || m >= p.na) ? 1u : 0u);
                    umma_commit(&empty[s]);
                    if (ck == 2 * n - 1) umma_commit(&tm_full[q & 1]);
                }
                __syncwarp();
                s = s_next; par = par_next;
            }
            u += n;
        }
    } else if (warp >= kExp0) {
        // ------------------------------ decode: packed records -> fp16 operand tiles ------------------------------
        const int ew = warp - kExp0, group = ew >> 3, e = ew & 7, g = lane >> 2, t = lane & 3;
        const uint32_t lut_lane = s32(lut) + (uint32_t)(lane & (kLutCopies - 1)) * 16;
        constexpr uint32_t kZeroWord = (WB == 4) ? 0x77777777u : (WB == 3) ? 0x33333333u : 0x11111111u;   // every code = the zero state
        const uint32_t row_off = (uint32_t)(e * 16 + g) * 128;   // row of the operand tile ((row & 7) == g, also for row + 8)
        bool ok = true;
        int i = 0, q = 0;        // unit of this CTA's range, part
        int slot = 0, st = 0;    // ring positions of unit i
        uint32_t pk_par = 0, st_par = 1;   // st_par: parity of the stage's previous release (the first round passes at once)
        for (int u = u0; u < u1 && ok; ++q) {
            const Part part = part_at(u, u1, p.k_blocks);
            const bool valid = (part.tile % p.tiles_x) * 8 + e < p.n_tiles;
            // a part with a unit of this group's: it cannot end, nor this barrier's next phase begin, before that unit is decoded
            if (part.n > 1 || (i & 1) == group) ok = __all_sync(0xFFFFFFFFu, mbar_wait(&sc_full[q & 1], (q >> 1) & 1, &abort_flag));
            const uint32_t rs_a = row_s[q & 1][e * 16 + g], rs_b = row_s[q & 1][e * 16 + 8 + g];
            __half2 cf[2] = {u2h(0u), u2h(0u)};   // {c1, c2} of rows g and g + 8, scaled (exactly: by a power of two)
            auto load_coef = [&](uint32_t unit, int jj) {
                if (valid) {
                    cf[0] = u2h(hmul2(lds32(unit + kCodeBytesPerUnit + (jj * 16 + g) * 4), rs_a));
                    cf[1] = u2h(hmul2(lds32(unit + kCodeBytesPerUnit + (jj * 16 + 8 + g) * 4), rs_b));
                }
            };
            for (int k = 0; k < part.n && ok; ++k, ++i) {
                if ((i & 1) == group) {
                    ok = __all_sync(0xFFFFFFFFu, mbar_wait(&pk_full[slot], pk_par, &abort_flag));
                    if (!ok) break;
                    const uint32_t unit = after_wait(s32(pk_ring) + slot * pk_bytes + e * p.unit_bytes);
                    uint4 wv0 = make_uint4(kZeroWord, kZeroWord, kZeroWord, kZeroWord), wv1 = wv0;
                    uint32_t mv0 = 0u, mv1 = 0u;
                    if (valid) {
                        wv0 = lds128(unit + lane * 16); wv1 = lds128(unit + 512 + lane * 16);
                        if constexpr (WB == 4) { mv0 = lds32(unit + p.meta_off + lane * 4); mv1 = lds32(unit + p.meta_off + 128 + lane * 4); }
                    }
                    if constexpr (GL == 7) load_coef(unit, 0);
                    // odd rows take the two 32-wide slices of a 64-wide chunk in the other order: the eight lanes of a store
                    // phase (two rows) then cover all eight 16-byte columns of the swizzled rows
                    const bool odd = g & 1;
                    const uint32_t w0[4] = {odd ? wv0.y : wv0.x, odd ? wv0.x : wv0.y, odd ? wv0.w : wv0.z, odd ? wv0.z : wv0.w};
                    const uint32_t w1[4] = {odd ? wv1.y : wv1.x, odd ? wv1.x : wv1.y, odd ? wv1.w : wv1.z, odd ? wv1.z : wv1.w};
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        const int s = st + half >= p.n_stages ? st + half - p.n_stages : st + half;
                        const uint32_t par = st + half >= p.n_stages ? st_par ^ 1u : st_par;
                        ok = __all_sync(0xFFFFFFFFu, mbar_wait(&empty[s], par, &abort_flag));
                        if (!ok) break;
                        const uint32_t a_tile = s32(a_tiles + s * kABytes) + row_off;
#pragma unroll
                        for (int cci = 0; cci < 2; ++cci) {
                            const int cc = cci ^ (g & 1), c = half * 2 + cc;
                            if constexpr (GL != 7) load_coef(unit, (c * 32 + t * 8) >> p.group_log2);
                            const uint32_t off = (uint32_t)(((cc * 4 + t) ^ g) << 4);
#pragma unroll
                            for (int v = 0; v < 2; ++v) {
                                const __half2 c1 = __low2half2(cf[v]), c2 = __high2half2(cf[v]);
                                uint32_t R[4], Q[4], o[4];
                                expand_bases<WB>(v ? w1[half * 2 + cci] : w0[half * 2 + cci], (v ? mv1 : mv0) >> (8 * c), lut_lane, R, Q);
                                const uint32_t dst = a_tile + v * (8 * 128) + off;
                                if constexpr (TWO) {
#pragma unroll
                                    for (int i4 = 0; i4 < 4; ++i4) o[i4] = h2u(__hmul2(c2, u2h(Q[i4])));
                                    sts128(dst + kChunkBytes, o[0], o[1], o[2], o[3]);
#pragma unroll
                                    for (int i4 = 0; i4 < 4; ++i4) o[i4] = h2u(__hmul2(c1, u2h(R[i4])));
                                } else {
#pragma unroll
                                    for (int i4 = 0; i4 < 4; ++i4) o[i4] = h2u(__hfma2(c2, u2h(Q[i4]), __hmul2(c1, u2h(R[i4]))));
                                }
                                sts128(dst, o[0], o[1], o[2], o[3]);
                            }
                        }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> tensor-core reads
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&full[s]);
                    }
                    if (!ok) break;
                    if (lane == 0) mbar_arrive(&pk_empty[slot]);   // after the __syncwarp above: every lane has read its record
                }
                if (++slot == p.n_pk) { slot = 0; pk_par ^= 1u; }
                st += 2;
                if (st >= p.n_stages) { st -= p.n_stages; st_par ^= 1u; }
            }
            u += part.n;
        }
    } else {
        // ------------------------------ warps 0..3: coefficient scales, epilogue ------------------------------
        // This lane's channel is 32 warp + lane of the tile, both where the coefficients are scanned and in tensor memory.
        auto publish = [&](uint32_t mx, int q) {   // 2^shift brings the channel's largest |c| to [2^6, 2^7); returns 2^-shift
            int ex = (int)(mx >> 10);
            if (ex > 30) ex = 30;
            int shift = mx == 0u ? 0 : 21 - max(ex, 1);
            shift = shift < -14 ? -14 : (shift > 15 ? 15 : shift);
            const uint32_t h = (uint32_t)(15 + shift) << 10;
            row_s[q & 1][warp * 32 + lane] = h | (h << 16);
            __syncwarp();
            if (lane == 0) mbar_arrive(&sc_full[q & 1]);
            return __uint_as_float((uint32_t)(127 - shift) << 23);
        };
        auto scan = [&](int u, int q) {   // the part that starts at unit u
            const Part part = part_at(u, u1, p.k_blocks);
            const int T = (part.tile % p.tiles_x) * 8 + 2 * warp + (lane >> 4);
            uint32_t mx = 0;
            if (T < p.n_tiles)
                mx = coef_max_of<16>(p.packed + unit_offset(T, part.kb, p.k_blocks, p.unit_bytes) + kCodeBytesPerUnit + (lane & 15) * 4, 0, 1,
                                     part.n << gpb_log2, gpb_log2, p.unit_bytes);
            return publish(mx, q);
        };
        float inv_row = publish(row_max[warp * 32 + lane], 0);
        asm volatile("griddepcontrol.wait;" ::: "memory");   // outputs, parked parts and the token scales: only after earlier kernels
        bool ok = true;
        int q = 0;
        for (int u = u0; u < u1 && ok; ++q) {
            const Part part = part_at(u, u1, p.k_blocks);
            const bool last_part = u + part.n >= u1;
            const float inv_next = last_part ? inv_row : scan(u + part.n, q + 1);
            if (last_part) break;   // drained by all warps, below
            ok = __all_sync(0xFFFFFFFFu, mbar_wait(&tm_full[q & 1], (q >> 1) & 1, &abort_flag, p.spin));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            drain(part, q, warp, 0, 16, inv_row);
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&tm_empty[q & 1]);
            inv_row = inv_next;
            u += part.n;
        }
    }
    // The epilogue warps come here once every earlier part is drained: from then on the barrier of the last part is in the phase that
    // is waited for (the warps that run ahead would find the phase before the last completed and take it for this one).
    __syncthreads();
    // ---- the range's last part: every warp drains its quarter's columns, in turn with the others of that quarter ----
    const int last_tile = (u1 - 1) / p.k_blocks, q_last = last_tile - u0 / p.k_blocks;
    const Part last = part_at(max(u0, last_tile * p.k_blocks), u1, p.k_blocks);
    {
        const int quarter = warp & 3, rank = warp >> 2, peers = (kThreads / 32 - quarter + 3) / 4;
        bool ok = __all_sync(0xFFFFFFFFu, mbar_wait(&tm_full[q_last & 1], (q_last >> 1) & 1, &abort_flag, p.spin));
        if (ok) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t scale = row_s[q_last & 1][quarter * 32 + lane] >> 26;   // exponent field of the fp16 power of two
            drain(last, q_last, quarter, rank * 16, peers * 16, __uint_as_float((142u - scale) << 23));
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        }
    }
    __syncthreads();
    if (abort_flag) {
        settle_after_give_up();
        if (tid == 0) atomicExch(p.status, (int)GOQ_ERR_TIMEOUT);
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_dealloc<kTmemCols>(tmem_base);
    }
}

// ---- host side ------------------------------------------------------------------------------------
static size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

struct Plan {
    int n_cols, tiles_x, t_tiles, units, grid, n_stages, n_pk;
    size_t smem, inv_off, xh_off, partial_off, total;
};
static bool make_plan(const Geometry& g, int m, bool two, Plan* p) {
    p->t_tiles = (m + 255) / 256;
    p->tiles_x = (g.n_pad + kTileN - 1) / kTileN;
    long long units = (long long)p->t_tiles * p->tiles_x * g.k_blocks;
    // One to four units an SM and wide parts: parking and summing them costs more than the decode, and half as much for a narrower
    // tile: twice the token tiles (us at 256 tokens: 2048 x 2048 21.6 -> 18.8, 1024 x 8192 28.5 -> 25.9, 1500 x 4096 24.0 -> 22.6; with
    // seven units, 4096 x 4096, 26.1 -> 26.8; with less than one, 512 x 2048, 13.6 -> 14.5; 1500 x 4096 at 64 tokens 15.8 -> 18.6).
    if (m > 128 && units >= sm_count() && units < 4 * sm_count()) { p->t_tiles *= 2; units *= 2; }
    p->n_cols = ((m + p->t_tiles - 1) / p->t_tiles + 15) & ~15;   // equal token tiles
    if (units >= (1ll << 30)) return false;
    p->units = (int)units;
    p->grid = (int)(units < sm_count() ? units : sm_count());
    // Rings: four k-blocks of packed records, then as many operand stages as fit (at least three): a fourth stage counts for more
    // than a fifth record block (8192 x 8192 at 192 tokens 46.5 -> 43.7 us). Six blocks where that is most of a CTA's range, read
    // while the pre-pass still runs, and for the exact form, whose stages are larger anyway.
    const size_t budget = 227 * 1024 - 4 * 1024 - 8192 - kLutBytes;   // static variables, alignment of the table, the table
    const size_t stage = (size_t)(two ? 2 : 1) * kChunkBytes + (size_t)p->n_cols * 128, pk = (size_t)8 * g.unit_bytes;
    p->n_pk = two || p->units <= 12 * p->grid ? 6 : 4;
    // (an even number, so that a slot comes round to the same group of decoding warps: with one phase bit a barrier, another group
    // might take the slot's records before for its own)
    while (p->n_pk > 2 && p->n_pk * pk + 3 * stage > budget) p->n_pk -= 2;
    if (p->n_pk * pk + 3 * stage > budget) return false;
    p->n_stages = (int)((budget - p->n_pk * pk) / stage);
    if (p->n_stages > kMaxStages) p->n_stages = kMaxStages;
    p->smem = 8192 + kLutBytes + p->n_stages * stage + p->n_pk * pk;
    p->inv_off = kWsScratchOff;
    p->xh_off = p->inv_off + align256((size_t)(m + 16) * sizeof(float));
    p->partial_off = align256(p->xh_off + (size_t)m * g.k_in * 2);
    p->total = p->partial_off + (size_t)p->grid * 2 * p->n_cols * kTileN * sizeof(float);
    return true;
}

template <int WB, bool TWO, int GL>
static cudaError_t launch_gl(const Geometry& g, const Plan& pl, const void* packed, int m, void* y, int y_dtype, uint8_t* ws, int spin_limit, cudaStream_t st) {
    CUtensorMap map, pmap;
    if (cudaError_t e = encode_packed_map(&pmap, packed, g, 8)) return e;
    if (cudaError_t e = encode_x_map(&map, ws + pl.xh_off, g.k_in, m, pl.n_cols)) return e;
    Params p;
    p.packed = (const uint8_t*)packed;
    p.y = y;
    p.inv_scale = (const float*)(ws + pl.inv_off);
    p.status = (int*)ws;
    p.partial = (float*)(ws + pl.partial_off);
    p.unit_bytes = g.unit_bytes; p.meta_off = g.meta_off; p.k_blocks = g.k_blocks; p.n_tiles = g.n_tiles; p.n_out = g.n_out;
    p.m = m; p.y_dtype = y_dtype;
    int lg = 3;
    while ((1 << lg) < g.group) ++lg;
    p.group_log2 = lg;
    p.n_cols = pl.n_cols;
    p.na = TWO ? 8 : (pl.n_cols <= 64 ? 4 : pl.n_cols <= 128 ? 2 : 1);
    p.tiles_x = pl.tiles_x; p.units = pl.units; p.n_stages = pl.n_stages; p.n_pk = pl.n_pk; p.pk_pieces = packed_pieces(g);
    p.spin = spin_limit > 0 ? spin_limit : kSpin;
    static SmemAttrCache smem_attr;
    if (cudaError_t e = ensure_dynamic_smem(gemm_mid_kernel<WB, TWO, GL>, pl.smem, smem_attr)) return e;
    // programmatic dependent of the pre-pass: tables, rings, coefficient scan and decode run ahead; only the activations' TMA
    // and the outputs wait for it
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pl.grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaError_t e = cudaLaunchKernelEx(&cfg, gemm_mid_kernel<WB, TWO, GL>, p, map, pmap)) return e;
    // whole tiles only: one k-block a tile, or every range a whole number of tiles
    if (g.k_blocks == 1 || (p.units % pl.grid == 0 && (p.units / pl.grid) % g.k_blocks == 0)) return cudaSuccess;
    const FinishParams f = {p.partial, p.inv_scale, y, y_dtype, g.n_out, m, pl.n_cols, pl.tiles_x, g.k_blocks, pl.units, pl.grid};
    cfg.gridDim = dim3(pl.tiles_x * pl.t_tiles, (pl.n_cols + kFinishTokens - 1) / kFinishTokens);
    cfg.blockDim = dim3(kFinishThreads);
    cfg.dynamicSmemBytes = 0;
    return cudaLaunchKernelEx(&cfg, finish_kernel, f);
}

template <int WB, bool TWO>
static cudaError_t launch(const Geometry& g, const Plan& pl, const void* packed, int m, void* y, int y_dtype, uint8_t* ws, int spin_limit, cudaStream_t st) {
    return g.group == 128 ? launch_gl<WB, TWO, 7>(g, pl, packed, m, y, y_dtype, ws, spin_limit, st)
                          : launch_gl<WB, TWO, 0>(g, pl, packed, m, y, y_dtype, ws, spin_limit, st);
}

}  // namespace mid

bool gemm_mid_supported(const Geometry& g, int m, bool exact) {
    mid::Plan p;
    return g.k_in % 8 == 0 && tc::packed_map_supported(g) && mid::make_plan(g, m, exact && !g.k1, &p);
}
// Estimated time of a call: a unit's decode plus a share that grows with its tokens, or the drain of its tile by four warps where
// the tile has few k-blocks, and 14 us for the pre-pass, the start and the shared tiles. (W3 g128, us a unit: 0.75 at 64 tokens, 1.4
// at 256; 0.15 more at W4, and more in narrow groups; 18 us for the drain of 256 tokens.)
float gemm_mid_us(const Geometry& g, int m) {
    mid::Plan p;
    if (!mid::make_plan(g, m, false, &p)) return 1e30f;
    const float unit = 0.55f + 0.0032f * (float)p.n_cols + (g.wbits == 4 ? 0.15f : 0.f) + (g.group == 128 ? 0.f : g.group >= 32 ? 0.05f : g.group == 16 ? 0.1f : 0.3f);
    const float drain = 0.07f * (float)p.n_cols / (float)g.k_blocks;
    return 14.f + (float)((p.units + p.grid - 1) / p.grid) * (unit > drain ? unit : drain);
}
int gemm_mid_ctas() { return sm_count(); }
size_t gemm_mid_workspace(const Geometry& g, int m, bool exact) {
    mid::Plan p;
    return mid::make_plan(g, m, exact && !g.k1, &p) ? p.total : 0;
}
size_t gemm_mid_workspace_upto(const Geometry& g, int m) {
    if (!(g.k_in % 8 == 0 && tc::packed_map_supported(g))) return 0;
    // the offsets of make_plan; token tiles no wider than 256 or the call, and no more CTAs than units (more token tiles than one per
    // 256 rows only where the units fill the SMs anyway)
    const long long units = (long long)((m + 255) / 256) * ((g.n_pad + mid::kTileN - 1) / mid::kTileN) * g.k_blocks;
    const size_t grid = units < sm_count() ? (size_t)units : (size_t)sm_count(), cols = m < 256 ? (m + 15) & ~15 : 256;
    const size_t xh_off = kWsScratchOff + mid::align256((size_t)(m + 16) * sizeof(float));
    return mid::align256(xh_off + (size_t)m * g.k_in * 2) + grid * 2 * cols * mid::kTileN * sizeof(float);
}
cudaError_t launch_gemm_mid(const Geometry& g, const void* packed, const void* x, int m, void* y, int y_dtype, void* ws, bool exact,
                            int spin_limit, cudaStream_t st) {
    const bool two = exact && !g.k1;   // single-basis weights: c1 b1 alone is exact already
    mid::Plan p;
    if (!mid::make_plan(g, m, two, &p)) return cudaErrorInvalidValue;
    uint8_t* b = (uint8_t*)ws;
    if (cudaError_t e = tc::launch_x_to_f16(x, g.k_in, m, (uint16_t*)(b + p.xh_off), (float*)(b + p.inv_off), st)) return e;
#define GOQ_MID(WB_) \
    (two ? mid::launch<WB_, true>(g, p, packed, m, y, y_dtype, b, spin_limit, st) : mid::launch<WB_, false>(g, p, packed, m, y, y_dtype, b, spin_limit, st))
    return g.wbits == 4 ? GOQ_MID(4) : g.wbits == 3 ? GOQ_MID(3) : GOQ_MID(2);
#undef GOQ_MID
}

}  // namespace goq
