// Prefill GEMM (float activations, many tokens) on the 5th-generation tensor cores: the pre-pass of every such call, and the kernel for up to 256 tokens and
// for the formats that goq_gemm_pair.cu does not hold.
//
// Eq. 4 of the paper with the coefficients folded into the weight operand:
//   y[m,n] = sum_k x[m,k] * w_hat[n,k],   w_hat[n,k] = c1[n,j] b1[n,k] + c2[n,j] b2[n,k]   (Section 3.1)
// Each CTA computes a tile of 128 output channels x up to 512 tokens (two halves of at most 256). Per 64-wide k-chunk
//   - a producer thread bulk-copies the packed unit records of the 128 rows (cp.async.bulk, 8 records per
//     128 k) and loads the 512 x 64 fp16 activation tile with two 2-D TMA copies (128-byte swizzle);
//   - eight expander warps decode the records (same byte-table decode and record lookup as the GEMV:
//     b1 from the code bytes, b2 = byte-permuted b1 with pair signs, Section 3.3), form
//     w_hat = c1*b1 + c2*b2 with one half2 multiply and one half2 fma (a single rounding to fp16: the products
//     c*b are exact scalings of c) and store the 128 x 64 operand tile to shared
//     memory in the K-major, 128-byte-swizzled layout the tensor core reads;
//   - one thread issues tcgen05.mma (M=128, N=256, K=16, fp16 x fp16 -> fp32) into a 128 x 512 fp32
//     accumulator that fills the SM's tensor memory, and commits each stage back to the producers.
// After the last chunk the warps read the accumulator with tcgen05.ld and store y.
//
// Operand precision. One rounding of w_hat to bf16 (8 significant bits) costs about 2e-3 normwise on the
// output, the whole error budget; fp16 keeps 11 bits (about 2.5e-4) for the same tensor work, where a
// bf16 hi + lo pair needs twice the MMAs. Both MMA operands must then be fp16, so a pre-pass rewrites
// the bf16 activations as fp16, each token scaled by the power of two that puts its largest magnitude in
// [2^14, 2^15): bf16's 8 significant bits are kept exactly, and only elements more than 2^-28 below the
// token's largest lose bits to fp16's range (they vanish below 2^-39 of it). The epilogue undoes the scale.
// The coefficients of every output channel are first multiplied by a power of two chosen from the channel's largest
// coefficient (undone in the epilogue), so w_hat stays in fp16's normal range whatever the scale of the weights.
//
// Every mbarrier wait is bounded; on expiry the CTA raises an abort flag, skips the remaining work, waits for what it
// has in flight, frees its tensor memory and records GOQ_ERR_TIMEOUT in the status word.
#include "goq_tc_core.cuh"
#include "goq_internal.h"

namespace goq {
namespace tc {

constexpr int kTileN = 128;     // output channels per CTA (MMA M)
constexpr int kTileM = 512;     // tokens per CTA (two MMA N = 256 halves)
constexpr int kChunkK = 64;     // k per pipeline stage: 128 bytes of fp16 = one swizzle row
constexpr int kStages = 2;
constexpr int kExpanders = 8;   // expander warps; each owns one 16-row unit record per k-block
constexpr int kThreads = (2 + kExpanders) * 32;
constexpr int kATileBytes = kTileN * kChunkK * 2;   // 16 KiB, the weight operand tile of a stage
constexpr int kBTileBytes = kTileM * kChunkK * 2;   // 64 KiB

struct GemmParams {
    const uint8_t* packed;
    void* y;
    const float* inv_scale;   // [m_total] 2^-s of each token (the activations the tensor map covers are x * 2^s in fp16)
    const uint32_t* row_scale;   // [n_pad] per-channel power of two for the coefficients, fp16 in both halves
    const float* row_inv;        // [n_pad] its inverse
    int* status;
    int unit_bytes, meta_off, k_blocks, n_tiles, n_out, m_total, y_dtype, group_log2;
    // Tile schedule (1-D grid). CTAs [0, n_full) take whole tiles (2 * half tokens), numbered channel-tile fastest; the remaining
    // CTAs take the last tiles as token halves, so that a last wave that would fill less than half of
    // the SMs runs for half as long on twice as many.
    // With at most 256 tokens in all, every tile is one half (halves_per_tile = 1).
    int n_full, n_tiles_x, halves_per_tile;
    int half;   // tokens of a half tile (MMA N): a multiple of 16, at most 256
    // Split-K (only with at most 256 tokens, where the tiles alone would leave most SMs idle): n_split CTAs share a
    // tile, each takes kb_per_split k-blocks and parks its fp32 partial tile in `partial`; the CTA that arrives last
    // at the tile's counter adds the partials in split order (the result does not depend on timing), scales and
    // stores, and leaves the counter zero.
    int n_split, kb_per_split;
    float* partial;      // [tile][split][256 tokens][128 channels]
    int* tile_counter;   // [tile], zero on entry, left zero
};

template <int WB>
__global__ void __launch_bounds__(kThreads, 1)
gemm_tc_kernel(const GemmParams p, const __grid_constant__ CUtensorMap x_map) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((8192u - (s32(smem_raw) & 8191u)) & 8191u);  // 8 KiB boundary: table offsets are OR-ed in
    unsigned char* lut = base;
    unsigned char* a_tiles = lut + kLutBytes;
    unsigned char* b_tiles = a_tiles + kStages * kATileBytes;
    unsigned char* pk_ring = b_tiles + kStages * kBTileBytes;
    const int pk_slot_bytes = kExpanders * p.unit_bytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(pk_ring + 2 * pk_slot_bytes);
    uint64_t* full_b = bars;            // [kStages] activation tile landed (tx bytes)
    uint64_t* full_a = bars + 2;        // [kStages] weight tile written by the 8 expander warps
    uint64_t* empty = bars + 4;         // [kStages] tensor core finished reading the stage
    uint64_t* pk_full = bars + 6;       // [2] packed records landed
    uint64_t* pk_empty = bars + 8;      // [2] expanders finished with the records
    uint64_t* tmem_full = bars + 10;    // accumulator complete
    uint64_t* epi_bar = bars + 11;      // [2] epilogue rendezvous of the four warps of a token half
    __shared__ uint32_t tmem_base_slot;
    __shared__ __align__(16) float inv_s[kTileM];   // 2^-s of this CTA's tokens (1 for tokens past the end)
    __shared__ uint32_t row_s[kTileN];              // per-channel coefficient scale (fp16 x 2) of this CTA's 128 channels
    __shared__ float row_i[kTileN];                 // ... and its inverse
    __shared__ volatile int abort_flag;
    __shared__ volatile int split_last;   // (split-K) this CTA completed its tile's counter

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int bid = blockIdx.x;
    const int unit_id = bid / p.n_split, split = bid - unit_id * p.n_split;   // n_split > 1 only when every tile is one half
    const int tile = unit_id < p.n_full ? unit_id : p.n_full + (unit_id - p.n_full) / p.halves_per_tile;
    const int tile_x = tile % p.n_tiles_x;
    const int T0 = tile_x * (kTileN / kTileRows);  // first 16-row tile of this CTA
    const int tok0 = (tile / p.n_tiles_x) * 2 * p.half + (unit_id < p.n_full ? 0 : ((unit_id - p.n_full) % p.halves_per_tile) * p.half);
    const int n_half = unit_id < p.n_full && tok0 + p.half < p.m_total ? 2 : 1;   // token halves this CTA computes
    const int kb0 = split * p.kb_per_split;            // this CTA's k-blocks: [kb0, kb0 + nkb)
    const int nkb = tok0 < p.m_total ? min(p.kb_per_split, p.k_blocks - kb0) : 0;
    const int n_chunks = 2 * nkb;

    if (tid == 0) {
        abort_flag = 0;
        for (int i = 0; i < kStages; ++i) { mbar_init(&full_b[i], 1); mbar_init(&full_a[i], kExpanders); mbar_init(&empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&pk_full[i], 1); mbar_init(&pk_empty[i], kExpanders); }
        mbar_init(tmem_full, 1);
        mbar_init(&epi_bar[0], 4);
        mbar_init(&epi_bar[1], 4);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fill_lut<WB>(lut, tid, kThreads);
    if (warp == 1) tmem_alloc<512>(&tmem_base_slot);
    // Everything above needs nothing from the activation pre-pass, which may still be running (programmatic dependent
    // launch: this grid is scheduled as soon as the pre-pass lets it); what follows reads what the pre-pass wrote.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // (the next call's pre-pass gets in place behind this grid)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int i = tid; i < kTileM; i += kThreads) {
        const int col = i & 255, tok = tok0 + (i >> 8) * p.half + col;
        inv_s[i] = (col < p.half && tok < p.m_total) ? __ldcg(&p.inv_scale[tok]) : 1.0f;
    }
    for (int i = tid; i < kTileN; i += kThreads) {
        const bool in = T0 * kTileRows + i < p.n_tiles * kTileRows;
        row_s[i] = in ? __ldcg(&p.row_scale[T0 * kTileRows + i]) : 0x3C003C00u;   // 1.0
        row_i[i] = in ? __ldcg(&p.row_inv[T0 * kTileRows + i]) : 1.0f;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_base_slot;

    if (warp == 0) {
        // ------------------------------ producer ------------------------------
        if (lane == 0) {
            int n_rec = p.n_tiles - T0;
            if (n_rec > kExpanders) n_rec = kExpanders;
            bool ok = true;
            for (int kb = 0; kb < nkb && ok; ++kb) {
                const int ps = kb & 1;
                if (kb >= 2) ok = mbar_wait(&pk_empty[ps], ((kb >> 1) - 1) & 1, &abort_flag);
                if (!ok) break;
                mbar_expect_tx(&pk_full[ps], (uint32_t)n_rec * p.unit_bytes);
                for (int r = 0; r < n_rec; ++r)
                    bulk_g2s(pk_ring + ps * pk_slot_bytes + r * p.unit_bytes,
                             p.packed + unit_offset(T0 + r, kb0 + kb, p.k_blocks, p.unit_bytes), p.unit_bytes, &pk_full[ps]);
                for (int half = 0; half < 2 && ok; ++half) {
                    const int chunk = 2 * kb + half, s = chunk % kStages;
                    if (chunk >= kStages) ok = mbar_wait(&empty[s], ((chunk / kStages) - 1) & 1, &abort_flag);
                    if (!ok) break;
                    mbar_expect_tx(&full_b[s], (uint32_t)(n_half * p.half) * (kChunkK * 2));
                    tma_load_2d(b_tiles + s * kBTileBytes, &x_map, (2 * kb0 + chunk) * kChunkK, tok0, &full_b[s]);
                    if (n_half == 2)
                        tma_load_2d(b_tiles + s * kBTileBytes + kBTileBytes / 2, &x_map, (2 * kb0 + chunk) * kChunkK, tok0 + p.half, &full_b[s]);
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ------------------------------
        if (lane == 0) {
            bool ok = true;
            const uint32_t idesc = idesc_f16((uint32_t)p.half);
            for (int chunk = 0; chunk < n_chunks; ++chunk) {
                const int s = chunk % kStages;
                const uint32_t par = (chunk / kStages) & 1;
                ok = mbar_wait(&full_b[s], par, &abort_flag) && mbar_wait(&full_a[s], par, &abort_flag);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t adesc = smem_desc_sw128(s32(a_tiles + s * kATileBytes));
                const uint64_t bdesc0 = smem_desc_sw128(s32(b_tiles + s * kBTileBytes));
                const uint64_t bdesc1 = smem_desc_sw128(s32(b_tiles + s * kBTileBytes + kBTileBytes / 2));
#pragma unroll
                for (int ks = 0; ks < kChunkK / 16; ++ks) {
                    const uint32_t acc = (chunk > 0 || ks > 0) ? 1u : 0u;
                    umma_f16(tmem_base, adesc + 2 * ks, bdesc0 + 2 * ks, idesc, acc);         // first half's tokens
                    if (n_half == 2) umma_f16(tmem_base + 256, adesc + 2 * ks, bdesc1 + 2 * ks, idesc, acc);   // second half's
                }
                umma_commit(&empty[s]);
            }
            if (ok) umma_commit(tmem_full);
        }
    } else {
        // ------------------------------ expanders, then epilogue ------------------------------
        const int e = warp - 2, g = lane >> 2, t = lane & 3;
        const uint32_t lut_lane = s32(lut) + (uint32_t)(lane & (kLutCopies - 1)) * 16;
        const bool valid = (T0 + e) < p.n_tiles;
        const uint32_t rs_a = row_s[e * 16 + g], rs_b = row_s[e * 16 + 8 + g];   // scales of this lane's two channels
        constexpr uint32_t kZeroWord = (WB == 4) ? 0x77777777u : (WB == 3) ? 0x33333333u : 0x11111111u;  // every code = the zero state
        bool ok = true;
        for (int kb = 0; kb < nkb && ok; ++kb) {
            const int ps = kb & 1;
            ok = __all_sync(0xFFFFFFFFu, mbar_wait(&pk_full[ps], (kb >> 1) & 1, &abort_flag));
            if (!ok) break;
            const uint32_t unit = after_wait(s32(pk_ring) + ps * pk_slot_bytes + e * p.unit_bytes);
            uint4 wv0 = make_uint4(kZeroWord, kZeroWord, kZeroWord, kZeroWord), wv1 = wv0;
            uint32_t mv0 = 0u, mv1 = 0u;   // (W4) the exchange records of this lane's eight words, one byte each
            if (valid) {
                wv0 = lds128(unit + lane * 16); wv1 = lds128(unit + 512 + lane * 16);
                if constexpr (WB == 4) { mv0 = lds32(unit + p.meta_off + lane * 4); mv1 = lds32(unit + p.meta_off + 128 + lane * 4); }
            }
            const uint32_t w0[4] = {wv0.x, wv0.y, wv0.z, wv0.w}, w1[4] = {wv1.x, wv1.y, wv1.z, wv1.w};
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int chunk = 2 * kb + half, s = chunk % kStages;
                if (chunk >= kStages) ok = __all_sync(0xFFFFFFFFu, mbar_wait(&empty[s], ((chunk / kStages) - 1) & 1, &abort_flag));
                if (!ok) break;
                const uint32_t a_tile = s32(a_tiles + s * kATileBytes);
#pragma unroll
                for (int cci = 0; cci < 2; ++cci) {
                    // odd rows take the chunk's two 32-wide slices in the other order: the eight lanes of a quarter warp
                    // (two rows) then store to all eight 16-byte columns of the swizzled rows instead of four, twice
                    const int cc = cci ^ (g & 1);
                    const int c = half * 2 + cc;
                    const uint32_t wa = (g & 1) ? w0[half * 2 + (cci ^ 1)] : w0[half * 2 + cci];
                    const uint32_t wb = (g & 1) ? w1[half * 2 + (cci ^ 1)] : w1[half * 2 + cci];
                    const int jj = (c * 32 + t * 8) >> p.group_log2;  // macro-block of this micro-block inside the k-block
                    uint32_t cfa = 0u, cfb = 0u;   // {c1, c2} as stored: fp16 pairs
                    if (valid) {
                        cfa = hmul2(lds32(unit + kCodeBytesPerUnit + (jj * 16 + g) * 4), rs_a);        // exact: a power of two
                        cfb = hmul2(lds32(unit + kCodeBytesPerUnit + (jj * 16 + 8 + g) * 4), rs_b);
                    }
                    const uint32_t c1a = prmt(cfa, cfa, 0x1010u), c2a = prmt(cfa, cfa, 0x3232u);
                    const uint32_t c1b = prmt(cfb, cfb, 0x1010u), c2b = prmt(cfb, cfb, 0x3232u);
                    uint32_t oa[4], ob[4];
                    expand_what<WB>(wa, mv0 >> (8 * c), lut_lane, c1a, c2a, oa);
                    expand_what<WB>(wb, mv1 >> (8 * c), lut_lane, c1b, c2b, ob);
                    // K-major tile, 128-byte rows, 16-byte chunk j of row r stored at chunk j ^ (r & 7)
                    const int j = cc * 4 + t;
                    const int ra = e * 16 + g, rb = ra + 8;  // (ra & 7) == (rb & 7) == g
                    const uint32_t off = (uint32_t)((j ^ g) << 4);
                    sts128(a_tile + ra * 128 + off, oa[0], oa[1], oa[2], oa[3]);
                    sts128(a_tile + rb * 128 + off, ob[0], ob[1], ob[2], ob[3]);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic writes -> tensor-core reads
                __syncwarp();
                if (lane == 0) mbar_arrive(&full_a[s]);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&pk_empty[ps]);
        }
        // ---- epilogue: tensor memory -> registers -> y ----
        if (ok) ok = mbar_wait(tmem_full, 0, &abort_flag);
        ok = __all_sync(0xFFFFFFFFu, ok);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (ok && (e < 4 || n_half == 2)) {
            // Each thread holds one output channel (a TMEM lane) for 32 tokens; stored directly that is one 4-byte store
            // per token and thread, 2048 128-byte requests per CTA, and the request rate of that burst, not its bytes,
            // set the epilogue's time. So the four warps of a token half transpose 32 tokens x 128 channels through
            // shared memory (the activation ring is idle by now) and store 16 bytes per thread: a quarter of the requests.
            const int q = warp & 3, col_half = (e >= 4) ? 1 : 0;
            const int row4 = tile_x * kTileN + 4 * lane;
            const bool f32 = p.y_dtype == GOQ_F32;
            const bool vec = (tile_x + 1) * kTileN <= p.n_out && (p.n_out & 3) == 0 &&
                             (reinterpret_cast<uintptr_t>(p.y) & (f32 ? 15u : 7u)) == 0;
            auto store4 = [&](int tok, float4 f) {   // four channels of one token
                const size_t o = (size_t)tok * p.n_out + row4;
                if (f32) {
                    float* y = reinterpret_cast<float*>(p.y);
                    if (vec) *reinterpret_cast<float4*>(y + o) = f;
                    else {
                        if (row4 + 0 < p.n_out) y[o + 0] = f.x;
                        if (row4 + 1 < p.n_out) y[o + 1] = f.y;
                        if (row4 + 2 < p.n_out) y[o + 2] = f.z;
                        if (row4 + 3 < p.n_out) y[o + 3] = f.w;
                    }
                } else {
                    uint16_t* y = reinterpret_cast<uint16_t*>(p.y);
                    const uint32_t h01 = pack_bf16x2(f.x, f.y), h23 = pack_bf16x2(f.z, f.w);   // round to nearest even, in hardware
                    if (vec) *reinterpret_cast<uint2*>(y + o) = make_uint2(h01, h23);
                    else {
                        if (row4 + 0 < p.n_out) y[o + 0] = (uint16_t)(h01 & 0xFFFFu);
                        if (row4 + 1 < p.n_out) y[o + 1] = (uint16_t)(h01 >> 16);
                        if (row4 + 2 < p.n_out) y[o + 2] = (uint16_t)(h23 & 0xFFFFu);
                        if (row4 + 3 < p.n_out) y[o + 3] = (uint16_t)(h23 >> 16);
                    }
                }
            };
            const int n_cb = (p.half + 31) / 32;
#pragma unroll 1
            for (int cb = 0; cb < n_cb && ok; ++cb) {
                uint32_t v[32];
                const int col0 = col_half * 256 + cb * 32;
                __syncwarp();   // the stores before may have diverged: the warp reads tensor memory as one
                tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)col0, v);
                float* st = reinterpret_cast<float*>(b_tiles) + (col_half * 2 + (cb & 1)) * (32 * kTileN);
                const float irs = row_i[q * 32 + lane];   // this lane's channel: undo the coefficient scale (a power of two)
#pragma unroll
                for (int j4 = 0; j4 < 8; ++j4) {   // the 32 tokens' inverse scales: eight broadcast 16-byte loads
                    const float4 f = *reinterpret_cast<const float4*>(&inv_s[col0 + 4 * j4]);
                    st[(4 * j4 + 0) * kTileN + q * 32 + lane] = __uint_as_float(v[4 * j4 + 0]) * (f.x * irs);
                    st[(4 * j4 + 1) * kTileN + q * 32 + lane] = __uint_as_float(v[4 * j4 + 1]) * (f.y * irs);
                    st[(4 * j4 + 2) * kTileN + q * 32 + lane] = __uint_as_float(v[4 * j4 + 2]) * (f.z * irs);
                    st[(4 * j4 + 3) * kTileN + q * 32 + lane] = __uint_as_float(v[4 * j4 + 3]) * (f.w * irs);
                }
                // bounded rendezvous of the half's four warps (a named barrier could not give up)
                __syncwarp();
                if (lane == 0) mbar_arrive(&epi_bar[col_half]);
                ok = __all_sync(0xFFFFFFFFu, mbar_wait(&epi_bar[col_half], cb & 1, &abort_flag));
                if (!ok) break;
                if (p.n_split > 1) {   // park the (already scaled) partial rows: [token][128 channels], 512 bytes per warp store
                    float* part = p.partial + ((size_t)tile * p.n_split + split) * (256 * kTileN);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int jt = q * 8 + i;
                        __stcg(reinterpret_cast<float4*>(part + (size_t)(cb * 32 + jt) * kTileN + 4 * lane),
                               *reinterpret_cast<const float4*>(&st[jt * kTileN + 4 * lane]));
                    }
                    continue;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int jt = q * 8 + i, tok = tok0 + col_half * p.half + cb * 32 + jt;
                    if (cb * 32 + jt < p.half && tok < p.m_total) store4(tok, *reinterpret_cast<const float4*>(&st[jt * kTileN + 4 * lane]));
                }
            }
            if (p.n_split > 1 && ok) {
                // Every warp's partial rows are on their way: make them visible, meet, and let one thread count this CTA
                // in. The epilogue barrier has been through n_cb phases.
                __threadfence();
                __syncwarp();
                if (lane == 0) mbar_arrive(&epi_bar[0]);
                ok = __all_sync(0xFFFFFFFFu, mbar_wait(&epi_bar[0], n_cb & 1, &abort_flag));
                if (ok) {
                    if (lane == 0) {
                        if (q == 0) {
                            split_last = (atomicAdd(&p.tile_counter[tile], 1) == p.n_split - 1) ? 1 : 0;
                            __threadfence();
                        }
                        mbar_arrive(&epi_bar[0]);
                    }
                    ok = __all_sync(0xFFFFFFFFu, mbar_wait(&epi_bar[0], (n_cb + 1) & 1, &abort_flag));
                }
                if (ok && split_last) {
                    const float* part = p.partial + (size_t)tile * p.n_split * (256 * kTileN);
                    for (int jt = q * 64; jt < q * 64 + 64; ++jt) {
                        const int tok = tok0 + jt;
                        if (tok >= p.m_total) break;
                        float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
                        for (int sp = 0; sp < p.n_split; ++sp) {   // split order: the sum does not depend on which CTA came last
                            const float4 a = __ldcg(reinterpret_cast<const float4*>(part + ((size_t)sp * 256 + jt) * kTileN + 4 * lane));
                            f.x += a.x; f.y += a.y; f.z += a.z; f.w += a.w;
                        }
                        store4(tok, f);
                    }
                    if (q == 0 && lane == 0) p.tile_counter[tile] = 0;
                }
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    __syncthreads();
    if (abort_flag) {
        settle_after_give_up();
        if (tid == 0) atomicExch(p.status, (int)GOQ_ERR_TIMEOUT);
    }
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_dealloc<512>(tmem_base);
    }
}


// ---- activation pre-pass: bf16 -> scaled fp16, one CTA per token ------------------------------------
// xh[tok][k] = fp16(x[tok][k] * 2^s), inv_scale[tok] = 2^-s, s chosen from the exponent field of the token's largest
// magnitude (an all-zero token gets the largest scale, harmlessly). Finite elements never reach fp16's top; inf / nan stay inf / nan and
// make the token's outputs that.
constexpr int kPrepThreads = 256;
constexpr int kPrepHold = 6;   // 16-byte vectors a thread keeps: rows up to 12288
// Blocks beyond the tokens compute the per-channel scales of the weight operand, one 16-row tile each: w_hat is
// formed in fp16, whose normal range ends at 2^-14, so every channel's coefficients are multiplied by the power of two
// that puts the channel's largest |c1|, |c2| in [2^6, 2^7) (exact in fp16) and the epilogue divides it out again.
// Coefficients down to 2^-13 of their channel's largest then keep full precision even times the smallest PoT state.
__global__ void __launch_bounds__(kPrepThreads) x_to_f16_kernel(const uint16_t* __restrict__ x, int k_in, uint16_t* __restrict__ xh,
                                                                float* __restrict__ inv_scale, int m_total,
                                                                const uint8_t* __restrict__ packed, int unit_bytes, int k_blocks,
                                                                int groups_per_block, uint32_t* __restrict__ row_scale,
                                                                float* __restrict__ row_inv) {
    // Launched as a dependent itself. It lets its own dependents in only when everything before it is complete: the GEMM's CTAs may then
    // read the packed weights at once, in stream order, and set themselves up beside this pass.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if ((int)blockIdx.x >= m_total) {
        __shared__ uint32_t part_max[kPrepThreads / 16][16];
        const int T = (int)blockIdx.x - m_total, r = threadIdx.x & 15, part = threadIdx.x >> 4;
        uint32_t mx = 0;
        for (int bk = part; bk < k_blocks; bk += kPrepThreads / 16) {
            const uint32_t* cw = reinterpret_cast<const uint32_t*>(packed + ((size_t)T * k_blocks + bk) * unit_bytes + kCodeBytesPerUnit);
            for (int jj = 0; jj < groups_per_block; ++jj) {
                const uint32_t w = __ldg(&cw[jj * 16 + r]);
                mx = max(mx, max(w & 0x7FFFu, (w >> 16) & 0x7FFFu));   // fp16 magnitudes order like their bit patterns
            }
        }
        part_max[part][r] = mx;
        __syncthreads();
        if (threadIdx.x < 16) {
            for (int q = 1; q < kPrepThreads / 16; ++q) mx = max(mx, part_max[q][r]);
            int e = (int)(mx >> 10);                 // biased exponent of the largest coefficient (0: zero or subnormal)
            if (e > 30) e = 30;                      // inf / nan coefficients: leave them alone
            int shift = (mx == 0u) ? 0 : 21 - max(e, 1);   // 2^shift brings it to [2^6, 2^7)
            shift = shift < -14 ? -14 : (shift > 15 ? 15 : shift);
            const uint32_t h = (uint32_t)(15 + shift) << 10;
            row_scale[T * 16 + r] = h | (h << 16);
            row_inv[T * 16 + r] = __uint_as_float((uint32_t)(127 - shift) << 23);
        }
        return;
    }
    // one token: the row stays in registers between the maximum and the conversion (rows longer than kPrepHold vectors a
    // thread are read twice), so the pass costs one trip to memory
    const int tok = blockIdx.x, tid = threadIdx.x;
    const uint4* row = reinterpret_cast<const uint4*>(x + (size_t)tok * k_in);
    uint4* out = reinterpret_cast<uint4*>(xh + (size_t)tok * k_in);
    const int n_vec = k_in / 8;   // k_in is a multiple of 8 (checked by the launcher)
    __shared__ uint32_t warp_max[kPrepThreads / 32];
    uint32_t amax = 0;
    auto largest = [&](const uint4& v) {
        const uint32_t in32[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) amax = max(amax, max(in32[j] & 0x7FFFu, (in32[j] >> 16) & 0x7FFFu));
    };
    uint4 held[kPrepHold];
#pragma unroll
    for (int h = 0; h < kPrepHold; ++h) {
        if (h * kPrepThreads >= n_vec) break;
        const int i = tid + h * kPrepThreads;
        held[h] = i < n_vec ? __ldg(&row[i]) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int h = 0; h < kPrepHold; ++h) {
        if (h * kPrepThreads >= n_vec) break;
        largest(held[h]);
    }
    for (int i = tid + kPrepHold * kPrepThreads; i < n_vec; i += kPrepThreads) largest(__ldg(&row[i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = max(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, o));
    if ((tid & 31) == 0) warp_max[tid >> 5] = amax;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kPrepThreads / 32; ++w) amax = max(amax, warp_max[w]);
    int sfield = 268 - (int)(amax >> 7);   // exponent field of 2^s: the largest magnitude lands in [2^14, 2^15)
    sfield = sfield < 1 ? 1 : (sfield > 253 ? 253 : sfield);
    const float mult = __uint_as_float((uint32_t)sfield << 23);
    auto convert = [&](int i, const uint4& v) {
        const uint32_t in32[4] = {v.x, v.y, v.z, v.w};
        uint32_t o32[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            o32[j] = pack_f16x2(__uint_as_float(in32[j] << 16) * mult, __uint_as_float(in32[j] & 0xFFFF0000u) * mult);
        out[i] = make_uint4(o32[0], o32[1], o32[2], o32[3]);
    };
#pragma unroll
    for (int h = 0; h < kPrepHold; ++h) {
        if (h * kPrepThreads >= n_vec) break;
        if (tid + h * kPrepThreads < n_vec) convert(tid + h * kPrepThreads, held[h]);
    }
    for (int i = tid + kPrepHold * kPrepThreads; i < n_vec; i += kPrepThreads) convert(i, __ldg(&row[i]));
    if (tid == 0) inv_scale[tok] = __uint_as_float((uint32_t)(254 - sfield) << 23);
}

// ---- host side ------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)ptr;
    }
    return fn;
}

// fp16 activations [m][k_in] as boxes of 64 k x `rows` tokens, 128-byte swizzle
cudaError_t encode_x_map(CUtensorMap* map, void* xh, int k_in, int m, int rows) {
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return cudaErrorNotSupported;
    const cuuint64_t dims[2] = {(cuuint64_t)k_in, (cuuint64_t)m};
    const cuuint64_t strides[1] = {(cuuint64_t)k_in * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, xh, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidTexture;   // distinct code: the tensor map could not be encoded
}
// int8 activations [m][k_in] as boxes of 128 k x `rows` tokens, 128-byte swizzle
cudaError_t encode_i8_map(CUtensorMap* map, const void* x, int k_in, int m, int rows) {
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return cudaErrorNotSupported;
    const cuuint64_t dims[2] = {(cuuint64_t)k_in, (cuuint64_t)m};
    const cuuint64_t strides[1] = {(cuuint64_t)k_in};
    const cuuint32_t box[2] = {128, (cuuint32_t)rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(x), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidTexture;
}
// fp32 matrix [rows][cols] as boxes of `bc` columns (16: 64 bytes, 64-byte swizzle) x `br` rows
cudaError_t encode_f32_map(CUtensorMap* map, const float* w, int cols, int rows, int bc, int br) {
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return cudaErrorNotSupported;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * 4};
    const cuuint32_t box[2] = {(cuuint32_t)bc, (cuuint32_t)br};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(w), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidTexture;
}
bool packed_map_supported(const Geometry& g) {
    return (unsigned long long)g.k_blocks * g.unit_bytes / 8 < (1ull << 31);
}
cudaError_t encode_packed_map(CUtensorMap* map, const void* packed, const Geometry& g, int row_tiles) {
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return cudaErrorNotSupported;
    const int pieces = packed_pieces(g), piece = g.unit_bytes / pieces;   // bytes of a piece: a multiple of 16
    const cuuint64_t dims[3] = {(cuuint64_t)piece / 8, (cuuint64_t)g.k_blocks * pieces, (cuuint64_t)g.n_tiles};
    const cuuint64_t strides[2] = {(cuuint64_t)piece, (cuuint64_t)g.k_blocks * g.unit_bytes};
    const cuuint32_t box[3] = {(cuuint32_t)piece / 8, (cuuint32_t)pieces, (cuuint32_t)row_tiles};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3, const_cast<void*>(packed), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidTexture;
}
// The activation pre-pass (and, with `row_tiles` blocks more, the channel scales) as a programmatic dependent of what precedes it:
// its launch overlaps the tail of that kernel.
cudaError_t launch_pre_pass(const void* x, int k_in, int m, int row_tiles, uint16_t* xh, float* inv_scale, const void* packed,
                            int unit_bytes, int k_blocks, int gpb, uint32_t* row_scale, float* row_inv, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(m + row_tiles);
    cfg.blockDim = dim3(kPrepThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, x_to_f16_kernel, (const uint16_t*)x, k_in, xh, inv_scale, m, (const uint8_t*)packed, unit_bytes,
                              k_blocks, gpb, row_scale, row_inv);
}
cudaError_t launch_x_to_f16(const void* x, int k_in, int m, uint16_t* xh, float* inv_scale, cudaStream_t st) {
    return launch_pre_pass(x, k_in, m, 0, xh, inv_scale, nullptr, 0, 0, 0, nullptr, nullptr, st);
}

// Token tiles of a call, equally wide (600 tokens: 2 of 320, not 512 and 88). More of them than 512 tokens each allow where that
// makes the waves over the SMs clearly shorter (a call with few channel tiles leaves SMs idle): a CTA takes, for each k-block,
// the weights' decode plus a share that grows with its tokens (4096 x 4096 W3, us a k-block: 1.1 at 128 tokens, 1.3 at 256, 1.6 at
// 512), and about 8 us to start and to drain. 2000 x 11008 at 2048 tokens: 8 tiles 142 us, 4 tiles 176. Where every SM has work
// anyway more tiles only decode more (4096 x 4096 at 4096 tokens: 9 tiles 153 us, 8 tiles 141; the estimates differ by 2.3 %), hence
// the margin of 2.5 %.
static float wave_us(int k_blocks, int tokens) { return 8.f + (float)k_blocks * (0.95f + 0.00135f * (float)tokens); }
struct TokenTiles { int n, half, n_full, n_tail; float us; };   // tiles of 2 * half tokens; n_full CTAs take whole tiles, n_tail tiles go as halves
static TokenTiles token_tiles(const Geometry& g, int m) {
    const int sms = sm_count(), tiles_x = (g.n_pad + kTileN - 1) / kTileN;
    TokenTiles best = {};
    if (m <= 256) { best.n = 1; best.half = (m + 15) & ~15; best.n_tail = tiles_x; return best; }
    const int n0 = (m + kTileM - 1) / kTileM;
    for (int n = n0; n <= n0 + 4; ++n) {
        TokenTiles t;
        t.half = ((m + 2 * n - 1) / (2 * n) + 15) & ~15;
        t.n = (m + 2 * t.half - 1) / (2 * t.half);
        const int tiles = tiles_x * t.n, tail = tiles % sms;   // tiles of the last, partial wave
        t.n_tail = (tiles > sms && 2 * tail <= sms) ? tail : 0;
        t.n_full = tiles - t.n_tail;
        t.us = (float)((t.n_full + sms - 1) / sms) * wave_us(g.k_blocks, 2 * t.half) + (t.n_tail ? 4.f + wave_us(g.k_blocks, t.half) : 0.f);
        if (best.n == 0 || t.us < 0.975f * best.us) best = t;
    }
    return best;
}
// Split-K factor for a call (1 = none): only with at most 256 tokens, when the channel tiles alone would leave at
// least half of the SMs idle, and never below four k-blocks per CTA.
static int split_factor(const Geometry& g, int m) {
    if (m > 256) return 1;
    const int tiles_x = (g.n_pad + kTileN - 1) / kTileN;
    int s = sm_count() / tiles_x;
    if (s > 4) s = 4;
    if (s > g.k_blocks / 4) s = g.k_blocks / 4;
    if (s < 2) return 1;
    const int per = (g.k_blocks + s - 1) / s;
    return (g.k_blocks + per - 1) / per;   // no empty split
}

static size_t smem_bytes(const Geometry& g) {
    return 8192 /* alignment slack */ + kLutBytes + (size_t)kStages * (kATileBytes + kBTileBytes) +
           (size_t)2 * kExpanders * g.unit_bytes + 16 * sizeof(uint64_t);
}

// More than 256 tokens: pairs of SMs wherever their four stages fit (all but groups of 8, and W4 in groups of 16). Faster at every shape measured
// (goq_gemm_pair.cu), 2048 x 2048 at 2048 tokens 34 -> 30 us, 4096 x 4096 at 300 52 -> 44, 16000 x 512 at 512 23.1 -> 22.7.
static bool takes_pairs(const Geometry& g, int m) { return gemm_pair_supported(g, m); }

template <int WB>
static cudaError_t launch_wb(const Geometry& g, const void* packed, const void* x, int m, void* y, int y_dtype, int* status,
                             float* inv_scale, uint32_t* row_scale, float* row_inv, uint16_t* xh, int* tile_counter, float* partial,
                             int spin_limit, cudaStream_t st) {
    if (g.k_in % 8 != 0) return cudaErrorInvalidValue;
    if (cudaError_t e = launch_pre_pass(x, g.k_in, m, g.n_tiles, xh, inv_scale, packed, g.unit_bytes, g.k_blocks, g.groups_per_block,
                                        row_scale, row_inv, st)) return e;
    if (takes_pairs(g, m)) return launch_gemm_pair(g, packed, xh, inv_scale, row_scale, row_inv, m, y, y_dtype, status, spin_limit, st);
    CUtensorMap map;
    const TokenTiles tt = token_tiles(g, m);
    if (cudaError_t e = encode_x_map(&map, xh, g.k_in, m, tt.half)) return e;
    const size_t smem = smem_bytes(g);
    static SmemAttrCache smem_attr;
    if (cudaError_t e = ensure_dynamic_smem(gemm_tc_kernel<WB>, smem, smem_attr)) return e;
    GemmParams p;
    p.packed = (const uint8_t*)packed;
    p.y = y;
    p.inv_scale = inv_scale;
    p.row_scale = row_scale;
    p.row_inv = row_inv;
    p.status = status;
    p.unit_bytes = g.unit_bytes;
    p.meta_off = g.meta_off;
    p.k_blocks = g.k_blocks;
    p.n_tiles = g.n_tiles;
    p.n_out = g.n_out;
    p.m_total = m;
    p.y_dtype = y_dtype;
    int lg = 3;
    while ((1 << lg) < g.group) ++lg;
    p.group_log2 = lg;
    const int tiles_x = (g.n_pad + kTileN - 1) / kTileN, tiles = tiles_x * tt.n;
    p.n_tiles_x = tiles_x;
    p.half = tt.half;
    p.halves_per_tile = (m <= 256) ? 1 : 2;
    p.n_full = tt.n_full;
    p.n_split = split_factor(g, m);
    p.kb_per_split = (g.k_blocks + p.n_split - 1) / p.n_split;
    p.partial = partial;
    p.tile_counter = tile_counter;
    const int n_ctas = (m <= 256) ? tiles * p.n_split : p.n_full + 2 * tt.n_tail;
    // Programmatic dependent launch on the pre-pass just enqueued: the CTAs fill their tables, allocate tensor memory
    // and initialise their barriers while it runs, and wait (griddepcontrol.wait) before the first read of its outputs.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_ctas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = (m > 256) ? 1 : 0;   // measured: with at most 256 tokens (two waves of split-K CTAs) the early launch costs ~5 us
    return cudaLaunchKernelEx(&cfg, gemm_tc_kernel<WB>, p, map);
}

}  // namespace tc
}  // namespace goq

namespace goq {
bool gemm_tc_supported(const Geometry& g) { return g.wbits <= 4 && g.k_in % 8 == 0 && tc::smem_bytes(g) + 2048 <= 227 * 1024; }
// Scratch: status word and tile counters in the common areas; behind them the per-token inverse scales, the fp16
// copy of the activations and (split-K) the partial tiles.
static size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }
namespace {
struct TcScratch { size_t inv_off, rs_off, ri_off, xh_off, partial_off, total; };
TcScratch tc_scratch(const Geometry& g, int m) {
    TcScratch t;
    t.inv_off = kWsScratchOff;
    t.rs_off = t.inv_off + align256((size_t)m * sizeof(float));
    t.ri_off = t.rs_off + align256((size_t)g.n_pad * sizeof(uint32_t));
    t.xh_off = t.ri_off + align256((size_t)g.n_pad * sizeof(float));
    t.partial_off = align256(t.xh_off + (size_t)m * g.k_in * 2);
    const int split = tc::split_factor(g, m);
    const size_t tiles_x = (size_t)(g.n_pad + tc::kTileN - 1) / tc::kTileN;
    t.total = t.partial_off + (split > 1 ? tiles_x * split * 256 * tc::kTileN * sizeof(float) : 0);
    return t;
}
}  // namespace
// estimated time of a call of more than 256 tokens (pre-pass and launch 9 us)
float gemm_tc_us(const Geometry& g, int m) { return tc::takes_pairs(g, m) ? gemm_pair_us(g, m) : 9.f + tc::token_tiles(g, m).us; }
size_t gemm_tc_workspace(const Geometry& g, int m) { return tc_scratch(g, m).total; }
cudaError_t launch_gemm_tc(const Geometry& g, const void* packed, const void* x, int m, void* y, int y_dtype, void* ws,
                           int spin_limit, cudaStream_t st) {
    int* status = (int*)ws;
    const TcScratch t = tc_scratch(g, m);
    uint8_t* b = (uint8_t*)ws;
    float* inv_scale = (float*)(b + t.inv_off);
    uint32_t* rs = (uint32_t*)(b + t.rs_off);
    float* ri = (float*)(b + t.ri_off);
    uint16_t* xh = (uint16_t*)(b + t.xh_off);
    int* counters = (int*)(b + kWsStatusBytes);   // at most sm_count / 2 tiles when the split is on
    float* partial = (float*)(b + t.partial_off);
    if (g.wbits == 4) return tc::launch_wb<4>(g, packed, x, m, y, y_dtype, status, inv_scale, rs, ri, xh, counters, partial, spin_limit, st);
    return g.wbits == 3 ? tc::launch_wb<3>(g, packed, x, m, y, y_dtype, status, inv_scale, rs, ri, xh, counters, partial, spin_limit, st)
                        : tc::launch_wb<2>(g, packed, x, m, y, y_dtype, status, inv_scale, rs, ri, xh, counters, partial, spin_limit, st);
}
}  // namespace goq
