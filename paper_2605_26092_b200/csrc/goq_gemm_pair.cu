// Prefill GEMM (float activations, many tokens) on pairs of SMs: one tcgen05.mma of cta_group::2 for 256 output channels x 256 tokens.
//
//   y[m,n] = sum_k x[m,k] * w_hat[n,k],   w_hat[n,k] = c1[n,j] b1[n,k] + c2[n,j] b2[n,k]   (Section 3.1, Eq. 4)
//
// The operands are those of goq_gemm_tc.cu: w_hat rounded once to fp16 by expander warps, activations as fp16 from its pre-pass. What a pair changes is
// the traffic of the activations: each CTA expands its own 128 channels, but of the tokens it loads only half, and an MMA reads a token's row once for both
// CTAs' channels. Per 64-wide chunk of 512 tokens a CTA takes 32 KB from L2 instead of 64 (at 64 bytes a clock and SM, half the MMAs' time instead of all
// of it) and its MMAs read 64 bytes of shared memory a clock instead of 96.
// The CTA of even rank issues the MMAs for both. "Operands are there" crosses to it as the copies' bytes (the other CTA's activation copies count on its
// barrier: cp.async.bulk.tensor with .cta_group::2) and by one arrival a chunk (a thread of the other CTA passes on that its expander warps have finished);
// "stage is free" comes back to both by one multicast commit. Four stages of 48 KB (A 16, B 32) hold more than these hops.
// Bound: MMA rate at the clock the power limit leaves, and for few tokens the round of expanders and hops (~1 us a k-block). Measured, W3 g128, us, pre-pass
// included, goq_gemm_tc.cu -> this: 4096 x 4096 at 512 / 1024 / 2048 tokens 53 / 59 / 70 -> 50 / 56 / 60; 11008 x 4096 at 1024 / 2048 116 / 188 -> 95 / 158;
// 4096 x 11008 at 2048 193 -> 154 to 164; 8192 x 8192 at 2048 274 -> 211 to 239; 28672 x 8192 at 512 258 -> 198. What it took: one thread's arrival across with a
// release restricted to shared memory (arrive_cluster; eight warps arriving across 95 us for the first at 2048), a warp that issues as one (from one lane's registers eight
// MMAs took 830 clocks: 61 at 1024 tokens, now 56), sixteen expander warps, and a warp of its own for the records.
// Every mbarrier wait is bounded; on expiry the CTA raises an abort flag (its partner's waits run out too), skips the remaining work, waits for what it has
// in flight, frees its tensor memory and records GOQ_ERR_TIMEOUT in the status word.
#include "goq_tc_core.cuh"
#include "goq_internal.h"

namespace goq {
namespace tc2 {

using namespace tc;

constexpr int kTileN = 128;     // output channels of a CTA; a pair has 256
constexpr int kChunkK = 64;     // k of a stage
constexpr int kStages = 4;      // an even number: a stage belongs to one group of expanders (a barrier has one phase bit)
constexpr int kExpanders = 8;   // warps of a group, one 16-row record each; two groups, one for either 64-wide half of a k-block
constexpr int kPkWarp = 2, kExp0 = 3, kThreads = (kExp0 + 2 * kExpanders) * 32;
constexpr int kABytes = kTileN * 128, kBBytes = 256 * 128, kStageBytes = kABytes + kBBytes;

struct Params {
    const uint8_t* packed;
    void* y;
    const float* inv_scale;      // [m] 2^-s of each token
    const uint32_t* row_scale;   // [n_pad] per-channel power of two for the coefficients, fp16 in both halves
    const float* row_inv;        // [n_pad] its inverse
    int* status;
    int unit_bytes, meta_off, k_blocks, n_tiles, n_out, m, y_dtype, group_log2;
    int pairs_x;    // pairs of channel tiles
    int n_full;     // pairs [0, n_full) take whole tiles (2 * half tokens); the rest take the last tiles as token halves
    int half;       // tokens of a half tile (MMA N): a multiple of 32, at most 256
    int spin;       // polls of a wait
};

__device__ __forceinline__ uint2 lds64(uint32_t addr) {
    uint2 v;
    asm("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// What crosses from CTA to CTA by generic writes is a weight tile: written and fenced for the tensor cores by its expanders, whose arrivals one thread of their CTA
// waits for; that thread's release of cluster scope and the issuing warp's acquire order the tile before the MMA. The fences are restricted to shared memory: a
// release that orders every kind of memory took 0.7 us a chunk (4096 x 4096 at 2048 tokens 58 -> 72 us, by two such threads in turn 62; restricted 58).
__device__ __forceinline__ void arrive_cluster(uint32_t bar) {
    asm volatile("fence.release.sync_restrict::shared::cta.cluster;\n\tmbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void acquire_cluster() { asm volatile("fence.acquire.sync_restrict::shared::cluster.cluster;" ::: "memory"); }
// mbar_test of a phase that the other CTA completes; acquire_cluster() behind it
__device__ __forceinline__ bool test_cluster(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(s32(b)), "r"(parity) : "memory");
    return ok != 0;
}
// Wait without suspending: a thread that try_wait has put to sleep is woken late when the phase is completed from the other CTA or by a commit.
template <int SLEEP, bool PEER = false>
__device__ __forceinline__ bool poll(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int limit) {
    for (int it = 0; it < limit; ++it) {
        if (PEER ? test_cluster(bar, parity) : mbar_test(bar, parity)) return true;
        if ((it & 63) == 63 && *abort_flag) return false;
        if constexpr (SLEEP > 0) __nanosleep(SLEEP);
    }
    *abort_flag = 1;
    return false;
}
// tile into this CTA's shared memory, bytes counted on a barrier of the pair (no multicast)
__device__ __forceinline__ void tma_load_pair(void* dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(s32(dst)), "l"(map), "r"(c0), "r"(c1), "r"(bar) : "memory");
}
// kind::f16 over the pair: M = 256 (128 rows of each CTA's A), N tokens (half of them in each CTA's B)
__host__ __device__ constexpr uint32_t idesc_pair(uint32_t n) { return (1u << 4) | ((n >> 3) << 17) | ((256u >> 4) << 24); }
__device__ __forceinline__ void umma_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void commit_pair(uint64_t* bar) {   // arrives at the same place in both CTAs
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(s32(bar)), "h"((uint16_t)3) : "memory");
}

template <int WB>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
gemm_pair_kernel(const Params p, const __grid_constant__ CUtensorMap x_map) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024u - (s32(smem_raw) & 1023u)) & 1023u);   // (the same offset in both CTAs)
    unsigned char* stages = base;                                                   // [stage][A 16 KB, B 32 KB]
    unsigned char* lut = stages + kStages * kStageBytes;
    unsigned char* pk_ring = lut + kLutBytes;
    const int pk_bytes = kExpanders * p.unit_bytes;
    __shared__ uint64_t full_a[kStages], peer_a[kStages], full_b[kStages], empty[kStages], pk_full[2], pk_empty[2], tmem_full, epi_bar[4];
    __shared__ uint32_t tmem_slot;
    __shared__ uint32_t row_s[kTileN];
    __shared__ float row_i[kTileN];
    __shared__ volatile int abort_flag;

    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
    const int rank = (int)cluster_rank(), unit_id = (int)blockIdx.x >> 1;
    const int tile = unit_id < p.n_full ? unit_id : p.n_full + (unit_id - p.n_full) / 2;
    const int tile_x = (tile % p.pairs_x) * 2 + rank;
    const int T0 = tile_x * (kTileN / kTileRows);   // first 16-row tile of this CTA
    const int tok0 = (tile / p.pairs_x) * 2 * p.half + (unit_id < p.n_full ? 0 : ((unit_id - p.n_full) & 1) * p.half);
    const int n_half = unit_id < p.n_full && tok0 + p.half < p.m ? 2 : 1;
    const int n_chunks = tok0 < p.m ? 2 * p.k_blocks : 0;

    if (tid == 0) {
        abort_flag = 0;
        for (int i = 0; i < kStages; ++i) { mbar_init(&full_a[i], kExpanders); mbar_init(&peer_a[i], 1); mbar_init(&full_b[i], 1); mbar_init(&empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&pk_full[i], 1); mbar_init(&pk_empty[i], 2 * kExpanders); }
        for (int i = 0; i < 4; ++i) mbar_init(&epi_bar[i], 4);
        mbar_init(&tmem_full, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fill_lut<WB>(lut, tid, kThreads);
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(s32(&tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    // What follows reads what the pre-pass wrote (programmatic dependent launch: all of the above may run beside it)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int i = tid; i < kTileN; i += kThreads) {
        const bool in = T0 * kTileRows + i < p.n_tiles * kTileRows;
        row_s[i] = in ? __ldcg(&p.row_scale[T0 * kTileRows + i]) : 0x3C003C00u;   // 1.0
        row_i[i] = in ? __ldcg(&p.row_inv[T0 * kTileRows + i]) : 1.0f;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();   // both CTAs' barriers are initialised and their tensor memory is there
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_slot;

    if (warp == 0) {
        // ------------------------------ activations: this CTA's half of the tokens ------------------------------
        if (lane == 0) {
            const int rows = p.half / 2;
            bool ok = true;
            int s = 0, round = 0;
            for (int chunk = 0; chunk < n_chunks; ++chunk) {
                if (round > 0) ok = poll<0>(&empty[s], (round - 1) & 1, &abort_flag, p.spin);
                if (!ok) break;
                unsigned char* b = stages + s * kStageBytes + kABytes;
                if (rank == 0) mbar_expect_tx(&full_b[s], (uint32_t)(n_half * p.half) * 128u);   // both CTAs' bytes
                const uint32_t bar = map_rank(s32(&full_b[s]), 0);
                tma_load_pair(b, &x_map, chunk * kChunkK, tok0 + rank * rows, bar);
                if (n_half == 2) tma_load_pair(b + kBBytes / 2, &x_map, chunk * kChunkK, tok0 + p.half + rank * rows, bar);
                if (++s == kStages) { s = 0; ++round; }
            }
        }
    } else if (warp == kPkWarp) {
        // ------------------------------ packed records of this CTA's channels, a lane a record ------------------------------
        const int n_rec = min(kExpanders, max(0, p.n_tiles - T0));
        for (int kb = 0; 2 * kb < n_chunks; ++kb) {
            const int ps = kb & 1;
            if (kb >= 2 && !__all_sync(0xFFFFFFFFu, mbar_wait(&pk_empty[ps], ((kb >> 1) - 1) & 1, &abort_flag, p.spin))) break;
            if (lane == 0) mbar_expect_tx(&pk_full[ps], (uint32_t)(n_rec * p.unit_bytes));
            __syncwarp();
            if (lane < n_rec)
                bulk_g2s(pk_ring + ps * pk_bytes + lane * p.unit_bytes, p.packed + unit_offset(T0 + lane, kb, p.k_blocks, p.unit_bytes), p.unit_bytes, &pk_full[ps]);
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issue, for both CTAs ------------------------------
        if (rank == 0) {
            // The whole warp runs the loop and one elected lane issues: descriptors stay in uniform registers (from one lane's registers the eight MMAs of a
            // chunk took 830 clocks to issue, whatever their size). A wait takes a few hundred clocks even where it holds already, and there are three a
            // chunk: the next chunk's barriers are probed before this one's MMAs are issued.
            const uint32_t idesc = idesc_pair((uint32_t)p.half);
            const uint64_t ad0 = smem_desc_sw128(s32(stages)), bd0 = smem_desc_sw128(s32(stages + kABytes));
            const bool leader = elect_one();
            bool ok = true, ready = false;
            int s = 0;
            uint32_t par = 0;
            for (int chunk = 0; chunk < n_chunks; ++chunk) {
                if (!__all_sync(0xFFFFFFFFu, ready)) {
                    ok = poll<0>(&full_b[s], par, &abort_flag, p.spin) && poll<0>(&full_a[s], par, &abort_flag, p.spin) && poll<0, true>(&peer_a[s], par, &abort_flag, p.spin);
                    ok = __all_sync(0xFFFFFFFFu, ok);
                    if (!ok) break;
                }
                acquire_cluster();
                const int next = s + 1 == kStages ? 0 : s + 1;
                const uint32_t par_next = next == 0 ? par ^ 1u : par;
                {
                    const bool rb = mbar_test(&full_b[next], par_next), ra = mbar_test(&full_a[next], par_next), rp = test_cluster(&peer_a[next], par_next);
                    ready = rb && ra && rp;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (leader) {
                    const uint64_t ad = ad0 + (uint32_t)(s * (kStageBytes >> 4)), bd = bd0 + (uint32_t)(s * (kStageBytes >> 4));
#pragma unroll
                    for (int ks = 0; ks < kChunkK / 16; ++ks) {
                        const uint32_t acc = (chunk > 0 || ks > 0) ? 1u : 0u;
                        umma_pair(tmem_base, ad + 2 * ks, bd + 2 * ks, idesc, acc);
                        if (n_half == 2) umma_pair(tmem_base + 256, ad + 2 * ks, bd + (kBBytes / 2 >> 4) + 2 * ks, idesc, acc);
                    }
                    commit_pair(&empty[s]);
                }
                __syncwarp();
                s = next; par = par_next;
            }
            if (ok && leader && n_chunks > 0) commit_pair(&tmem_full);
        } else if (lane == 0) {
            // the other CTA's weight tiles: passed on by one thread (an arrival that the whole pair sees costs an expander warp as much as its tile)
            int s = 0;
            uint32_t par = 0;
            for (int chunk = 0; chunk < n_chunks; ++chunk) {
                if (!poll<0>(&full_a[s], par, &abort_flag, p.spin)) break;
                arrive_cluster(map_rank(s32(&peer_a[s]), 0));
                if (++s == kStages) { s = 0; par ^= 1u; }
            }
        }
    } else {
        // ------------------------------ expanders, then epilogue ------------------------------
        const int group = (warp - kExp0) >> 3, e = (warp - kExp0) & 7, g = lane >> 2, t = lane & 3;
        const uint32_t lut_lane = s32(lut) + (uint32_t)(lane & (kLutCopies - 1)) * 16;
        const bool valid = T0 + e < p.n_tiles;
        const uint32_t rs_a = row_s[e * 16 + g], rs_b = row_s[e * 16 + 8 + g];   // scales of this lane's two channels
        constexpr uint32_t kZeroWord = (WB == 4) ? 0x77777777u : (WB == 3) ? 0x33333333u : 0x11111111u;   // every code = the zero state
        bool ok = true;
        int s = group;
        uint32_t par = 1;   // parity of the stage's previous release (the first round passes at once)
        for (int kb = 0; 2 * kb < n_chunks && ok; ++kb) {
            const int ps = kb & 1;
            ok = __all_sync(0xFFFFFFFFu, mbar_wait(&pk_full[ps], (kb >> 1) & 1, &abort_flag, p.spin));
            if (!ok) break;
            const uint32_t unit = after_wait(s32(pk_ring) + ps * pk_bytes + e * p.unit_bytes);
            uint2 wv0 = make_uint2(kZeroWord, kZeroWord), wv1 = wv0;   // its two words of rows g and g + 8
            uint32_t mv0 = 0u, mv1 = 0u;                               // (W4) the exchange records of its eight words, one byte each
            uint32_t cf[2][2] = {{0u, 0u}, {0u, 0u}};                  // {c1, c2} of the rows, for either word
            if (valid) {
                wv0 = lds64(unit + lane * 16 + group * 8); wv1 = lds64(unit + 512 + lane * 16 + group * 8);
                if constexpr (WB == 4) { mv0 = lds32(unit + p.meta_off + lane * 4); mv1 = lds32(unit + p.meta_off + 128 + lane * 4); }
#pragma unroll
                for (int cc = 0; cc < 2; ++cc) {
                    const uint32_t at = unit + kCodeBytesPerUnit + (((((group * 2 + cc) * 32 + t * 8) >> p.group_log2) * 16 + g) * 4);
                    cf[cc][0] = lds32(at); cf[cc][1] = lds32(at + 32);
                }
            }
            ok = __all_sync(0xFFFFFFFFu, poll<20>(&empty[s], par, &abort_flag, p.spin));
            if (!ok) break;
            const uint32_t a_tile = s32(stages + s * kStageBytes);
#pragma unroll
            for (int cci = 0; cci < 2; ++cci) {
                // odd rows take the chunk's two 32-wide slices in the other order: the eight lanes of a quarter warp
                // (two rows) then store to all eight 16-byte columns of the swizzled rows
                const int cc = cci ^ (g & 1), c = group * 2 + cc;
                const uint32_t wa = cc ? wv0.y : wv0.x, wb = cc ? wv1.y : wv1.x;
                const uint32_t cfa = hmul2(cc ? cf[1][0] : cf[0][0], rs_a), cfb = hmul2(cc ? cf[1][1] : cf[0][1], rs_b);   // exact: a power of two
                uint32_t oa[4], ob[4];
                expand_what<WB, true>(wa, mv0 >> (8 * c), lut_lane, prmt(cfa, cfa, 0x1010u), prmt(cfa, cfa, 0x3232u), oa);
                expand_what<WB, true>(wb, mv1 >> (8 * c), lut_lane, prmt(cfb, cfb, 0x1010u), prmt(cfb, cfb, 0x3232u), ob);
                const int ra = e * 16 + g;   // (ra & 7) == g, also for row + 8
                const uint32_t off = (uint32_t)(((cc * 4 + t) ^ g) << 4);
                sts128(a_tile + ra * 128 + off, oa[0], oa[1], oa[2], oa[3]);
                sts128(a_tile + (ra + 8) * 128 + off, ob[0], ob[1], ob[2], ob[3]);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> tensor-core reads
            __syncwarp();
            // (the record's slot only now: released right behind its loads, it was overwritten while they were on their way, and sums were wrong)
            if (lane == 0) { mbar_arrive(&full_a[s]); mbar_arrive(&pk_empty[ps]); }
            s += 2;
            if (s >= kStages) { s -= kStages; par ^= 1u; }
        }
        // ---- epilogue: tensor memory -> registers -> shared memory (transposed) -> y ----
        if (n_chunks == 0) ok = false;
        if (ok) ok = mbar_wait(&tmem_full, 0, &abort_flag, p.spin);
        ok = __all_sync(0xFFFFFFFFu, ok);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int set = (warp - kExp0) >> 2, col_half = set & 1;   // four warps: every second 32 tokens of a half
        if (ok && (col_half == 0 || n_half == 2)) {
            // The four warps of a token half transpose 32 tokens x 128 channels through the idle ring and store 16 bytes a thread: a quarter of the
            // requests that a store per token and channel would make.
            const int q = warp & 3;
            const int row4 = tile_x * kTileN + 4 * lane;
            const bool f32 = p.y_dtype == GOQ_F32;
            const bool vec = (tile_x + 1) * kTileN <= p.n_out && (p.n_out & 3) == 0 && (reinterpret_cast<uintptr_t>(p.y) & (f32 ? 15u : 7u)) == 0;
            const float irs = row_i[q * 32 + lane];   // this lane's channel: undo the coefficient scale (a power of two)
            const int n_cb = (p.half + 31) / 32;
#pragma unroll 1
            for (int cb = set >> 1, it = 0; cb < n_cb; cb += 2, ++it) {
                const int first = tok0 + col_half * p.half + cb * 32;   // 32 tokens
                const float inv = __ldcg(&p.inv_scale[min(first + lane, p.m - 1)]);
                uint32_t v[32];
                __syncwarp();   // the stores before may have diverged: the warp reads tensor memory as one
                tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(col_half * 256 + cb * 32), v);
                float* st = reinterpret_cast<float*>(stages) + (set * 2 + (it & 1)) * (32 * kTileN);
#pragma unroll
                for (int j = 0; j < 32; ++j) st[j * kTileN + q * 32 + lane] = __uint_as_float(v[j]) * (__shfl_sync(0xFFFFFFFFu, inv, j) * irs);
                // bounded rendezvous of the half's four warps (a named barrier could not give up)
                __syncwarp();
                if (lane == 0) mbar_arrive(&epi_bar[set]);
                ok = __all_sync(0xFFFFFFFFu, mbar_wait(&epi_bar[set], it & 1, &abort_flag, p.spin));
                if (!ok) break;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int jt = q * 8 + i, tok = first + jt;
                    if (cb * 32 + jt >= p.half || tok >= p.m) continue;
                    const float4 f = *reinterpret_cast<const float4*>(&st[jt * kTileN + 4 * lane]);
                    const size_t o = (size_t)tok * p.n_out + row4;
                    if (f32) {
                        float* y = reinterpret_cast<float*>(p.y) + o;
                        if (vec) *reinterpret_cast<float4*>(y) = f;
                        else {
                            if (row4 + 0 < p.n_out) y[0] = f.x;
                            if (row4 + 1 < p.n_out) y[1] = f.y;
                            if (row4 + 2 < p.n_out) y[2] = f.z;
                            if (row4 + 3 < p.n_out) y[3] = f.w;
                        }
                    } else {
                        uint16_t* y = reinterpret_cast<uint16_t*>(p.y) + o;
                        const uint32_t h01 = pack_bf16x2(f.x, f.y), h23 = pack_bf16x2(f.z, f.w);
                        if (vec) *reinterpret_cast<uint2*>(y) = make_uint2(h01, h23);
                        else {
                            if (row4 + 0 < p.n_out) y[0] = (uint16_t)(h01 & 0xFFFFu);
                            if (row4 + 1 < p.n_out) y[1] = (uint16_t)(h01 >> 16);
                            if (row4 + 2 < p.n_out) y[2] = (uint16_t)(h23 & 0xFFFFu);
                            if (row4 + 3 < p.n_out) y[3] = (uint16_t)(h23 >> 16);
                        }
                    }
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
    cluster_sync();   // MMAs read, barriers are arrived at, in both CTAs: neither leaves before the other has finished
    if (warp == 1) {
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

// ---- host side ------------------------------------------------------------------------------------
static size_t smem_for(const Geometry& g) { return 1024 + (size_t)kStages * kStageBytes + kLutBytes + (size_t)2 * kExpanders * g.unit_bytes; }
// Token tiles of a call, equally wide, as in goq_gemm_tc.cu, over pairs of SMs
static float wave_us(int k_blocks, int tokens) { return 8.f + (float)k_blocks * (0.75f + 0.00085f * (float)tokens); }
struct TokenTiles { int n, half, n_full, n_tail; float us; };
static TokenTiles token_tiles(const Geometry& g, int m) {
    const int pairs = sm_count() / 2, pairs_x = (g.n_pad + 2 * kTileN - 1) / (2 * kTileN);
    TokenTiles best = {};
    const int n0 = (m + 511) / 512;
    for (int n = n0; n <= n0 + 4; ++n) {
        TokenTiles t;
        t.half = ((m + 2 * n - 1) / (2 * n) + 31) & ~31;
        t.n = (m + 2 * t.half - 1) / (2 * t.half);
        const int tiles = pairs_x * t.n, tail = tiles % pairs;
        t.n_tail = (tiles > pairs && 2 * tail <= pairs) ? tail : 0;
        t.n_full = tiles - t.n_tail;
        t.us = (float)((t.n_full + pairs - 1) / pairs) * wave_us(g.k_blocks, 2 * t.half) + (t.n_tail ? 4.f + wave_us(g.k_blocks, t.half) : 0.f);
        if (best.n == 0 || t.us < 0.975f * best.us) best = t;
    }
    return best;
}

template <int WB>
static cudaError_t launch(const Geometry& g, const Params& p0, const void* xh, int m, cudaStream_t st) {
    Params p = p0;
    const TokenTiles tt = token_tiles(g, m);
    CUtensorMap map;
    if (cudaError_t e = encode_x_map(&map, const_cast<void*>(xh), g.k_in, m, tt.half / 2)) return e;
    p.half = tt.half;
    p.pairs_x = (g.n_pad + 2 * kTileN - 1) / (2 * kTileN);
    p.n_full = tt.n_full;
    const size_t smem = smem_for(g);
    static SmemAttrCache smem_attr;
    if (cudaError_t e = ensure_dynamic_smem(gemm_pair_kernel<WB>, smem, smem_attr)) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (tt.n_full + 2 * tt.n_tail));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gemm_pair_kernel<WB>, p, map);
}

}  // namespace tc2

bool gemm_pair_supported(const Geometry& g, int m) { return m > 256 && g.k_in % 8 == 0 && tc2::smem_for(g) + 2048 <= 227 * 1024; }
float gemm_pair_us(const Geometry& g, int m) { return 9.f + tc2::token_tiles(g, m).us; }
cudaError_t launch_gemm_pair(const Geometry& g, const void* packed, const void* xh, const float* inv_scale, const uint32_t* row_scale, const float* row_inv,
                             int m, void* y, int y_dtype, int* status, int spin_limit, cudaStream_t st) {
    tc2::Params p;
    p.packed = (const uint8_t*)packed; p.y = y; p.inv_scale = inv_scale; p.row_scale = row_scale; p.row_inv = row_inv; p.status = status;
    p.spin = spin_limit > 0 ? spin_limit : tc::kSpin;
    p.unit_bytes = g.unit_bytes; p.meta_off = g.meta_off; p.k_blocks = g.k_blocks; p.n_tiles = g.n_tiles; p.n_out = g.n_out; p.m = m; p.y_dtype = y_dtype;
    int lg = 3;
    while ((1 << lg) < g.group) ++lg;
    p.group_log2 = lg;
    return g.wbits == 4 ? tc2::launch<4>(g, p, xh, m, st) : g.wbits == 3 ? tc2::launch<3>(g, p, xh, m, st) : tc2::launch<2>(g, p, xh, m, st);
}

}  // namespace goq
