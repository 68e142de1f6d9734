// One decode GEMV (batch <= 4) in integer operands: the arithmetic, the split of the records and the reduction order of the
// chain kernel (goq_gemv_chain.cu; the outputs are the same bits), laid out for a call of its own.
//
// A single linear of 8-24 MB is 2-8 us of work, so what surrounds it counts: a cooperative launch cannot overlap the kernel before
// it, and its 17 KB of parameters for up to 256 linears are copied on every call. This kernel takes 150 bytes of parameters and is a
// programmatic dependent of the kernel before it: on an SM that has room, the ring of packed records fills, tables and barriers are set up while
// that one still runs; activations, outputs and scratch are touched after griddepcontrol.wait. (Behind a call of its own kind a CTA, 576 threads of 88
// registers, finds room only where that call's CTA has ended.)
//
// Tiles shared by several CTAs: every CTA but the one that holds the tile's end posts its part (at most one per CTA) in the
// zero-kept counter area, a word a value: zero means "not there yet" and a sum of +0 is posted as -0. The finisher polls the words it
// needs and zeroes them again: no fence, no counter, no launch number. It waits on lower-numbered CTAs only. That these run is not a
// guarantee of an ordinary launch: it relies on CTAs being dispatched in the order of their numbers, one per SM, as they are in practice;
// were they not, the wait would run out and be reported. Every wait is bounded (abort flag, GOQ_ERR_TIMEOUT in the status word).
// Bound: instruction issue of the decode (see goq_gemv_chain.cu) plus ~4 us of start, conversion and hand-over latency.
#include "goq_int_core.cuh"
#include "goq_internal.h"
#include <type_traits>

namespace goq {
namespace chain {

constexpr int kOneThreads = (kNW + 2) * 32;   // consumer warps, one control warp, one producer warp
constexpr int kPostWords = 64;                // 16 rows x 4 tokens

struct One {
    const uint8_t* packed;
    const uint16_t* x;
    void* y;
    uint32_t* posts;   // [CTA][kPostWords], zero on entry, left zero
    int* status;
    unsigned long long kb_magic, g_magic, m_magic;   // as in the chain kernel: divisions by k_blocks, by the number of CTAs, by m
    unsigned int units, uq, ur;
    int k_blocks, k_in, n_out, m, y_dtype, unit_bytes, n_stages, spin;
};

template <int WB, int CPG, bool K1>
__global__ void __launch_bounds__(kOneThreads, 1) gemv_one_kernel(const __grid_constant__ One p) {
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char* lut = smem + ((8192u - (smem_u32(smem) & 8191u)) & 8191u);   // 8 KiB boundary: slot offsets are OR-ed in
    const int stage_bytes = kStageRecs * p.unit_bytes;
    unsigned char* ring = lut + kLutBytes;
    float* red = reinterpret_cast<float*>(ring + (size_t)p.n_stages * stage_bytes);     // [slot][warp][64]
    float* xsc = red + kTileSlots * kNW * 64;                                           // [k-block][4 tokens]
    unsigned char* xq = reinterpret_cast<unsigned char*>(xsc + kMaxKBlocks * 4);        // [2 m][k_pad + kXPad] int8 planes
    __shared__ uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], part_bar[kTileSlots];
    __shared__ volatile int abort_flag;
    __shared__ volatile int done_gen[kTileSlots];

    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
    const int G = (int)gridDim.x, cta = (int)blockIdx.x;
    const int spin = p.spin;
    const Walk wk = make_walk(p, cta, p.g_magic);
    const unsigned kb = (unsigned)p.k_blocks;

    // one stage of the ring: positions j0 .. of the walk, one run of records or two if it straddles the walk's turn
    auto issue = [&](unsigned j0, int slot) {
        const unsigned n = min((unsigned)kStageRecs, wk.L - j0), n1 = (j0 < wk.L1) ? min(n, wk.L1 - j0) : 0u;
        unsigned char* dst = ring + (size_t)slot * stage_bytes;
        mbar_arrive_expect_tx(&full_bar[slot], n * (unsigned)p.unit_bytes);
        if (n1) bulk_copy_g2s(dst, p.packed + (size_t)walk_record(wk, j0) * p.unit_bytes, n1 * (unsigned)p.unit_bytes, &full_bar[slot]);
        if (n > n1)
            bulk_copy_g2s(dst + (size_t)n1 * p.unit_bytes, p.packed + (size_t)walk_record(wk, j0 + n1) * p.unit_bytes,
                          (n - n1) * (unsigned)p.unit_bytes, &full_bar[slot]);
    };
    constexpr int kProd = kNW + 1, kCtrl = kNW;
    unsigned j_next = 0;
    if (warp == kProd && lane == 0) {   // fill the ring before anything else
        for (int s = 0; s < p.n_stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], kNW); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int s = 0; s < p.n_stages && j_next < wk.L; ++s, j_next += kStageRecs) issue(j_next, s);
    }
    if (tid == 0) {
        abort_flag = 0;
        for (int i = 0; i < kTileSlots; ++i) { done_gen[i] = 0; mbar_init(&part_bar[i], kNW); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < 64 * kLutCopies; i += kOneThreads) {
        const uint32_t* e = c_exchange_lut.v[i / kLutCopies];
        *reinterpret_cast<uint4*>(lut + (size_t)i * 16) = make_uint4(e[0], e[1], (e[2] >> 7) * 255u, (e[3] >> 7) * 255u);
    }
    __syncthreads();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // ================= producer =================
    if (warp == kProd) {
        if (lane == 0) {
            int slot = 0, round = 1, issued = (int)(j_next / kStageRecs);
            bool ok = true;
            for (; j_next < wk.L; j_next += kStageRecs) {
                if (!wait_bar(&empty_bar[slot], (round - 1) & 1, &abort_flag, spin)) { ok = false; break; }
                issue(j_next, slot);
                if (++slot == p.n_stages) { slot = 0; ++round; }
                ++issued;
            }
            if (!ok || abort_flag) {   // copies in flight must land before the CTA's shared memory goes away
                drain_issued_stages(full_bar, issued, p.n_stages);
                atomicExch(p.status, (int)GOQ_ERR_TIMEOUT);
            }
        }
        return;
    }

    asm volatile("griddepcontrol.wait;" ::: "memory");   // activations, outputs and scratch: only after earlier kernels

    // ================= control: reduction and stores =================
    if (warp == kCtrl) {
        bool ok = true;
        const unsigned rem_a = (unsigned)cta * p.ur - (unsigned)G * mul_shift32((unsigned)cta * p.ur, p.g_magic);
        const int tok0 = lane & 3;
        const bool tokv = tok0 < p.m, y32 = p.y_dtype == GOQ_F32;
        for (int q = 0; q < wk.P; ++q) {
            const int rs = q % kTileSlots;
            const int T = walk_tile_of_part(wk, q);
            const unsigned r_lo = (unsigned)T * kb, r_hi = r_lo + kb;
            const bool finisher = r_hi <= wk.b;          // this CTA holds the tile's end
            const size_t yoff = (size_t)tok0 * p.n_out + T * 16 + (lane >> 2);
            const bool rowv[2] = {T * 16 + (lane >> 2) < p.n_out, T * 16 + (lane >> 2) + 8 < p.n_out};
            const float* rall = red + (size_t)rs * kNW * 64 + lane;
            // A tile finished for others: their parts were posted early (every CTA starts with the tile that is open at the end of
            // its range), so they are fetched before this CTA's own sums are ready - nearest CTA first.
            float below[2] = {0.f, 0.f};
            if (r_lo < wk.a && finisher) {
                unsigned bc = wk.a, remc = rem_a;   // upper boundary of CTA cc's range
                for (int cc = cta - 1; cc >= 0 && bc > r_lo && ok; --cc) {
                    const unsigned borrow = remc < p.ur ? 1u : 0u;
                    const unsigned ac = bc - p.uq - borrow;
                    remc = remc - p.ur + (borrow ? (unsigned)G : 0u);
                    if (ac != bc) {
                        uint32_t* pc = p.posts + (size_t)cc * kPostWords + lane;
                        int spins = 0;
                        for (;;) {
                            uint32_t w0, w1;
                            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(w0) : "l"(pc) : "memory");
                            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(w1) : "l"(pc + 32) : "memory");
                            if (__all_sync(0xFFFFFFFFu, w0 != 0u && w1 != 0u)) {
                                below[0] += __uint_as_float(w0); below[1] += __uint_as_float(w1);
                                pc[0] = 0u; pc[32] = 0u;   // left zero for the next call
                                break;
                            }
                            ++spins;
                            if (__any_sync(0xFFFFFFFFu, abort_flag != 0) || spins > kGlobalSpin || spins > spin) { abort_flag = 1; ok = false; break; }
                        }
                    }
                    bc = ac;
                }
                if (!ok) break;
            }
            if (!wait_bar(&part_bar[rs], (q / kTileSlots) & 1u, &abort_flag, spin)) { ok = false; break; }
            float out[2];
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                float v[kNW];
#pragma unroll
                for (int w2 = 0; w2 < kNW; ++w2) v[w2] = rall[(size_t)w2 * 64 + hh * 32];
#pragma unroll
                for (int sft = kNW / 2; sft >= 1; sft >>= 1)   // fixed pairing: deterministic
#pragma unroll
                    for (int w2 = 0; w2 < sft; ++w2) v[w2] += v[w2 + sft];
                out[hh] = v[0] + below[hh];
            }
            __syncwarp();
            if (lane == 0) done_gen[rs] = q + 1;   // every lane has read the slot: it may be parked in again
            if (!finisher) {
                uint32_t* post = p.posts + (size_t)cta * kPostWords + lane;
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const uint32_t bits = __float_as_uint(out[hh]);
                    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(post + hh * 32), "r"(bits ? bits : 0x80000000u) : "memory");
                }
            } else if (tokv) {
#pragma unroll
                for (int hh = 0; hh < 2; ++hh)
                    if (rowv[hh]) {
                        if (y32) reinterpret_cast<float*>(p.y)[yoff + hh * 8] = out[hh];
                        else {
                            uint32_t h;
                            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(0.f), "f"(out[hh]));
                            reinterpret_cast<uint16_t*>(p.y)[yoff + hh * 8] = (uint16_t)(h & 0xFFFFu);
                        }
                    }
            }
        }
        if (lane == 0 && abort_flag) atomicExch(p.status, (int)GOQ_ERR_TIMEOUT);
        return;
    }

    // ================= consumers =================
    const int g = lane >> 2, t = lane & 3;
    const int k_pad = p.k_blocks * kBlockK, plane = k_pad + kXPad, m = p.m;
    {   // activations -> block fixed point, by all consumer warps; only the k-blocks this CTA's records use (a range shorter than a
        // tile's row of records needs that many). Half warps take (k-block, token) pairs; four loads a lane in flight.
        const unsigned kb0 = wk.a - (unsigned)wk.Ta * kb, total = min(wk.L, kb) * (unsigned)m * 16u;
        constexpr unsigned kBatch = 4;
        for (unsigned c0 = (unsigned)warp * 32u; c0 < total; c0 += kNW * 32u * kBatch) {
            uint4 v[kBatch];
            unsigned at[kBatch];   // token << 16 | first k
#pragma unroll
            for (unsigned i = 0; i < kBatch; ++i) {
                if (i > 0 && c0 + i * (kNW * 32u) >= total) break;   // warp-uniform
                const unsigned c = c0 + i * (kNW * 32u) + (unsigned)lane, pair = c >> 4;
                unsigned j = mul_shift32(pair, p.m_magic);
                const unsigned r = pair - j * (unsigned)m;
                j += kb0;
                if (j >= kb) j -= kb;
                const unsigned k0 = j * kBlockK + (c & 15u) * 8u;
                at[i] = (r << 16) | k0;
                v[i] = make_uint4(0u, 0u, 0u, 0u);
                if (c < total && k0 < (unsigned)p.k_in) v[i] = __ldcg(reinterpret_cast<const uint4*>(p.x + (size_t)r * p.k_in + k0));
            }
#pragma unroll
            for (unsigned i = 0; i < kBatch; ++i) {
                if (c0 + i * (kNW * 32u) < total) {   // warp-uniform: the conversion shuffles
                    const unsigned r = at[i] >> 16, k0 = at[i] & 0xFFFFu;
                    convert_chunk<WB>(v[i], c0 + i * (kNW * 32u) + (unsigned)lane < total, xq + (size_t)(2 * r) * plane + k0, plane,
                                      xsc + (k0 >> 7) * 4 + r);
                }
            }
        }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(kNW * 32) : "memory");   // consumer warps only; none of them has left yet

    const uint32_t lut_lane = smem_u32(lut) + (lane & (kLutCopies - 1)) * 16;
    const uint32_t unit_bytes = (uint32_t)p.unit_bytes;
    const uint32_t full_addr = smem_u32(full_bar), empty_addr = smem_u32(empty_bar);
    // B fragment of lane (g, t): column g = plane g (token g/2, slice g&1); planes of tokens that do not exist alias the last real one
    const uint32_t xrow = order_after_wait(smem_u32(xq) + (uint32_t)(min(g, 2 * m - 1) * plane + t * 8));
    const uint32_t xs_tok = smem_u32(xsc + min(t, m - 1));
    FlushCtx fc;
    fc.red_addr = smem_u32(red); fc.part_bar_addr = smem_u32(part_bar); fc.done_gen = done_gen; fc.abort_flag = &abort_flag; fc.spin = spin;
    bool alive = true;
    int cur_q = 0;
    float acc[2] = {0.f, 0.f};
    auto flush_to = [&](int qn) {   // hand over the parts this warp has passed (or never touched: zeros)
        for (; cur_q < qn && alive; ++cur_q) {
            Sums4 sums;
            sums.v[0] = acc[0]; sums.v[1] = acc[1]; sums.v[2] = sums.v[3] = 0.f;
            if (!flush_part<1>(fc, (unsigned)cur_q, sums)) alive = false;
            acc[0] = acc[1] = 0.f;
        }
    };
    // chunks cb .. ce-1 of a record (all four in the full stages)
    auto record = [&](uint32_t unit, uint32_t kbi, auto whole, unsigned cb, unsigned ce) {
        constexpr bool kWhole = decltype(whole)::value;
        const uint4 wv0 = lds128(unit), wv1 = lds128(unit + 512);
        const uint32_t coef_addr = unit - lane * 16 + kCodeBytesPerUnit + g * 4;
        const uint32_t w0[4] = {wv0.x, wv0.y, wv0.z, wv0.w}, w1[4] = {wv1.x, wv1.y, wv1.z, wv1.w};
        int s1[1][4], s2[1][4], s3[1][4];
        float rec[1][2] = {{0.f, 0.f}};
#pragma unroll
        for (int r = 0; r < 4; ++r) s1[0][r] = s2[0][r] = s3[0][r] = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (kWhole || ((unsigned)c >= cb && (unsigned)c < ce)) {   // warp-uniform
                uint32_t pa0, pb0, qa0, qb0, fa0, fb0, pa1, pb1, qa1, qb1, fa1, fb1;
                decode_word<WB, K1>(w0[c], lut_lane, pa0, pb0, qa0, qb0, fa0, fb0);
                decode_word<WB, K1>(w1[c], lut_lane, pa1, pb1, qa1, qb1, fa1, fb1);
                const uint2 xf = lds64(xrow + kbi * kBlockK + c * 32);
                mma_s8(s1[0], pa0, pa1, pb0, pb1, xf.x, xf.y);
                if constexpr (!K1) {
                    mma_s8(s2[0], qa0, qa1, qb0, qb1, xf.x, xf.y);
                    mma_s8(s3[0], fa0, fa1, fb0, fb1, xf.x, xf.y);
                }
                if (((c + 1) % CPG) == 0 || (!kWhole && (unsigned)(c + 1) == ce))
                    group_end<1, K1>(s1, s2, s3, lds32(coef_addr + (c / CPG) * 64), lds32(coef_addr + (c / CPG) * 64 + 32), rec);
            }
        }
        const float sv = lds_f32(xs_tok + kbi * 16);   // undo the activation scale of this k-block
        acc[0] = fmaf(sv, rec[0][0], acc[0]);
        acc[1] = fmaf(sv, rec[0][1], acc[1]);
    };

    const unsigned n_full = wk.L / kStageRecs, n_tail = wk.L - n_full * kStageRecs;
    const uint32_t unit0 = smem_u32(ring) + (uint32_t)warp * unit_bytes + (uint32_t)lane * 16;
    int slot = 0, phase = 0;
    uint32_t stage_off = 0, bar_off = 0;
    {
        unsigned j = (unsigned)warp;
        unsigned kbi = 0;
        int q = 0;
        bool locate = true;
        for (unsigned st = 0; st < n_full && alive; ++st) {
            if (locate) {
                const unsigned rho = walk_record(wk, j);
                const int T = (int)mul_shift32(rho, p.kb_magic);
                kbi = rho - (unsigned)T * kb;
                q = walk_part_of_tile(wk, T);
                locate = false;
            }
            if (cur_q < q) { flush_to(q); if (!alive) break; }
            {   // bounded wait, written out so that the record loop contains no call
                int polls = 0;
                while (!try_wait_a(full_addr + bar_off, phase)) {
                    if (++polls >= spin || ((polls & 255) == 0 && abort_flag)) { abort_flag = 1; alive = false; break; }
                }
            }
            record(order_after_wait(unit0 + stage_off), kbi, std::true_type{}, 0u, 4u);
            __syncwarp();
            if (lane == 0) arrive_a(empty_addr + bar_off);
            stage_off += (uint32_t)stage_bytes; bar_off += 8;
            if (++slot == p.n_stages) { slot = 0; phase ^= 1; stage_off = 0; bar_off = 0; }
            const bool before_turn = j < wk.L1;
            j += kStageRecs;
            kbi += kStageRecs;
            while (kbi >= kb) { kbi -= kb; ++q; }
            if (before_turn && j >= wk.L1) locate = true;
        }
    }
    if (n_tail && alive) {   // the last stage, shared out by 32-wide chunks
        const unsigned share = c_tail_share.v[n_tail][warp];
        const unsigned rloc = share & 15u, cb = (share >> 4) & 7u, ce = (share >> 7) & 7u;
        if (rloc < n_tail && cb < ce) {
            const unsigned rho = walk_record(wk, n_full * kStageRecs + rloc);
            const unsigned T = mul_shift32(rho, p.kb_magic);
            flush_to(walk_part_of_tile(wk, (int)T));
            if (alive && !wait_a(full_addr + bar_off, phase, &abort_flag, spin)) alive = false;
            if (alive) record(order_after_wait(smem_u32(ring) + slot * stage_bytes + rloc * unit_bytes + lane * 16), rho - T * kb, std::false_type{}, cb, ce);
        }
    }
    flush_to(wk.P);
    if (lane == 0 && abort_flag) atomicExch(p.status, (int)GOQ_ERR_TIMEOUT);
}

static constexpr size_t kOneSmemMax = 226 * 1024;   // the opt-in limit is 227 KiB per CTA, static shared variables included
static size_t one_fixed_smem(const Geometry& g, int m) {
    return 8192 /* alignment slack */ + (size_t)kLutBytes + (size_t)kTileSlots * kNW * 64 * sizeof(float) +
           (size_t)kMaxKBlocks * 4 * sizeof(float) + (((size_t)2 * m * (g.k_pad + kXPad) + 127) & ~(size_t)127);
}

template <int WB, int CPG, bool K1>
static cudaError_t launch_one_cfg(const Geometry& g, One& p, int grid, cudaStream_t st) {
    auto kernel = gemv_one_kernel<WB, CPG, K1>;
    const size_t fixed = one_fixed_smem(g, p.m), stage = (size_t)kStageRecs * g.unit_bytes;
    int n_stages = (int)((kOneSmemMax - fixed) / stage);
    if (n_stages > kMaxStages) n_stages = kMaxStages;
    const int need = (int)((p.units / (unsigned)grid + 1 + kStageRecs - 1) / kStageRecs);   // stages of the longest range
    if (n_stages > need) n_stages = need;
    p.n_stages = n_stages;
    const size_t smem = fixed + (size_t)n_stages * stage;
    static SmemAttrCache smem_attr;
    if (cudaError_t e = ensure_dynamic_smem(kernel, smem, smem_attr)) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kOneThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

}  // namespace chain

bool gemv_one_supported(const Geometry& g, int m) {
    return m <= 4 && gemv_seq_supported(g, m) && chain::one_fixed_smem(g, m) + (size_t)2 * chain::kStageRecs * g.unit_bytes <= chain::kOneSmemMax &&
           (size_t)sm_count() * chain::kPostWords * sizeof(uint32_t) <= kWsCounterBytes;
}

cudaError_t launch_gemv_one(const Geometry& g, const void* packed, const void* x, int m, void* y, int y_dtype, void* ws, int spin_limit,
                            cudaStream_t st) {
    chain::One p;
    p.packed = (const uint8_t*)packed;
    p.x = (const uint16_t*)x;
    p.y = y;
    p.status = (int*)ws;
    p.posts = (uint32_t*)((uint8_t*)ws + kWsStatusBytes);
    p.units = (unsigned)g.n_units;
    const int sms = sm_count(), grid = p.units < (unsigned)sms ? (int)p.units : sms;
    p.kb_magic = ((1ull << 32) + (unsigned)g.k_blocks - 1) / (unsigned)g.k_blocks;
    p.g_magic = ((1ull << 32) + (unsigned)grid - 1) / (unsigned)grid;
    p.m_magic = ((1ull << 32) + (unsigned)m - 1) / (unsigned)m;
    p.uq = p.units / (unsigned)grid;
    p.ur = p.units % (unsigned)grid;
    p.k_blocks = g.k_blocks; p.k_in = g.k_in; p.n_out = g.n_out; p.m = m; p.y_dtype = y_dtype; p.unit_bytes = g.unit_bytes;
    p.spin = spin_limit > 0 ? spin_limit : kSpinLimit;
#define GOQ_ONE(WB_, K1_)                                                                                        \
    (g.group == 32 ? chain::launch_one_cfg<WB_, 1, K1_>(g, p, grid, st) : g.group == 64 ? chain::launch_one_cfg<WB_, 2, K1_>(g, p, grid, st) \
                                                                                       : chain::launch_one_cfg<WB_, 4, K1_>(g, p, grid, st))
    if (g.k1) return g.wbits == 3 ? GOQ_ONE(3, true) : GOQ_ONE(2, true);
    return g.wbits == 3 ? GOQ_ONE(3, false) : GOQ_ONE(2, false);
#undef GOQ_ONE
}

}  // namespace goq
