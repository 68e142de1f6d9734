// What follows gemm_f8_kernel (goq_gemm_f8.cu): the sums of the tiles that several CTAs share, and the outputs of the tokens that its pre-pass has marked (elements
// that its activation slices do not hold), from the bf16 activations themselves as gemv_mma_kernel computes them: a 16-row tile after the other, its k-blocks
// over the CTA's warps, sums in warp order.
// Marked tokens add, whatever their number, 53 us to a call of 8192 x 8192 at 16 tokens and 215 to one of 28672 x 8192 (gemv_mma_kernel's own calls take 27 and 83):
// latency of few warps' loads; they are rare. grid: (channel tiles x token tiles, token slices, shares of a channel tile's rows for that).
#include "goq_streamk.cuh"
#include "goq_fragment.cuh"
#include "goq_internal.h"

namespace goq {
namespace f8 {

using streamk::FinishParams;
using streamk::kFinishThreads;
using streamk::kFinishTokens;

struct MarkedParams {
    const uint8_t* packed;
    const uint16_t* x;
    const int* marks;   // [m]
    int unit_bytes, meta_off, k_in, n_tiles;
};

template <int WB, int CPG>
__global__ void __launch_bounds__(kFinishThreads, 3) finish_f8_kernel(const __grid_constant__ FinishParams p, const __grid_constant__ MarkedParams e) {
    constexpr int kWarps = kFinishThreads / 32;
    __shared__ __align__(128) unsigned char lut[kLutBytes];
    __shared__ __align__(16) float red[kWarps][32 * 8];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tile = blockIdx.x, tok0 = (tile / p.tiles_x) * p.n_cols + blockIdx.y * kFinishTokens;
    const int n = min(min(kFinishTokens, p.n_cols - (int)blockIdx.y * kFinishTokens), p.m - tok0);
    uint32_t marked = 0u;
    auto look = [&] { return marked = __ballot_sync(0xFFFFFFFFu, lane < n && __ldcg(e.marks + tok0 + lane) != 0); };
    if (blockIdx.z == 0) streamk::finish_tile(p, look);
    else {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        look();
    }
    if (marked == 0u) return;
    gmma::fill_table<WB>(lut);
    const int g = lane >> 2, t = lane & 3, T0 = (tile % p.tiles_x) * (streamk::kTileN / kTileRows);
    const uint32_t lane16 = (uint32_t)(lane & (kLutCopies - 1)) * 16u;
    const uint16_t* xp[2];
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) xp[nt] = e.x + (size_t)(tok0 + min(nt * 8 + g, n - 1)) * e.k_in + t * 8;
    for (int T = T0 + blockIdx.z; T < min(T0 + streamk::kTileN / kTileRows, e.n_tiles); T += gridDim.z) {
        __syncthreads();   // the table is filled; the sums of the tile before are read
        float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
        gmma::Record<WB, 4 / CPG> next;
        int bk = warp;
        if (bk < p.k_blocks) next.load(e.packed + unit_offset(T, bk, p.k_blocks, e.unit_bytes), e.meta_off);
        for (; bk < p.k_blocks; bk += kWarps) {
            const gmma::Record<WB, 4 / CPG> rec = next;
            uint4 xa[2][4];
            gmma::load_activations<2>(xp, bk, e.k_in, xa);
            if (bk + kWarps < p.k_blocks) next.load(e.packed + unit_offset(T, bk + kWarps, p.k_blocks, e.unit_bytes), e.meta_off);
            gmma::add_record<WB, 2, CPG>(rec, xa, lut, lane16, acc);
        }
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) *reinterpret_cast<float4*>(&red[warp][lane * 8 + nt * 4]) = make_float4(acc[nt][0], acc[nt][1], acc[nt][2], acc[nt][3]);
        __syncthreads();
        const int o = threadIdx.x, ln = o >> 3, r = o & 3, col = ((o >> 2) & 1) * 8 + (ln & 3) * 2 + (r & 1), ch = T * kTileRows + (ln >> 2) + ((r & 2) ? 8 : 0);
        float s = 0.f;
        for (int w = 0; w < kWarps; ++w) s += red[w][o];
        if (((marked >> col) & 1u) && ch < p.n_out) {
            const streamk::Output out = {p.y, p.y_dtype, p.n_out};
            out.store1(tok0 + col, ch, s);
        }
    }
}

template <int WB, int CPG>
static cudaError_t launch(const FinishParams& f, const MarkedParams& e, dim3 grid, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kFinishThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, finish_f8_kernel<WB, CPG>, f, e);
}

}  // namespace f8

cudaError_t launch_f8_finish(const Geometry& g, const void* packed, const void* x, int m, void* y, int y_dtype, const float* partial, const float* inv_scale,
                             const int* marks, int tile_tokens, int tiles_x, int t_tiles, int units, int n_ctas, cudaStream_t st) {
    const f8::FinishParams f = {partial, inv_scale, y, y_dtype, g.n_out, m, tile_tokens, tiles_x, g.k_blocks, units, n_ctas};
    const f8::MarkedParams e = {(const uint8_t*)packed, (const uint16_t*)x, marks, g.unit_bytes, g.meta_off, g.k_in, g.n_tiles};
    const int slices = (tile_tokens + f8::kFinishTokens - 1) / f8::kFinishTokens, ctas = tiles_x * t_tiles * slices;
    // (shares only while all CTAs run at once: most launches find no mark)
    const dim3 grid(tiles_x * t_tiles, slices, ctas >= 2 * sm_count() ? 1 : ctas * 8 <= 2 * sm_count() ? 8 : 2 * sm_count() / ctas);
#define GOQ_FIN(WB_) (g.group == 32 ? f8::launch<WB_, 1>(f, e, grid, st) : g.group == 64 ? f8::launch<WB_, 2>(f, e, grid, st) : f8::launch<WB_, 4>(f, e, grid, st))
    return g.wbits == 4 ? GOQ_FIN(4) : g.wbits == 3 ? GOQ_FIN(3) : GOQ_FIN(2);
#undef GOQ_FIN
}

}  // namespace goq
