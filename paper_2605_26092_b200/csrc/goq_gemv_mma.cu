// Decode GEMV on bf16 tensor-core fragments (batch <= 16, wbits 2..4, group >= 32), one 16-row tile per CTA or per cluster.
//
// Eq. 4 of the paper read per macro-block:  y[m,n] = sum_j ( c1[n,j] S1 + c2[n,j] S2 ): b1 and b2 enter mma.sync as exact bf16 PoT
// operands (a PoT factor only shifts the activation's exponent), sums are fp32, the coefficients multiply the group sums outside.
//
// Layout of the work. A warp takes unit records (16 rows x 128 k) of one tile, k-block by k-block, straight from global memory into
// registers, the next record's words and coefficients in flight while one is decoded; lane (g, t) owns whole micro-blocks of rows
// g and g + 8, so the exchange of Section 3.3 never leaves the thread. The activations come through L1, which has the whole SM's
// memory here (12 KB of shared memory a CTA): a ring of weights in shared memory leaves no L1, and with more
// than 40 KB of activations every fragment then came from L2 (4096 x 4096, 8 tokens: 13.9 us). A tile's k-blocks are split
// over the warps of a CTA and, where the tiles are fewer than the chip wants, over the CTAs of a cluster; sums are added in warp
// order, then in rank order through distributed shared memory: deterministic, and no scratch.
// The launch is a programmatic dependent: tables and, in goq_gemv, first records are fetched while the kernel before still runs.
// Bound: instruction issue of the decode (about 280 a record) and, with one or two CTAs a SM, the last wave. 128 registers and 16 warps a
// SM beat 80 and 24 (spills). Measured, W3 g128: 256 x 256 1.5 us in a graph (streaming kernel 5.8), 4096 x 4096 6.4 us at 8 tokens and 8.2
// at 16 (13.9, 15.5), 8192 x 8192 21.7 and 27.3 (30.0, 36.8); W4 26.3 at 8 tokens (the earlier fragment kernel 34.4).
#include <cooperative_groups.h>
#include "goq_fragment.cuh"
#include "goq_internal.h"

namespace goq {
namespace gmma {

constexpr int kMaxWarps = 8;

struct Params {
    const uint8_t* packed;
    const uint16_t* x;
    void* y;
    int unit_bytes, meta_off, y_dtype, n_out, k_in, k_blocks, m, cluster;
    int early;   // records may be read before the kernels ahead on the stream are complete
};

// NT: 8-token columns (1, 2); CPG: 32-wide chunks per macro-block (1, 2, 4)
template <int WB, int NT, int CPG>
__global__ void __launch_bounds__(kMaxWarps * 32, 2) gemv_mma_kernel(const Params p) {
    constexpr int GPB = 4 / CPG;
    __shared__ __align__(128) unsigned char lut[kLutBytes];
    __shared__ __align__(16) float red[kMaxWarps][32 * NT * 4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, n_warps = blockDim.x >> 5;
    const int T = blockIdx.x / p.cluster, rank = blockIdx.x - T * p.cluster;
    const int kb0 = p.k_blocks * rank / p.cluster, kb1 = p.k_blocks * (rank + 1) / p.cluster;   // this CTA's k-blocks
    const uint8_t* unit = p.packed + unit_offset(T, kb0 + warp, p.k_blocks, p.unit_bytes);
    const size_t step = (size_t)n_warps * p.unit_bytes;

    if (!p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    Record<WB, GPB> next;
    int bk = kb0 + warp;
    if (bk < kb1) next.load(unit, p.meta_off);
    fill_table<WB>(lut);
    __syncthreads();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");   // activations and outputs: only after earlier kernels

    const uint32_t lane16 = (uint32_t)(lane & (kLutCopies - 1)) * 16u;
    // lane (g, t): token nt * 8 + g, 8 k from 8 t of a chunk. Tokens that do not exist repeat the last one: an output column depends
    // on its own B column only, and theirs are never stored.
    const uint16_t* xp[NT];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) xp[nt] = p.x + (size_t)min(nt * 8 + g, p.m - 1) * p.k_in + t * 8;
    float acc[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[nt][r] = 0.f;

    for (; bk < kb1; bk += n_warps) {
        const Record<WB, GPB> rec = next;
        unit += step;
        uint4 xa[NT][4];
        load_activations<NT>(xp, bk, p.k_in, xa);
        if (bk + n_warps < kb1) next.load(unit, p.meta_off);
        add_record<WB, NT, CPG>(rec, xa, lut, lane16, acc);
    }

    // ---- sums: warps in order, then the ranks of the cluster in order ----
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
        *reinterpret_cast<float4*>(&red[warp][lane * (NT * 4) + nt * 4]) = make_float4(acc[nt][0], acc[nt][1], acc[nt][2], acc[nt][3]);
    __syncthreads();
    const int o = threadIdx.x;   // element: lane o / (4 NT), accumulator o % (4 NT)
    float s = 0.f;
    if (o < 32 * NT * 4) {
        for (int w = 0; w < n_warps; ++w) s += red[w][o];
    }
    for (int o2 = o + blockDim.x; o2 < 32 * NT * 4; o2 += blockDim.x) {   // (fewer threads than elements: small k only)
        float v = 0.f;
        for (int w = 0; w < n_warps; ++w) v += red[w][o2];
        red[0][o2] = v;
    }
    if (p.cluster > 1) {
        namespace cg = cooperative_groups;
        cg::cluster_group cl = cg::this_cluster();
        __syncthreads();
        if (o < 32 * NT * 4) red[0][o] = s;
        cl.sync();
        if (rank == 0 && o < 32 * NT * 4)
            for (int r = 1; r < p.cluster; ++r) s += *cl.map_shared_rank(&red[0][o], r);
        cl.sync();   // the others' shared memory must outlive the reads
        if (rank != 0) return;
    }
    auto store = [&](int e, float v) {
        const int ln = e / (NT * 4), q = e % (NT * 4), r = q & 3;
        const int row = T * kTileRows + (ln >> 2) + ((r & 2) ? 8 : 0), tok = (q >> 2) * 8 + (ln & 3) * 2 + (r & 1);
        if (row < p.n_out && tok < p.m) {
            if (p.y_dtype == GOQ_F32) reinterpret_cast<float*>(p.y)[(size_t)tok * p.n_out + row] = v;
            else reinterpret_cast<uint16_t*>(p.y)[(size_t)tok * p.n_out + row] = f32_to_bf16_rne(v);
        }
    };
    if (o < 32 * NT * 4) store(o, s);
    for (int o2 = o + blockDim.x; o2 < 32 * NT * 4; o2 += blockDim.x) store(o2, red[0][o2]);
}

template <int WB, int NT, int CPG>
static cudaError_t launch(const Geometry& g, Params& p, cudaStream_t st) {
    int warps = g.k_blocks < kMaxWarps ? (g.k_blocks < 4 ? 4 : g.k_blocks) : kMaxWarps;
    // Few k-blocks and many tiles: what a CTA costs beside its records (table, start, sums) counts, and half the warps mean twice the CTAs
    // in flight and two records a warp
    if (g.k_blocks <= kMaxWarps && g.n_tiles > 4 * sm_count()) warps = 4;
    // A cluster per tile only while there are fewer CTAs than SMs and every warp keeps a record (1024 x 4096: 3.7 us, without 6.0; a
    // second CTA per SM by the same means costs more than it gives: 4096 x 4096 6.3 -> 9 us)
    int cluster = 1;
    while (cluster < 8 && g.n_tiles * cluster < sm_count() && g.k_blocks >= 2 * cluster * warps) cluster *= 2;
    p.cluster = cluster;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g.n_tiles * cluster);
    cfg.blockDim = dim3(warps * 32);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, gemv_mma_kernel<WB, NT, CPG>, p);
}

}  // namespace gmma

bool gemv_mma_supported(const Geometry& g, int m) { return g.group >= 32 && m <= 16 && g.n_tiles < (1 << 27); }

cudaError_t launch_gemv_mma(const Geometry& g, const void* packed, const void* x, int m, void* y, int y_dtype, bool early, cudaStream_t st) {
    gmma::Params p;
    p.packed = (const uint8_t*)packed; p.x = (const uint16_t*)x; p.y = y;
    p.unit_bytes = g.unit_bytes; p.meta_off = g.meta_off; p.y_dtype = y_dtype; p.n_out = g.n_out; p.k_in = g.k_in;
    p.k_blocks = g.k_blocks; p.m = m; p.early = early ? 1 : 0;
#define GOQ_GMMA_NT(WB_, NT_) \
    (g.group == 32 ? gmma::launch<WB_, NT_, 1>(g, p, st) : g.group == 64 ? gmma::launch<WB_, NT_, 2>(g, p, st) : gmma::launch<WB_, NT_, 4>(g, p, st))
#define GOQ_GMMA(WB_) (m <= 8 ? GOQ_GMMA_NT(WB_, 1) : GOQ_GMMA_NT(WB_, 2))
    return g.wbits == 4 ? GOQ_GMMA(4) : g.wbits == 3 ? GOQ_GMMA(3) : GOQ_GMMA(2);
#undef GOQ_GMMA
#undef GOQ_GMMA_NT
}

}  // namespace goq
