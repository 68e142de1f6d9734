// REF-mode coefficients (Section 3.4, Eq. 3) with the Gram matrix as int8 digits on the tensor cores; groups of 32 and more.
//
// Per row and macro-block column j:  c* = (A^T A + lambda I)^-1 A^T Y,  A = [X_q b1, X_q b2],  Y = X_q w.  With G = X_q^T X_q (float64, shared
// by all rows) and V_b = G b_b, the five entries of the normal equations are
//   b1.V_1   b1.V_2   b2.V_2   w.V_1   w.V_2 .
// b1 and b2 are small integers times 2^-emax. So V_b needs no float64 products: every row k of G is written as 64-bit fixed point against its
// largest element, |G_kl| 2^s_k < 2^62, and cut into eight signed byte digits; the digits times b_b are tcgen05 kind::i8 MMAs, exact in int32.
// Recombining the eight sums and the five products with b1, b2, w is all the float64 that is left: 8 operations per element and vector
// instead of 1.5 g. A G_kl is rounded to 2^-63 of its row's largest element. While that is at most 2^10 times the row's diagonal element, the rounding is at
// most 2^-53 G_kk, no more than that of a float64 product with a state of 1, and the result is no further from the exact one than float64 sums are (the
// entries of G itself are float64 sums, as in solve_ref_kernel). Where one channel is so much larger than another that a row goes beyond (some 10^4 times),
// rows of W with zero states there would see the rounding of elements that they multiply by zero (2^20 times: 6e-14): such a column is solved in float64 from
// G as it is (solve_wide), its digits unused. 4096 x 4096, 256 observations, every column so: 106 -> 317 us (solve_ref_kernel 324).
//
// A column belongs to a cluster of `C` CTAs: each forms 1 / C of the lower triangle of G (float64 tensor pipe), takes the others'
// blocks through distributed shared memory, cuts all of G into digits, and solves its share of the 128-row tiles. Roles: warps 0-15 add up V_1 and V_2
// (a thread is a row; half of the elements each), 16-19 decode codes and records into int8 operands, 20 issues MMAs, 21 fetches w (TMA). A pass is 32 elements of V
// (N = 256: 32 x 8 digits); V_1 and V_2 have half of tensor memory each, so one is read while the other is computed.
// Bound: instruction issue of the recombination (about 35 instructions an element and vector; issue 46 %, integer pipe 28 %, float64 15 %, int8 MMAs
// 14 %), 17.6 K clocks a tile of 128 rows x 128, and 35 K clocks at the start (G 19 K, its exchange 7 K, digits 8 K).
// Measured, W3, in groups of 128: 4096 x 4096 with 256 observations 324 -> 104 us (solve_ref_kernel before), 8192 x 8192 with 512 1227 -> 355, 512 x 512
// with 128 37 -> 29; groups of 64: 205 -> 92; of 32, W4: 201 -> 107. Not kept: V in passes of 8 elements with two passes a warp in tensor memory (134 us: a
// wait costs more than the overlap gives); eight recombining warps (134); operands and w set up while G is formed (111).
// Error against long double (2-norm, relative) 1.7e-16 where the float64 products had 2.7e-16, 3.3e-12 against 3.7e-12 where the observations' mean is 100
// times their deviation.
// Every mbarrier wait is bounded; a CTA that gives up writes NaN for its rows.
#include "goq_tc_core.cuh"
#include "goq_internal.h"
#include "goq_ref_rows.cuh"
#include <type_traits>

namespace goq {
namespace reftc {

using namespace tc;

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kEpiWarps = 16, kDec0 = 16, kDecWarps = 4, kMmaWarp = 20, kWWarp = 21;
constexpr int kThreads = 22 * 32;
constexpr int kRows = 128;          // rows of a tile
constexpr int kPassK = 32;          // elements of V in a pass
constexpr int kDigits = 8;
constexpr int kTileBytes = kRows * 128;
constexpr int kWK = 16, kWStages = 3, kWBytes = kRows * kWK * 4;   // w: 16 columns of a tile at a time
constexpr int kBlkRow = 9, kBlkStride = 74;   // doubles between rows of a block of G and between blocks: few bank conflicts while digits are cut
constexpr int kChunk = 64;          // observations staged at a time while G is formed

// Operand tiles of one row tile: b1, b2; W4 also the units by which +2^emax = 128 exceeds an int8
template <int WB> __host__ __device__ constexpr int tiles_per_buffer() { return WB == 4 ? 4 : 2; }
template <int WB, int G> __host__ __device__ constexpr int buffers() { return WB == 4 && G == 128 ? 1 : 2; }
template <int G> struct Gram {
    static constexpr int kNB = G / 8, kBlocks = kNB * (kNB + 1) / 2;   // 8 x 8 blocks of the lower triangle
    static constexpr int kStride = G + 8;                              // floats per staged observation: fragment reads are conflict-free
    static constexpr size_t kStageBytes = 2ull * kChunk * kStride * 4;
    static constexpr size_t kDigitBytes = (size_t)G * kDigits * 128;   // row (k, digit): 128 bytes of l
};
template <int WB, int G> struct Smem {
    // digits | operand tiles | w; while G is formed: observations at the start, the triangle at the end
    static constexpr size_t kA = Gram<G>::kDigitBytes, kW = kA + (size_t)buffers<WB, G>() * tiles_per_buffer<WB>() * kTileBytes;
    static constexpr size_t kRun = kW + kWStages * kWBytes;
    static constexpr size_t kTri = (size_t)Gram<G>::kBlocks * kBlkStride * 8;
    static constexpr size_t kForm = (Gram<G>::kStageBytes > Gram<G>::kDigitBytes ? Gram<G>::kStageBytes : Gram<G>::kDigitBytes) + kTri;
    static constexpr size_t kTriOff = (kRun > kForm ? kRun : kForm) - kTri;
    static constexpr size_t kBytes = (kRun > kForm ? kRun : kForm) + 1024;
    static_assert(quant::RefSmem<G / 8>::kFrags * 32 * sizeof(double) <= kTriOff && quant::RefSmem<G / 8>::kBytes + 1024 <= kBytes, "solve_wide");
};

struct Params {
    const uint8_t *codes, *meta;
    const float *xc, *w;
    uint16_t* coef;
    double* c_out;
    double lambda;
    int n_out, k_in, m, tiles, c, spin;   // c: CTAs of a cluster
};

// kind::i8: s8 x s8 -> s32, both K-major, M = 128, N = 256
constexpr uint32_t kIdesc = (2u << 4) | (1u << 7) | (1u << 10) | ((256u >> 3) << 17) | ((128u >> 4) << 24);
__device__ __forceinline__ void umma_i8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(kIdesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool on) {   // off: zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(on ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ double2 ld_cluster(uint32_t addr, uint32_t rank) {
    double2 v;
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(ra) : "memory");
    return v;
}
__device__ __forceinline__ uint4 lds128v(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts64(uint32_t addr, uint32_t a, uint32_t b) {
    asm volatile("st.shared.v2.u32 [%0], {%1,%2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
// 2^e as a double, -1022 <= e <= 1023
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }
// signed byte I of a word of eight-bit integers -> double; W4: 127 stands for 128
template <int WB, int I>
__device__ __forceinline__ double byte_value(uint32_t biased) {   // each byte + 128
    uint32_t u = prmt(biased, 0u, 0x4440u | I);
    if constexpr (WB == 4) u += (u + 1u) >> 8;
    return __hiloint2double(0x43300000, (int)u) - (4503599627370496.0 + 128.0);
}
// V = c sum_i d_i 256^i, c a power of two (or NaN): two 64-bit halves, exact as doubles, and one rounding
__device__ __forceinline__ double combine(const uint32_t* u, double c) {
    int d[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) d[i] = (int)u[i];
    const long long lo = (long long)(d[3] * 256 + d[2]) * 65536 + (long long)(d[1] * 256 + d[0]);
    const long long hi = (long long)(d[7] * 256 + d[6]) * 65536 + (long long)(d[5] * 256 + d[4]);
    // |lo|, |hi| < 2^46: 1.5 * 2^52 plus the integer
    const double l = __longlong_as_double(lo + 0x4338000000000000ll) - 6755399441055744.0;
    const double h = __longlong_as_double(hi + 0x4338000000000000ll) - 6755399441055744.0;
    const double c32 = __hiloint2double(__double2hiint(c) + (32 << 20), 0);   // (c NaN: the other product is)
    return fma(h, c32, l * c);
}

// The CTA's rows in float64, as solve_ref_kernel has them. H = the lower triangle of G and half its diagonal goes as operand fragments to the start of `room`; the
// triangle's own room is used again behind. A call of its own: its registers are not the other roles'.
template <int WB, int G>
__device__ __noinline__ void solve_wide(const float* w, const uint8_t* codes, const uint8_t* meta, double lambda, uint16_t* coef, double* c_out, int n_out, int k_in,
                                        unsigned char* base, int j, int rt_lo, int rt_hi) {
    constexpr int NB = G / 8;
    const double* tri = reinterpret_cast<const double*>(base + Smem<WB, G>::kTriOff);
    double* room = reinterpret_cast<double*>(base);
    const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31, lr = lane >> 2, lc = lane & 3;
    for (int ib = warp; ib < NB; ib += kThreads / 32)
        for (int s = 0; s < 2 * (ib + 1); ++s) {
            const int l = (s & 1) * 4 + lc;
            const double g = tri[(ib * (ib + 1) / 2 + (s >> 1)) * kBlkStride + lr * kBlkRow + l];
            room[(ib * (ib + 1) + s) * 32 + lane] = s >> 1 < ib || l < lr ? g : l == lr ? 0.5 * g : 0.0;
        }
    __syncthreads();
    if (warp < quant::kRefWarps)
        quant::solve_rows<WB, NB, false>(room, reinterpret_cast<float*>(room + quant::RefSmem<NB>::kFrags * 32), w, codes, meta, 0, lambda, coef, c_out, n_out, k_in, j, rt_lo,
                                         rt_hi);
}

template <int WB, int G>
__global__ void __launch_bounds__(kThreads, 1)
solve_ref_tc_kernel(const Params p, const __grid_constant__ CUtensorMap w_map) {
    using GR = Gram<G>;
    using SM = Smem<WB, G>;
    constexpr int NB = GR::kNB, kStride = GR::kStride, kPasses = G / kPassK, kBuf = buffers<WB, G>(), kTiles = tiles_per_buffer<WB>();
    constexpr int emax = (1 << (WB - 1)) - 1;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // (the offset is the same in every CTA of a cluster: distributed shared memory is addressed by it)
    unsigned char* base = smem_raw + ((1024u - (s32(smem_raw) & 1023u)) & 1023u);
    float* stage = reinterpret_cast<float*>(base);
    double* tri = reinterpret_cast<double*>(base + SM::kTriOff);
    __shared__ uint64_t a_full[2], a_empty[2], w_full[kWStages], w_empty[kWStages], tm_full[2], tm_empty[2], sums_full, sums_empty;
    __shared__ double scale[G];           // 2^(-s_k - 2 emax)
    __shared__ double sums[7][kRows];     // of the three groups of warps that do not solve: b1.V_1 and w.V_1 twice, b1.V_2, b2.V_2, w.V_2
    __shared__ uint2 flip_bytes[64];      // 0xFF where b2 takes the opposite sign
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    __shared__ int wide;   // wide: a row of G has an element more than 2^10 times its diagonal one

    const int tid = threadIdx.x, warp = __shfl_sync(kFull, tid >> 5, 0), lane = tid & 31, lr = lane >> 2, lc = lane & 3;
    const int j = (int)blockIdx.x / p.c, rank = (int)blockIdx.x - j * p.c, nj = p.k_in / G;

    if (tid == 0) {
        abort_flag = 0; wide = 0;
        for (int i = 0; i < 2; ++i) {
            mbar_init(&a_full[i], kDecWarps); mbar_init(&a_empty[i], kEpiWarps);
            mbar_init(&tm_full[i], 1); mbar_init(&tm_empty[i], kEpiWarps / 2);
        }
        mbar_init(&sums_full, 12); mbar_init(&sums_empty, 4);
        for (int i = 0; i < kWStages; ++i) { mbar_init(&w_full[i], 1); mbar_init(&w_empty[i], kEpiWarps / 2); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 64) {
        const uint32_t f = flip_mask((uint32_t)tid);
        uint32_t a = 0, b = 0;
        for (int i = 0; i < 4; ++i) { a |= ((f >> i) & 1u) * (0xFFu << (8 * i)); b |= ((f >> (4 + i)) & 1u) * (0xFFu << (8 * i)); }
        flip_bytes[tid] = make_uint2(a, b);
    }
    if (warp == kMmaWarp) tmem_alloc<512>(&tmem_slot);

    const int t_lo = (int)((long long)p.tiles * rank / p.c), t_hi = (int)((long long)p.tiles * (rank + 1) / p.c), my_tiles = t_hi - t_lo;
    for (int i = tid; i < kRows * (G / 32 + 1); i += kThreads) {   // the first tile's codes and weights on their way while G is formed
        const int r = i / (G / 32 + 1), q = i - r * (G / 32 + 1), row = t_lo * kRows + r;
        if (row < p.n_out) {
            const size_t o = (size_t)row * p.k_in + (size_t)j * G;
            const void* at = q < G / 32 ? (const void*)(p.w + o + q * 32) : (const void*)(p.codes + o);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(at));
        }
    }

    // ---- this CTA's blocks of G's lower triangle (block rows one after another) ----
    const int blk_lo = GR::kBlocks * rank / p.c, blk_hi = GR::kBlocks * (rank + 1) / p.c;
    auto form = [&](auto most) {
        constexpr int kMax = decltype(most)::value;   // blocks of a warp
        const float* xj = p.xc + (size_t)j * G;
        const int first = warp < 16 ? blk_lo + (blk_hi - blk_lo) * warp / 16 : 0, n = warp < 16 ? blk_lo + (blk_hi - blk_lo) * (warp + 1) / 16 - first : 0;
        int at_a[kMax], at_b[kMax];   // first channels of the blocks' rows and columns
        {
            int ib = 0, jb = first;
            while (jb > ib) { jb -= ib + 1; ++ib; }
#pragma unroll
            for (int i = 0; i < kMax; ++i) {
                at_a[i] = ib * 8; at_b[i] = jb * 8;   // (a warp with fewer repeats its last)
                if (i + 1 < n && ++jb > ib) { jb = 0; ++ib; }
            }
        }
        double acc[kMax][2];
#pragma unroll
        for (int i = 0; i < kMax; ++i) acc[i][0] = acc[i][1] = 0.0;
        const int chunks = (p.m + kChunk - 1) / kChunk;
        auto fetch = [&](int c) {
            float* dst = stage + (c & 1) * kChunk * kStride;
            for (int i = tid; i < kChunk * (G / 4); i += kThreads) {
                const int o = i / (G / 4), q = i - o * (G / 4), obs = c * kChunk + o;
                cp_async16(s32(dst + o * kStride + q * 4), xj + (size_t)(obs < p.m ? obs : 0) * p.k_in + q * 4, obs < p.m);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        fetch(0);
        for (int c = 0; c < chunks; ++c) {
            if (c + 1 < chunks) {
                fetch(c + 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            if (n > 0) {
                const float* x0 = stage + (c & 1) * kChunk * kStride + lc * kStride + lr;
                const int steps = (min(kChunk, p.m - c * kChunk) + 3) / 4;   // (the staged rows past the last observation are zeros)
#pragma unroll 4
                for (int s = 0; s < steps; ++s) {
                    const float* xs = x0 + s * 4 * kStride;
#pragma unroll
                    for (int i = 0; i < kMax; ++i)
                        if (i < n) quant::dmma(acc[i], (double)xs[at_a[i]], (double)xs[at_b[i]]);
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int i = 0; i < kMax; ++i)
            if (i < n) {
                double* d = tri + (first + i) * kBlkStride + lr * kBlkRow + 2 * lc;
                d[0] = acc[i][0]; d[1] = acc[i][1];
            }
    };
    constexpr int kMost = (GR::kBlocks + 15) / 16;
    if (kMost > 3 && blk_hi - blk_lo > 80) form(std::integral_constant<int, kMost>{});
    else if (kMost > 3 && blk_hi - blk_lo > 48) form(std::integral_constant<int, 5>{});
    else form(std::integral_constant<int, 3>{});
    if (p.c > 1) {
        cluster_sync();
        constexpr int kWords = GR::kBlocks * (kBlkStride / 2), kLoads = 8;   // 16 bytes each; eight of a thread's in flight
        for (int i0 = tid; i0 < kWords; i0 += kThreads * kLoads) {
            double2 v[kLoads];
            bool other[kLoads];
#pragma unroll
            for (int q = 0; q < kLoads; ++q) {
                const int i = i0 + q * kThreads, b = i / (kBlkStride / 2);
                other[q] = i < kWords && (b < blk_lo || b >= blk_hi);
                if (!other[q]) continue;
                int owner = b * p.c / GR::kBlocks;   // floor: the owner or the one before
                if (GR::kBlocks * (owner + 1) / p.c <= b) ++owner;
                v[q] = ld_cluster(s32(tri) + (uint32_t)i * 16u, (uint32_t)owner);
            }
#pragma unroll
            for (int q = 0; q < kLoads; ++q)
                if (other[q]) reinterpret_cast<double2*>(tri)[i0 + q * kThreads] = v[q];
        }
        cluster_sync();   // nobody reuses its blocks before the others have them
    }
    __syncthreads();
    // ---- digits: four threads a row of G, every fourth block each ----
    if (tid < 4 * G) {
        const int k = tid >> 2, q = tid & 3, kb = k >> 3;
        double el[G / 32][8], big = 0.0;
        bool bad = false;
#pragma unroll
        for (int i = 0; i < G / 32; ++i) {
            const int lb = i * 4 + q;
            const double* from = lb <= kb ? tri + (kb * (kb + 1) / 2 + lb) * kBlkStride + (k & 7) * kBlkRow : tri + (lb * (lb + 1) / 2 + kb) * kBlkStride + (k & 7);
            const int step = lb <= kb ? 1 : kBlkRow;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                el[i][t] = from[t * step];
                const double a = fabs(el[i][t]);
                if (!(a <= 1.7976931348623157e308)) bad = true;
                else if (a > big) big = a;
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            big = fmax(big, __shfl_xor_sync(kFull, big, o));
            bad = __shfl_xor_sync(kFull, (int)bad, o) || bad;
        }
        const int e = big == 0.0 ? 61 : (int)((__double2hiint(big) >> 20) & 2047) - 1023;   // (sums of squares of fp32 numbers: never subnormal)
        const double up = pow2(61 - e);   // |G_kl| 2^(61 - e) < 2^62
        if (big > 1024.0 * tri[(kb * (kb + 1) / 2 + kb) * kBlkStride + (k & 7) * (kBlkRow + 1)] && !bad) wide = 1;
        if (q == 0) scale[k] = bad ? __longlong_as_double(0x7FF8000000000000ll) : pow2(e - 61 - 2 * emax);
        const uint32_t row0 = s32(base) + (uint32_t)k * (kDigits * 128);
#pragma unroll
        for (int i = 0; i < G / 32; ++i) {   // eight elements at a time
            const uint32_t piece = (uint32_t)(2 * i + (q >> 1)), half = (uint32_t)(q & 1) * 8u;
            uint32_t lo[8], hi[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const double a = bad ? 0.0 : el[i][t] * up;
                // v = sum d_s 256^s with signed digits: the bytes of v + 0x8080..80, each less 128
                const unsigned long long v = (unsigned long long)(__double2ll_rn(a) + 0x80808080808080ll) + 0x8000000000000000ull;
                lo[t] = (uint32_t)v ^ 0x80808080u; hi[t] = (uint32_t)(v >> 32) ^ 0x80808080u;
            }
#pragma unroll
            for (int s = 0; s < 8; ++s) {
                const uint32_t* w = s < 4 ? lo : hi;
                const uint32_t sel = (uint32_t)((s & 3) | (((s & 3) + 4) << 4));
                const uint32_t a = prmt(prmt(w[0], w[1], sel), prmt(w[2], w[3], sel), 0x5410u), b = prmt(prmt(w[4], w[5], sel), prmt(w[6], w[7], sel), 0x5410u);
                sts64(row0 + (uint32_t)s * 128 + ((piece ^ (uint32_t)s) << 4) + half, a, b);
            }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // digits -> tensor-core reads; the triangle's room -> TMA writes
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_slot;
    if (wide) {   // (all CTAs of the cluster have the same G and find the same)
        solve_wide<WB, G>(p.w, p.codes, p.meta, p.lambda, p.coef, p.c_out, p.n_out, p.k_in, base, j, t_lo * (kRows / 8),
                          min(t_hi * (kRows / 8), (p.n_out + 7) / 8));
        if (warp == kMmaWarp) {
            __syncwarp();
            tmem_dealloc<512>(tmem_base);
        }
        return;
    }
    const uint32_t a_base = s32(base + SM::kA), w_base = s32(base + SM::kW);

    if (warp == kWWarp) {
        if (lane == 0) {
            bool ok = true;
            int i = 0, s = 0;
            for (int t = 0; t < my_tiles && ok; ++t)
                for (int kc = 0; kc < G / kWK; ++kc, ++i) {
                    if (i >= kWStages) ok = mbar_wait(&w_empty[s], (i / kWStages - 1) & 1, &abort_flag, p.spin);
                    if (!ok) break;
                    mbar_expect_tx(&w_full[s], kWBytes);   // (rows past the last arrive as zeros)
                    tma_load_2d(base + SM::kW + s * kWBytes, &w_map, j * G + kc * kWK, (t_lo + t) * kRows, &w_full[s]);
                    if (++s == kWStages) s = 0;
                }
        }
    } else if (warp == kMmaWarp) {
        if (lane == 0) {
            const uint64_t bdesc0 = smem_desc_sw128(s32(base)), adesc0 = smem_desc_sw128(a_base);
            bool ok = true;
            int i = 0;
            for (int t = 0; t < my_tiles && ok; ++t) {
                const int buf = t % kBuf;
                ok = mbar_wait(&a_full[buf], (t / kBuf) & 1, &abort_flag, p.spin);
                for (int kc = 0; kc < kPasses && ok; ++kc, ++i)
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        if (i > 0) ok = ok && mbar_wait(&tm_empty[v], (i - 1) & 1, &abort_flag, p.spin);
                        if (!ok) break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint64_t bd = bdesc0 + (uint32_t)(kc * (256 * 128 >> 4)), ad = adesc0 + (uint32_t)((buf * kTiles + v) * (kTileBytes >> 4));
#pragma unroll
                        for (int ks = 0; ks < G / 32; ++ks) {
                            umma_i8(tmem_base + v * 256, ad + 2 * ks, bd + 2 * ks, ks > 0 ? 1u : 0u);
                            if constexpr (WB == 4) umma_i8(tmem_base + v * 256, ad + 2 * (kTileBytes >> 4) + 2 * ks, bd + 2 * ks, 1u);
                        }
                        umma_commit(&tm_full[v]);
                    }
            }
        }
    } else if (warp >= kDec0) {
        // ------------------------------ codes and records -> int8 operands ------------------------------
        const int dt = tid - kDec0 * 32;
        constexpr int kPerTile = kRows * NB / (kDecWarps * 32), kPer = kPerTile < 8 ? kPerTile : 8;   // micro-blocks of a thread; in flight
        const bool codes8 = (reinterpret_cast<uintptr_t>(p.codes) & 7u) == 0;
        // 2^emax b1 by code: W3 8 4 2 0 -8 -4 -2 -1;  W2 2 0 -2 -1;  W4 64 (see below) 64 32 .. by e and sign
        bool ok = true;
        for (int t = 0; t < my_tiles; ++t) {
            const int buf = t % kBuf;
            const uint32_t at = a_base + (uint32_t)(buf * kTiles * kTileBytes);
#pragma unroll 1
            for (int i0 = 0; i0 < kPerTile && ok; i0 += kPer) {
            uint2 cw[kPer];
            uint32_t rec[kPer];
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int u = dt + (i0 + i) * kDecWarps * 32, r = u / NB, mb = u - r * NB, row = (t_lo + t) * kRows + r;
                cw[i] = make_uint2(0u, 0u); rec[i] = 64u;
                if (row < p.n_out) {
                    const size_t o = (size_t)row * p.k_in + (size_t)j * G + mb * 8;
                    if (codes8) cw[i] = *reinterpret_cast<const uint2*>(p.codes + o);
                    else {
                        const uint8_t* c = p.codes + o;
                        cw[i].x = c[0] | (c[1] << 8) | (c[2] << 16) | ((uint32_t)c[3] << 24);
                        cw[i].y = c[4] | (c[5] << 8) | (c[6] << 16) | ((uint32_t)c[7] << 24);
                    }
                    rec[i] = p.meta[o / 8] & 63u;
                }
            }
            if (i0 == 0 && t >= kBuf) ok = __all_sync(kFull, mbar_wait(&a_empty[buf], (t / kBuf - 1) & 1, &abort_flag, p.spin));
            if (!ok) break;
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int u = dt + (i0 + i) * kDecWarps * 32, r = u / NB, mb = u - r * NB;
                const uint32_t dst = at + (uint32_t)(r * 128 + (((mb >> 1) ^ (r & 7)) << 4) + (mb & 1) * 8);
                const uint32_t none = rec[i] == 64u ? 0u : 0xFFFFFFFFu;   // rows past the last: zeros
                auto selector = [](uint32_t c) { c &= 0x07070707u; c |= c >> 4; return prmt(c, 0u, 0x4420u); };   // four bytes -> four nibbles
                const uint32_t sa = selector(cw[i].x), sb = selector(cw[i].y);
                const uint32_t s = (rec[i] & 3u) + 1u, pa = 0x3210u ^ (s * 0x1111u), pb = 0x7654u ^ (s * 0x1111u);
                const uint2 fl = flip_bytes[rec[i] & 63u];
                if constexpr (WB <= 3) {
                    constexpr uint32_t t0 = WB == 3 ? 0x00020408u : 0xFFFE0002u, t1 = WB == 3 ? 0xFFFEFCF8u : 0u;
                    const uint32_t a = prmt(t0, t1, sa) & none, b = prmt(t0, t1, sb) & none;
                    sts64(dst, a, b);
                    // -q = ~(q - 1) = (q ^ FF) + 1 byte by byte, without a carry between bytes
                    auto negate = [](uint32_t q, uint32_t f) { const uint32_t x = q ^ f; return ((x & 0x7F7F7F7Fu) + (f & 0x01010101u)) ^ (x & 0x80808080u); };
                    sts64(dst + kTileBytes, negate(prmt(a, b, pa), fl.x), negate(prmt(a, b, pb), fl.y));
                } else {
                    // magnitudes 128 64 .. 1 as bytes; zero: code 7. A positive 128 becomes 127 here and 1 in the tile of units.
                    auto sign = [](uint32_t c) { return ((c >> 3) & 0x01010101u) * 0xFFu; };
                    const uint32_t na = sign(cw[i].x), nb = sign(cw[i].y);
                    uint32_t ma = prmt(0x10204080u, 0x01020408u, sa), mb4 = prmt(0x10204080u, 0x01020408u, sb);
                    ma &= (na | ~((ma & 0x01010101u) * 0xFFu)) & none; mb4 &= (nb | ~((mb4 & 0x01010101u) * 0xFFu)) & none;   // (e = 7: +1 is the zero)
                    auto put = [&](uint32_t to, uint32_t m0, uint32_t m1, uint32_t n0, uint32_t n1) {
                        uint32_t v[2], c[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint32_t m = h ? m1 : m0, n = h ? n1 : n0;
                            const uint32_t top = (m >> 7) & 0x01010101u & ~n;         // +128
                            c[h] = top;
                            const uint32_t q = m - top, x = q ^ n;                    // (no borrow: top only where the byte is 128)
                            v[h] = ((x & 0x7F7F7F7Fu) + (n & 0x01010101u)) ^ (x & 0x80808080u);
                        }
                        sts64(to, v[0], v[1]);
                        sts64(to + 2 * kTileBytes, c[0], c[1]);
                    };
                    put(dst, ma, mb4, na, nb);
                    put(dst + kTileBytes, prmt(ma, mb4, pa), prmt(ma, mb4, pb), prmt(na, nb, pa) ^ fl.x, prmt(na, nb, pb) ^ fl.y);
                }
            }
            }
            if (!ok) break;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&a_full[buf]);
        }
    } else {
        // ------------------------------ V_1 and V_2: a thread is a row, a warp 16 of a pass's 32 elements ------------------------------
        auto work = [&](auto second) {
            constexpr bool SECOND = decltype(second)::value;
            constexpr int v = SECOND ? 1 : 0;
            const int r = (warp & 3) * 32 + lane, half = warp >> 3;
            const uint32_t ta = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(v * 256 + half * 128), flip = (uint32_t)(r & 7);
            int i = 0, ws = half;   // the half's stages of w: every second
            uint32_t w_par = 0;
            for (int t = 0; t < my_tiles; ++t) {
                const int buf = t % kBuf;
                bool ok = __all_sync(kFull, mbar_wait(&a_full[buf], (t / kBuf) & 1, &abort_flag, p.spin));
                if (!ok) return;
                const uint32_t row1 = a_base + (uint32_t)(buf * kTiles * kTileBytes + r * 128);
                double t1 = 0.0, t2 = 0.0, tw = 0.0;   // b1.V, b2.V (V_2 only), w.V
#pragma unroll 1
                for (int kc = 0; kc < kPasses; ++kc, ++i) {
                    const uint32_t piece = ((uint32_t)(kc * 2 + half) ^ flip) << 4;
                    const uint4 q1 = lds128v(row1 + piece), q2 = SECOND ? lds128v(row1 + kTileBytes + piece) : make_uint4(0u, 0u, 0u, 0u);
                    ok = __all_sync(kFull, mbar_wait(&w_full[ws], w_par, &abort_flag, p.spin) && mbar_wait(&tm_full[v], i & 1, &abort_flag, p.spin));
                    if (!ok) return;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t wrow = w_base + (uint32_t)(ws * kWBytes + r * 64);
                    const uint32_t b1w[4] = {q1.x ^ 0x80808080u, q1.y ^ 0x80808080u, q1.z ^ 0x80808080u, q1.w ^ 0x80808080u};
                    const uint32_t b2w[4] = {q2.x ^ 0x80808080u, q2.y ^ 0x80808080u, q2.z ^ 0x80808080u, q2.w ^ 0x80808080u};
                    double s1[2] = {0.0, 0.0}, s2[2] = {0.0, 0.0}, sw[2] = {0.0, 0.0};   // this pass's even and odd elements: short sums round less
#pragma unroll
                    for (int g4 = 0; g4 < 4; ++g4) {   // four elements
                        uint32_t d[32];
                        tmem_ld32(ta + (uint32_t)g4 * 32u, d);
                        const uint4 wq = lds128v(wrow + (((uint32_t)g4 ^ ((uint32_t)(r >> 1) & 3u)) << 4));
                        const float w4[4] = {__uint_as_float(wq.x), __uint_as_float(wq.y), __uint_as_float(wq.z), __uint_as_float(wq.w)};
                        const double b1v[4] = {byte_value<WB, 0>(b1w[g4]), byte_value<WB, 1>(b1w[g4]), byte_value<WB, 2>(b1w[g4]), byte_value<WB, 3>(b1w[g4])};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const double val = combine(d + 8 * e, scale[kc * kPassK + half * 16 + g4 * 4 + e]);
                            s1[e & 1] = fma(b1v[e], val, s1[e & 1]);
                            if constexpr (SECOND) {
                                const double b2v = e == 0 ? byte_value<WB, 0>(b2w[g4]) : e == 1 ? byte_value<WB, 1>(b2w[g4]) : e == 2 ? byte_value<WB, 2>(b2w[g4]) : byte_value<WB, 3>(b2w[g4]);
                                s2[e & 1] = fma(b2v, val, s2[e & 1]);
                            }
                            sw[e & 1] = fma((double)w4[e], val, sw[e & 1]);
                        }
                    }
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) { mbar_arrive(&tm_empty[v]); mbar_arrive(&w_empty[ws]); }
                    ws += 2;
                    if (ws >= kWStages) { ws -= kWStages; w_par ^= 1u; }
                    t1 += s1[0] + s1[1]; t2 += s2[0] + s2[1]; tw += sw[0] + sw[1];
                }
                if (lane == 0) mbar_arrive(&a_empty[buf]);
                if (!SECOND || half == 0) {
                    if (t > 0) ok = __all_sync(kFull, mbar_wait(&sums_empty, (t - 1) & 1, &abort_flag, p.spin));
                    if (!ok) return;
                    double (*to)[kRows] = sums + (SECOND ? 4 : 2 * half);
                    to[0][r] = t1;
                    if constexpr (SECOND) { to[1][r] = t2; to[2][r] = tw; }
                    else to[1][r] = tw;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sums_full);
                } else {
                    ok = __all_sync(kFull, mbar_wait(&sums_full, t & 1, &abort_flag, p.spin));
                    if (!ok) return;
                    const double up = pow2(emax);   // w carries no 2^emax
                    const double a = (sums[0][r] + sums[2][r]) + p.lambda, r1 = (sums[1][r] + sums[3][r]) * up;
                    const double g12 = sums[4][r] + t1, dd = (sums[5][r] + t2) + p.lambda, r2 = (sums[6][r] + tw) * up;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sums_empty);
                    const double det = a * dd - g12 * g12, c1 = (dd * r1 - g12 * r2) / det, c2 = (a * r2 - g12 * r1) / det;
                    const int row = (t_lo + t) * kRows + r;
                    if (row < p.n_out) {
                        const size_t o = ((size_t)row * nj + j) * 2;
                        p.coef[o] = __half_as_ushort(__double2half(c1));
                        p.coef[o + 1] = __half_as_ushort(__double2half(c2));
                        if (p.c_out) { p.c_out[o] = c1; p.c_out[o + 1] = c2; }
                    }
                }
            }
        };
        if (((warp >> 2) & 1) == 0) work(std::integral_constant<bool, false>{});
        else work(std::integral_constant<bool, true>{});
    }
    __syncthreads();
    if (abort_flag) {   // there is no status word: NaN for the CTA's rows
        settle_after_give_up();
        for (int r = t_lo * kRows + tid; r < t_hi * kRows && r < p.n_out; r += kThreads) {
            const size_t o = ((size_t)r * nj + j) * 2;
            p.coef[o] = p.coef[o + 1] = 0x7E00u;
            if (p.c_out) p.c_out[o] = p.c_out[o + 1] = __longlong_as_double(0x7FF8000000000000ll);
        }
    }
    if (warp == kMmaWarp) {
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tmem_dealloc<512>(tmem_base);
    }
}

template <int WB, int G>
static cudaError_t launch(const Geometry& g, Params& p, const CUtensorMap& w_map, cudaStream_t st) {
    constexpr size_t smem = Smem<WB, G>::kBytes;
    static_assert(smem + sizeof(double) * (G + 7 * kRows) + 64 * 8 + 256 <= 227 * 1024, "shared memory");
    static SmemAttrCache cache;
    if (cudaError_t e = ensure_dynamic_smem(solve_ref_tc_kernel<WB, G>, smem, cache)) return e;
    const int sms = sm_count();
    // CTAs of a column: the split whose waves cost least, in clocks: forming G (16 per product and scheduler), its exchange and digits, and the
    // tiles of the CTA that has most
    const int cols = g.k_in / G;
    double best = 0.0;
    for (int c = 1; c <= 8 && c <= p.tiles; c *= 2) {
        // clusters that were seen to run at once (a cluster lies in one group of SMs): 12 of eight CTAs did, 16 took two waves (1024 x 512 in groups of 32 at 32
        // observations 18 us; 512 rows, as clusters of four, 9.6)
        const int at_once = c == 8 ? sms / 12 : c == 4 ? sms * 8 / 37 : sms / c;
        const double waves = (double)((cols + at_once - 1) / at_once);
        const double cost = waves * (4.0 * Gram<G>::kBlocks / c * ((p.m + 3) / 4) + 8000.0 + (c > 1 ? 2500.0 : 0.0) + (double)((p.tiles + c - 1) / c) * (40.0 * G + 800.0));
        if (c == 1 || cost < best) { best = cost; p.c = c; }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cols * p.c));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)p.c; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, solve_ref_tc_kernel<WB, G>, p, w_map);
}
template <int WB>
static cudaError_t launch_group(const Geometry& g, Params& p, const CUtensorMap& w_map, cudaStream_t st) {
    return g.group == 128 ? launch<WB, 128>(g, p, w_map, st) : g.group == 64 ? launch<WB, 64>(g, p, w_map, st) : launch<WB, 32>(g, p, w_map, st);
}

}  // namespace reftc

bool solve_ref_tc_supported(const Geometry& g, const float* w, const float* x_calib, int m) {
    // Half as many observations as a group has channels: the observations one by one are as cheap and need no Gram matrix.
    if (g.group < 32 || 2 * m <= g.group || ((reinterpret_cast<uintptr_t>(w) | reinterpret_cast<uintptr_t>(x_calib)) & 15u) != 0) return false;
    // Few columns and few observations: solve_ref_kernel splits a column's rows over more CTAs than a cluster has, and G is cheap for either. Where the line
    // lies was measured at 592 sizes (512 to 8192 wide and high, 32 to 512 observations); us, solve_ref_kernel / this:
    const int cols = g.k_in / g.group, n = g.n_out, tiles = (n + reftc::kRows - 1) / reftc::kRows;
    // 600 x 768 at 100 observations 11.3 / 13.0, 1281 x 768 15.0 / 15.5, 512 x 1024 at 32 9.4 / 10.6, 64 x 4096 at 100 9.6 / 10.3; 512 x 1536 at 128 and 4096 x 1024 faster here
    if (g.group == 32) return cols > 24 && (m > 128 || (n > 128 && (cols > 32 || m > 32)));
    // 1500 x 512 W4 at 128 19.5 / 24.9, 6000 x 512 W4 45.1 / 46.5, 1281 x 640 at 100 19.2 / 21.5; 3000 x 640 41.3 / 26.0, 1281 x 768 at 200 28.4 / 24.9
    if (g.group == 64) return cols > 16 || m > 128 || (n > 2048 && g.wbits < 4);
    // in groups of 128 only where a cluster's CTAs get uneven shares or a few columns have many tiles: 600 x 640 at 100 35.2 / 36.9, 1500 x 512 W4 40.6 / 46.1, 8192 x 512 92 / 93
    return m > 128 || !((cols <= 6 && tiles > 4 && tiles < 8) || (cols <= 4 && tiles > 8));
}
cudaError_t launch_solve_ref_tc(const Geometry& g, const float* w, const uint8_t* codes, const uint8_t* meta, const float* x_calib, int m,
                                double lambda, uint16_t* coef, double* c_out, int spin_limit, cudaStream_t st) {
    CUtensorMap w_map;
    if (cudaError_t e = tc::encode_f32_map(&w_map, w, g.k_in, g.n_out, reftc::kWK, reftc::kRows)) return e;
    reftc::Params p;
    p.codes = codes; p.meta = meta; p.xc = x_calib; p.w = w; p.coef = coef; p.c_out = c_out; p.lambda = lambda;
    p.n_out = g.n_out; p.k_in = g.k_in; p.m = m; p.tiles = (g.n_out + reftc::kRows - 1) / reftc::kRows; p.c = 1;
    p.spin = spin_limit > 0 ? spin_limit : tc::kSpin;
    return g.wbits == 4 ? reftc::launch_group<4>(g, p, w_map, st) : g.wbits == 3 ? reftc::launch_group<3>(g, p, w_map, st)
                                                                               : reftc::launch_group<2>(g, p, w_map, st);
}

}  // namespace goq
