// C ABI of libgoq: argument checks on the host, then one launcher per call.
#include <atomic>
#include <cstdlib>
#include <vector>
#include "goq_common.cuh"
#include "goq_internal.h"

using goq::Geometry;

namespace {

std::atomic<int> g_gemv_variant{0};
std::atomic<int> g_wait_limit{0};   // 0: the kernels' own bound on device-side waits
constexpr int kGemmExactMaxTokens = 32;     // goq_gemm: fp32-accurate results up to here
constexpr int kGemmMidMaxTokens = 256;      // ... one token tile of the mid-batch kernel

bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// compute capability 10.x of the current device, cached per device index
goq_status check_arch() {
    static std::atomic<int> cached[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return GOQ_ERR_CUDA;
    if (dev >= 0 && dev < 64) {
        int c = cached[dev].load(std::memory_order_relaxed);
        if (c == 1) return GOQ_OK;
        if (c == 2) return GOQ_ERR_ARCH;
    }
    int major = 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return GOQ_ERR_CUDA;
    const bool ok = (major == 10);
    if (dev >= 0 && dev < 64) cached[dev].store(ok ? 1 : 2, std::memory_order_relaxed);
    return ok ? GOQ_OK : GOQ_ERR_ARCH;
}

// Estimated times of the other kernels for a few tokens, us (W3 g128, W4; the kernels in e4m3 operands have gemm_f8_us). One decode launch of up to
// 16 tokens: measured 5.2 for 2048 x 2048, 8.2 4096 x 4096, 19.1 11008 x 4096, 27.4 8192 x 8192, 83 28672 x 8192 at 16 tokens, 22 and 66 for the last two at 8.
float decode_us(const Geometry& g, int m) {
    return 4.f + (float)g.n_units * ((m > 8 ? 7.0e-4f : 5.5e-4f) + (g.wbits == 4 ? 1.0e-4f : 0.f));
}
// The mid-batch kernel up to 256 tokens: 34.6 for 8192 x 8192, 21 4096 x 4096, 18.5 2048 x 2048, 23 1024 x 8192 at 64 tokens, 39.5 and 23 for the first two at 128;
// with at most one unit for every SM 10.2 for 1024 x 512, 13.2 1024 x 2048, 15.9 512 x 4096 at 40.
float mid_us(const Geometry& g, int m, bool exact) {
    const int tiles = (g.n_tiles + 7) / 8, units = tiles * g.k_blocks, sms = goq::gemm_mid_ctas(), grid = units < sms ? units : sms;
    const float unit = (exact ? 0.8f : 0.55f + 0.0032f * (float)m) + (g.wbits == 4 ? 0.08f : 0.f) + (g.group < 128 ? 0.03f : 0.f);
    const float parts = (float)grid / (float)tiles;
    return units <= sms ? 9.5f + 0.17f * parts + unit : 13.f + 0.4f * parts + unit * (float)((units + grid - 1) / grid);
}
// goq_gemv on the kernel in e4m3 operands: above 4 tokens (or W4, which has no integer form), large linears only; W2 and W3 where a call needs scratch anyway
bool gemv_takes_f8(const Geometry& g, int m) {
    return (g.wbits == 4 || (m > 4 && goq::gemv_stream_supported(g))) && goq::gemm_f8_supported(g, m) && goq::gemm_f8_us(g, m) <= 0.97f * decode_us(g, m);
}

std::atomic<int> g_last_cuda_error{0};
goq_status from_cuda(cudaError_t e) { return goq::status_from_cuda(e); }

}  // namespace

namespace goq {
goq_status status_from_cuda(cudaError_t e) {
    if (e == cudaSuccess) return GOQ_OK;
    (void)cudaGetLastError();  // do not leave a non-sticky error behind for the next call to trip over
    g_last_cuda_error.store((int)e, std::memory_order_relaxed);
    return GOQ_ERR_CUDA;
}
}  // namespace goq

extern "C" {

const char* goq_status_string(goq_status s) {
    switch (s) {
        case GOQ_OK: return "ok";
        case GOQ_ERR_INVALID_ARG: return "invalid argument";
        case GOQ_ERR_UNSUPPORTED: return "unsupported configuration";
        case GOQ_ERR_ALIGNMENT: return "misaligned pointer";
        case GOQ_ERR_WORKSPACE: return "buffer too small";
        case GOQ_ERR_OVERFLOW_BOUND: return "int32 accumulator bound exceeded";
        case GOQ_ERR_ARCH: return "device is not sm_100";
        case GOQ_ERR_CUDA: return "CUDA runtime error";
        case GOQ_ERR_TIMEOUT: return "device-side wait timed out";
    }
    return "unknown status";
}

size_t goq_packed_bytes(const goq_desc* desc) {
    Geometry g;
    return goq::make_geometry(desc, &g) ? g.total_bytes : 0;
}

size_t goq_algorithmic_bytes(const goq_desc* desc) {
    Geometry g;
    if (!goq::make_geometry(desc, &g)) return 0;
    if (g.k1) return (size_t)g.n_out * g.k_in * g.wbits / 8 + (size_t)g.n_out * (g.k_in / g.group) * 2;   // codes + one fp16 scale
    // (wbits + 0.75) bits per weight = (4*wbits + 3) / 32 bytes
    return (size_t)g.n_out * g.k_in * (4 * g.wbits + 3) / 32 + (size_t)g.n_out * (g.k_in / g.group) * 4;
}

size_t goq_workspace_bytes(const goq_desc* desc, int op, int m) {
    Geometry g;
    if (!goq::make_geometry(desc, &g) || m <= 0) return 0;
    if (op == GOQ_OP_GEMV && m <= 16) {
        size_t need = 0;
        if (goq::gemv_stream_supported(g)) need = goq::gemv_stream_workspace(g);
        if (gemv_takes_f8(g, m)) {   // (with less the call takes another kernel)
            const size_t f8 = goq::gemm_f8_workspace(g, m);
            if (f8 > need) need = f8;
        }
        return need;
    }
    if (op == GOQ_OP_GEMM) {
        // every kernel a call of up to m rows may take, so that a buffer for the largest batch keeps the smaller ones on their kernels
        // (a kernel's own need can fall where m grows: 8192 x 8192 parks 39 MB of partial sums at 256 rows, 22 MB at 257)
        size_t need = 0;
        auto cover = [&](size_t bytes) { if (bytes > need) need = bytes; };
        if (goq::gemm_tc_supported(g)) {
            cover(goq::gemm_tc_workspace(g, m));
            if (m > 256) cover(goq::gemm_tc_workspace(g, 256));   // split-K partial sums, up to 256 rows
        }
        if (goq::gemv_stream_supported(g)) cover(goq::gemv_stream_workspace(g));
        cover(goq::gemm_mid_workspace_upto(g, m));
        cover(goq::gemm_f8_workspace_upto(g, m < kGemmMidMaxTokens ? m : kGemmMidMaxTokens));
        return need;
    }
    return 0;
}

goq_status goq_pack(const goq_desc* desc, const uint8_t* codes, const uint8_t* meta, const uint16_t* coef_f16,
                    void* packed, size_t packed_bytes, void* stream) {
    Geometry g;
    if (!goq::make_geometry(desc, &g) || !codes || !meta || !coef_f16 || !packed) return GOQ_ERR_INVALID_ARG;
    if (!aligned(packed, 128) || !aligned(coef_f16, 2)) return GOQ_ERR_ALIGNMENT;
    if (packed_bytes < g.total_bytes) return GOQ_ERR_WORKSPACE;
    if (goq_status s = check_arch()) return s;
    return from_cuda(goq::launch_pack(g, codes, meta, coef_f16, packed, (cudaStream_t)stream));
}

goq_status goq_unpack(const goq_desc* desc, const void* packed, uint8_t* codes_b1, uint8_t* codes_b2,
                      uint16_t* coef_f16, void* stream) {
    Geometry g;
    if (!goq::make_geometry(desc, &g) || !packed) return GOQ_ERR_INVALID_ARG;
    if (!codes_b1 && !codes_b2 && !coef_f16) return GOQ_ERR_INVALID_ARG;
    if (!aligned(packed, 128) || !aligned(coef_f16, 2)) return GOQ_ERR_ALIGNMENT;
    if (goq_status s = check_arch()) return s;
    return from_cuda(goq::launch_unpack(g, packed, codes_b1, codes_b2, coef_f16, (cudaStream_t)stream));
}

goq_status goq_gemv(const goq_desc* desc, const void* packed, const void* x_bf16, int batch, void* y, int y_dtype,
                    void* ws, size_t ws_bytes, void* stream) {
    Geometry g;
    if (!goq::make_geometry(desc, &g) || !packed || !x_bf16 || !y) return GOQ_ERR_INVALID_ARG;
    if (batch < 1 || batch > 16) return GOQ_ERR_INVALID_ARG;
    if (y_dtype != GOQ_BF16 && y_dtype != GOQ_F32) return GOQ_ERR_INVALID_ARG;
    if (!aligned(packed, 128) || !aligned(x_bf16, 16) || !aligned(y, y_dtype == GOQ_F32 ? 4 : 2))
        return GOQ_ERR_ALIGNMENT;
    if (goq_status s = check_arch()) return s;
    const int variant = g_gemv_variant.load(std::memory_order_relaxed);
    const bool use_stream = goq::gemv_stream_supported(g) && (variant == 0 || variant == 3 || variant == 5);
    if ((variant == 3 || variant == 5) && !use_stream) return GOQ_ERR_UNSUPPORTED;
    if (use_stream) {
        if (!ws || !aligned(ws, 256)) return ws ? GOQ_ERR_ALIGNMENT : GOQ_ERR_WORKSPACE;
        if (ws_bytes < goq::gemv_stream_workspace(g)) return GOQ_ERR_WORKSPACE;
        if (!goq::stream_hash_is_bijective()) return GOQ_ERR_UNSUPPORTED;
        // Up to 4 tokens on a large linear: integer operands, half the decode's instructions; below, the fragment kernel's shorter
        // start and end count for more. Measured, W3 g128, integer over fragment at 1 / 2 / 3 / 4 tokens: 4096 units (1024 x 8192) 1.03 / 1.07 /
        // 1.16 / 1.20, (8192 x 1024) 0.99 / 0.99 / 0.98 / 0.99; 8192 (4096 x 4096) 0.95 / 1.01 / 1.06 / 1.09, (2048 x 8192) 0.91 / 0.98 / 1.10 /
        // 1.16, (8192 x 2048) 0.80 / 0.82 / 0.85 / 0.86; 22016 (11008 x 4096) 0.75 / 0.77 / 0.78 / 0.80, (4096 x 11008) 0.77 / 0.84 / 0.93 / 0.97.
        // W2 and groups of 32 lie within 0.03 of these; single-basis weights, whose integer decode is shorter still, 0.1 to 0.25 below, so
        // that for them the line could lie lower. Between 8192 and 12000 units at 2 to 4 tokens it depends on the width: narrow ones lose.
        const bool one = goq::gemv_one_supported(g, batch) && (variant == 5 || (variant == 0 && g.n_units > (batch == 1 ? 6000u : 12000u)));
        if (variant == 5 && !one) return GOQ_ERR_UNSUPPORTED;
        if (one)
            return from_cuda(goq::launch_gemv_one(g, packed, x_bf16, batch, y, y_dtype, ws, g_wait_limit.load(std::memory_order_relaxed),
                                                  (cudaStream_t)stream));
        if (variant == 3) return from_cuda(goq::launch_gemv_stream(g, packed, x_bf16, batch, y, y_dtype, ws, (cudaStream_t)stream));
    }
    // Large linears above 4 tokens (W4: any number): both bases as e4m3 operands of the tensor cores, half the decode's instructions, for a pre-pass and a
    // summing kernel around it. us, fragment kernel / this: W3 28672 x 8192 66 / 55 at 8 tokens, 83 / 60 at 16; 8192 x 8192 22.0 / 23.0 and 27.4 / 25.0;
    // W4 25.6 / 24.3 at 8 tokens; 4096 x 4096 at 16 tokens 8.1 / 14.2.
    if (variant == 0 && gemv_takes_f8(g, batch) && ws && aligned(ws, 256) && ws_bytes >= goq::gemm_f8_workspace(g, batch))
        return from_cuda(goq::launch_gemm_f8(g, packed, x_bf16, batch, y, y_dtype, ws, g_wait_limit.load(std::memory_order_relaxed), (cudaStream_t)stream));
    if (variant == 0 && goq::gemv_mma_supported(g, batch))
        return from_cuda(goq::launch_gemv_mma(g, packed, x_bf16, batch, y, y_dtype, true, (cudaStream_t)stream));
    bool use_mma = goq::linear_mma_supported(g);
    if (variant == 1) use_mma = false;
    if (variant == 2 && !use_mma) return GOQ_ERR_UNSUPPORTED;
    if (use_mma) return from_cuda(goq::launch_linear_mma(g, packed, x_bf16, batch, y, y_dtype, (cudaStream_t)stream));
    return from_cuda(goq::launch_gemv_scalar(g, packed, x_bf16, batch, y, y_dtype, (cudaStream_t)stream));
}

goq_status goq_gemm(const goq_desc* desc, const void* packed, const void* x, int m, int x_dtype, const float* sx,
                    const int8_t* cq, const float* sc, void* y, int y_dtype, int32_t* acc, void* ws, size_t ws_bytes,
                    void* stream) {
    Geometry g;
    if (!goq::make_geometry(desc, &g) || !packed || !x || m < 1) return GOQ_ERR_INVALID_ARG;
    if (y && y_dtype != GOQ_BF16 && y_dtype != GOQ_F32) return GOQ_ERR_INVALID_ARG;
    if (!aligned(packed, 128) || !aligned(x, 16)) return GOQ_ERR_ALIGNMENT;
    if (y && !aligned(y, y_dtype == GOQ_F32 ? 4 : 2)) return GOQ_ERR_ALIGNMENT;
    if (x_dtype == GOQ_BF16) {
        if (!y) return GOQ_ERR_INVALID_ARG;
        if (goq_status s = check_arch()) return s;
        const int variant = g_gemv_variant.load(std::memory_order_relaxed);
        // Four kernels: the decode GEMV (16 tokens a launch), the kernel in e4m3 operands (a few tokens to about 128, fp32 accuracy, no rounding of
        // weights or activations), the mid-batch kernel (an even split of the packed records over the SMs; up to
        // 32 tokens with both bases as exact operands, above with w_hat rounded once to fp16) and the prefill kernel (128 x 512 tiles).
        //   Up to 32 tokens: groups of 8 and 16 have only the mid-batch kernel that keeps fp32 accuracy. Others take two decode launches
        //   unless the linear is large or wide (units = 16-row tiles x k-blocks). Measured at 17 tokens, W3 g128, us, mid-batch over decode:
        //   4096 x 4096 1.22, 8192 x 2048 0.99, 11008 x 2048 0.91, 4096 x 8192 0.96, 2048 x 11008 1.05, 16000 x 512 1.11, 28672 x 512 0.88.
        //   33 to 256 tokens: mid-batch (0.25 to 0.95 of the prefill kernel's time), except where the channel tiles fill most of one wave of
        //   the prefill kernel and the few k-blocks are soon decoded: at 256 tokens, mid-batch over prefill, 16000 x 256 1.23, x 512
        //   1.25, x 896 1.10, x 2048 1.00; 11008 x 512 1.06; 8192 x 512 (64 tiles, two splits of K) 0.88.
        //   Above: it decodes the weights once per 256 tokens, but spreads any number of tiles evenly; the two kernels' estimates decide
        //   (the prefill kernel's is the surer one, hence the margin). us, mid-batch / prefill: 1024 x 8192 W4 at 777 tokens 35 / 102;
        //   4096 x 4096 at 1024 52 / 54; 11008 x 4096 at 512 69 / 65; 16000 x 512 at 512 40 / 23.
        const bool exact = m <= kGemmExactMaxTokens, narrow = !goq::gemv_mma_supported(g, 16);
        bool mid_wanted = variant == 4, f8_wanted = variant == 6;
        if (variant == 0) {
            if (exact) {
                mid_wanted = narrow || (m > 16 && (g.n_units >= 12000 || (g.n_tiles >= 500 && g.n_units >= 8000) || g.n_tiles >= 1700));
            } else if (m <= kGemmMidMaxTokens) {
                const int wide_tiles = (g.n_tiles + 7) / 8, sms = goq::gemm_mid_ctas();
                mid_wanted = !(goq::gemm_tc_supported(g) && 2 * wide_tiles > sms && wide_tiles <= sms && g.k_blocks >= 2 && g.k_blocks < 8);
            } else {
                mid_wanted = !goq::gemm_tc_supported(g) || goq::gemm_mid_us(g, m) <= 0.95f * goq::gemm_tc_us(g, m);
            }
            //   Up to 256 tokens, groups of 32 and more: e4m3 operands where the estimates say so. us, the others / e4m3: at 32 tokens 4096 x 4096 17.4 / 16.1,
            //   28672 x 8192 98 / 77, 2048 x 2048 9.9 / 11.4, 1024 x 8192 13.6 / 15.5, in groups of 64 8192 x 8192 38 / 41; at 64 (two token tiles) 2048 x 4096
            //   18.4 / 16.0, 2048 x 8192 22.5 / 21.6; at 128 1024 x 3072 20.5 / 15.0, 2048 x 4096 19.9 / 21.1, 7200 x 512 16.2 / 16.4.
            if (m <= 16) f8_wanted = !narrow && gemv_takes_f8(g, m);
            else if (m <= kGemmMidMaxTokens && goq::gemm_f8_supported(g, m)) {
                const int second = m - 16;   // (up to 32 tokens: of the second decode launch)
                f8_wanted = goq::gemm_f8_us(g, m) <= 0.97f * (exact && !mid_wanted ? decode_us(g, 16) + decode_us(g, second) : mid_us(g, m, exact));
            }
        }
        if (f8_wanted && goq::gemm_f8_supported(g, m) && ws && aligned(ws, 256) && ws_bytes >= goq::gemm_f8_workspace(g, m))
            return from_cuda(goq::launch_gemm_f8(g, packed, x, m, y, y_dtype, ws, g_wait_limit.load(std::memory_order_relaxed), (cudaStream_t)stream));
        if (mid_wanted && goq::gemm_mid_supported(g, m, exact) && ws && aligned(ws, 256) && ws_bytes >= goq::gemm_mid_workspace(g, m, exact))
            return from_cuda(goq::launch_gemm_mid(g, packed, x, m, y, y_dtype, ws, exact, g_wait_limit.load(std::memory_order_relaxed), (cudaStream_t)stream));
        if (variant == 4 || variant == 6) return GOQ_ERR_UNSUPPORTED;
        // the decode GEMV, 16 tokens per launch
        if (exact && variant == 0 && goq::gemv_mma_supported(g, 16)) {
            if (goq::gemv_stream_supported(g)) {
                if (!ws || !aligned(ws, 256)) return ws ? GOQ_ERR_ALIGNMENT : GOQ_ERR_WORKSPACE;
                if (ws_bytes < goq::gemv_stream_workspace(g)) return GOQ_ERR_WORKSPACE;
                if (!goq::stream_hash_is_bijective()) return GOQ_ERR_UNSUPPORTED;
            }
            const size_t ybytes = (y_dtype == GOQ_F32) ? 4 : 2;
            for (int t0 = 0; t0 < m; t0 += 16) {
                const int nb = (m - t0 < 16) ? (m - t0) : 16;
                cudaError_t e = goq::launch_gemv_mma(g, packed, (const uint16_t*)x + (size_t)t0 * g.k_in, nb,
                                                     (uint8_t*)y + (size_t)t0 * g.n_out * ybytes, y_dtype, false, (cudaStream_t)stream);
                if (e != cudaSuccess) return from_cuda(e);
            }
            return GOQ_OK;
        }
        if (goq::gemm_tc_supported(g) && variant != 2) {
            if (!ws || !aligned(ws, 256)) return ws ? GOQ_ERR_ALIGNMENT : GOQ_ERR_WORKSPACE;
            if (ws_bytes < goq::gemm_tc_workspace(g, m)) return GOQ_ERR_WORKSPACE;
        }
        // (up to 32 rows of a narrow group in less scratch than documented: the scalar kernel, slow but of the stated accuracy)
        if (goq::gemm_tc_supported(g) && variant != 2 && !(variant == 0 && exact && narrow))
            return from_cuda(goq::launch_gemm_tc(g, packed, x, m, y, y_dtype, ws, g_wait_limit.load(std::memory_order_relaxed), (cudaStream_t)stream));
        if (goq::linear_mma_supported(g))
            return from_cuda(goq::launch_linear_mma(g, packed, x, m, y, y_dtype, (cudaStream_t)stream));
        // what is left of the groups narrower than 32: the scalar kernel, 16 tokens at a time
        const size_t ybytes = (y_dtype == GOQ_F32) ? 4 : 2;
        for (int t0 = 0; t0 < m; t0 += 16) {
            const int nb = (m - t0 < 16) ? (m - t0) : 16;
            cudaError_t e = goq::launch_gemv_scalar(g, packed, (const uint16_t*)x + (size_t)t0 * g.k_in, nb,
                                                    (uint8_t*)y + (size_t)t0 * g.n_out * ybytes, y_dtype,
                                                    (cudaStream_t)stream);
            if (e != cudaSuccess) return from_cuda(e);
        }
        return GOQ_OK;
    }
    if (x_dtype == GOQ_I8) {
        if (!cq || (!y && !acc)) return GOQ_ERR_INVALID_ARG;
        if (y && (!sx || !sc)) return GOQ_ERR_INVALID_ARG;
        if (!aligned(acc, 4) || !aligned(sx, 4) || !aligned(sc, 4) || !aligned(cq, 2)) return GOQ_ERR_ALIGNMENT;
        if (g.group < 16 || (g.k_in % 16)) return GOQ_ERR_UNSUPPORTED;
        // |ACC| <= k_in * 127 (x~) * 127 (c~) * 2^emax must stay below 2^31
        const long long bound = (long long)g.k_in * 127 * 127 * (1ll << ((1 << (g.wbits - 1)) - 1));
        if (bound >= (1ll << 31)) return GOQ_ERR_OVERFLOW_BOUND;
        if (goq_status s = check_arch()) return s;
        int* status = (ws && aligned(ws, 256) && ws_bytes >= goq::kWsStatusBytes) ? (int*)ws : nullptr;   // needs no scratch; reports there if it may
        return from_cuda(goq::launch_gemm_a8(g, packed, (const int8_t*)x, m, sx, cq, sc, y, y_dtype, acc, nullptr, status,
                                             g_wait_limit.load(std::memory_order_relaxed), (cudaStream_t)stream));
    }
    return GOQ_ERR_INVALID_ARG;
}

goq_status goq_gemm_i8_requant(const goq_desc* desc, const void* packed, const int8_t* x, int m, const float* sx,
                               const int8_t* cq, const float* sc, float* y, float* amax, int8_t* yq, float* sy, void* stream) {
    Geometry g;
    if (!goq::make_geometry(desc, &g) || !packed || !x || m < 1 || !sx || !cq || !sc || !y || !amax) return GOQ_ERR_INVALID_ARG;
    if ((yq == nullptr) != (sy == nullptr)) return GOQ_ERR_INVALID_ARG;
    if (!aligned(packed, 128) || !aligned(x, 16) || !aligned(y, 4) || !aligned(amax, 4) || !aligned(sx, 4) || !aligned(sc, 4) ||
        !aligned(cq, 2) || !aligned(sy, 4))
        return GOQ_ERR_ALIGNMENT;
    if (g.group < 16 || (g.k_in % 16)) return GOQ_ERR_UNSUPPORTED;
    const long long bound = (long long)g.k_in * 127 * 127 * (1ll << ((1 << (g.wbits - 1)) - 1));
    if (bound >= (1ll << 31)) return GOQ_ERR_OVERFLOW_BOUND;
    if (goq_status s = check_arch()) return s;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaError_t e = cudaMemsetAsync(amax, 0, (size_t)m * sizeof(float), st)) return from_cuda(e);
    if (cudaError_t e = goq::launch_gemm_a8(g, packed, x, m, sx, cq, sc, y, GOQ_F32, nullptr, amax, nullptr,
                                               g_wait_limit.load(std::memory_order_relaxed), st)) return from_cuda(e);
    if (yq) return from_cuda(goq::launch_quantize_act(y, GOQ_F32, m, g.n_out, 8, amax, yq, sy, st));
    return GOQ_OK;
}

goq_status goq_quantize_activations(const void* x, int x_dtype, int m, int k, int abits, const float* amax, int8_t* xq,
                                    float* sx, void* stream) {
    if (!x || !xq || !sx || m < 1 || k < 1 || abits < 2 || abits > 8) return GOQ_ERR_INVALID_ARG;
    if (x_dtype != GOQ_F32 && x_dtype != GOQ_BF16) return GOQ_ERR_INVALID_ARG;
    if (!aligned(x, x_dtype == GOQ_F32 ? 4 : 2) || !aligned(sx, 4) || !aligned(amax, 4)) return GOQ_ERR_ALIGNMENT;
    if (goq_status s = check_arch()) return s;
    return from_cuda(goq::launch_quantize_act(x, x_dtype, m, k, abits, amax, xq, sx, (cudaStream_t)stream));
}

goq_status goq_quantize_geo(const goq_desc* desc, const float* w, uint8_t* codes, uint8_t* meta, uint16_t* coef_f16,
                            void* stream) {
    Geometry g;
    if (!goq::make_geometry(desc, &g) || !w || !codes || !meta || !coef_f16) return GOQ_ERR_INVALID_ARG;
    if (!aligned(w, 16) || !aligned(codes, 4) || !aligned(coef_f16, 2)) return GOQ_ERR_ALIGNMENT;
    if (goq_status s = check_arch()) return s;
    return from_cuda(goq::launch_quantize_geo(g, w, codes, meta, coef_f16, (cudaStream_t)stream));
}

goq_status goq_solve_ref(const goq_desc* desc, const float* w, const uint8_t* codes, const uint8_t* meta,
                         const float* x_calib, int m, double lambda, uint16_t* coef_f16, double* c_f64, void* stream) {
    Geometry g;
    if (!goq::make_geometry(desc, &g) || !w || !codes || !meta || !x_calib || !coef_f16 || m < 1 || !(lambda >= 0.0))
        return GOQ_ERR_INVALID_ARG;
    if (g.k1) return GOQ_ERR_UNSUPPORTED;
    if (!aligned(w, 4) || !aligned(x_calib, 4) || !aligned(coef_f16, 2) || !aligned(c_f64, 8)) return GOQ_ERR_ALIGNMENT;
    if (goq_status s = check_arch()) return s;
    if (goq::solve_ref_tc_supported(g, w, x_calib, m))
        return from_cuda(goq::launch_solve_ref_tc(g, w, codes, meta, x_calib, m, lambda, coef_f16, c_f64,
                                              g_wait_limit.load(std::memory_order_relaxed), (cudaStream_t)stream));
    return from_cuda(goq::launch_solve_ref(g, w, codes, meta, x_calib, m, lambda, coef_f16, c_f64, (cudaStream_t)stream));
}

size_t goq_sequence_workspace_bytes(int n_items) { return n_items > 0 ? goq::gemv_seq_workspace(n_items) : 0; }

goq_status goq_gemv_sequence(const goq_gemv_item* items, int n_items, void* ws, size_t ws_bytes, void* stream) {
    if (!items || n_items < 1) return GOQ_ERR_INVALID_ARG;
    static thread_local std::vector<goq::SeqCall> calls;
    calls.resize((size_t)n_items);
    for (int i = 0; i < n_items; ++i) {
        const goq_gemv_item& it = items[i];
        goq::SeqCall& c = calls[(size_t)i];
        if (!goq::make_geometry(&it.desc, &c.g) || !it.packed || !it.x_bf16 || !it.y) return GOQ_ERR_INVALID_ARG;
        if (it.batch < 1 || it.batch > 16) return GOQ_ERR_INVALID_ARG;
        if (it.y_dtype != GOQ_BF16 && it.y_dtype != GOQ_F32) return GOQ_ERR_INVALID_ARG;
        if (!aligned(it.packed, 128) || !aligned(it.x_bf16, 16) || !aligned(it.y, it.y_dtype == GOQ_F32 ? 4 : 2))
            return GOQ_ERR_ALIGNMENT;
        if (!goq::gemv_seq_supported(c.g, it.batch)) return GOQ_ERR_UNSUPPORTED;
        if (c.g.wbits != calls[0].g.wbits || c.g.group != calls[0].g.group) return GOQ_ERR_UNSUPPORTED;
        c.packed = it.packed; c.x = it.x_bf16; c.y = it.y; c.m = it.batch; c.y_dtype = it.y_dtype; c.depends = it.depends ? 1 : 0;
    }
    if (!ws || !aligned(ws, 256)) return ws ? GOQ_ERR_ALIGNMENT : GOQ_ERR_WORKSPACE;
    if (ws_bytes < goq::gemv_seq_workspace(n_items)) return GOQ_ERR_WORKSPACE;
    if (goq_status s = check_arch()) return s;
    if (!goq::stream_hash_is_bijective()) return GOQ_ERR_UNSUPPORTED;
    for (int i0 = 0; i0 < n_items; i0 += goq::kSeqMaxItems) {
        const int n = (n_items - i0 < goq::kSeqMaxItems) ? (n_items - i0) : goq::kSeqMaxItems;
        // a chunk boundary is a kernel boundary on the stream: the first item of a chunk needs no counter wait
        cudaError_t e = goq::launch_gemv_seq(&calls[(size_t)i0], n, calls[0].g.wbits, calls[0].g.group, calls[0].g.unit_bytes, ws,
                                             g_wait_limit.load(std::memory_order_relaxed), (cudaStream_t)stream);
        if (e != cudaSuccess) return from_cuda(e);
    }
    return GOQ_OK;
}

goq_status goq_sequence_order(const goq_gemv_item* items, int n_items, int32_t* kind_out, int32_t* source_out) {
    if (!items || n_items < 1 || !kind_out) return GOQ_ERR_INVALID_ARG;
    std::vector<goq::SeqCall> calls((size_t)n_items);
    for (int i = 0; i < n_items; ++i) {
        const goq_gemv_item& it = items[i];
        goq::SeqCall& c = calls[(size_t)i];
        if (!goq::make_geometry(&it.desc, &c.g) || !it.x_bf16 || !it.y || it.batch < 1) return GOQ_ERR_INVALID_ARG;
        if (it.y_dtype != GOQ_BF16 && it.y_dtype != GOQ_F32) return GOQ_ERR_INVALID_ARG;
        c.packed = it.packed; c.x = it.x_bf16; c.y = it.y; c.m = it.batch; c.y_dtype = it.y_dtype; c.depends = it.depends ? 1 : 0;
    }
    std::vector<goq::SeqOrder> order((size_t)n_items);
    // a launch holds at most kSeqMaxItems items: a later chunk starts after the earlier ones have completed
    for (int i0 = 0; i0 < n_items; i0 += goq::kSeqMaxItems) {
        const int n = (n_items - i0 < goq::kSeqMaxItems) ? (n_items - i0) : goq::kSeqMaxItems;
        goq::plan_sequence(&calls[(size_t)i0], n, &order[(size_t)i0]);
        for (int j = 0; j < n; ++j) {
            kind_out[i0 + j] = order[(size_t)(i0 + j)].kind;
            if (source_out) source_out[i0 + j] = order[(size_t)(i0 + j)].source < 0 ? -1 : i0 + order[(size_t)(i0 + j)].source;
        }
    }
    return GOQ_OK;
}

goq_status goq_gemv_sequence_host(const goq_gemv_item* items, int n_items, const void* x_host, void* x_stage,
                                  size_t x_bytes, void* y_host, void* y_stage, size_t y_bytes, void* ws,
                                  size_t ws_bytes, void* stream) {
    if (!items || n_items < 1 || !x_host || !x_stage || !y_host || !y_stage || !x_bytes || !y_bytes) return GOQ_ERR_INVALID_ARG;
    const uintptr_t xs = (uintptr_t)x_stage, ys = (uintptr_t)y_stage;
    for (int i = 0; i < n_items; ++i) {
        const goq_gemv_item& it = items[i];
        if (it.batch < 1 || it.desc.k_in <= 0 || it.desc.n_out <= 0) return GOQ_ERR_INVALID_ARG;
        const size_t xb = (size_t)it.batch * it.desc.k_in * 2;
        const size_t yb = (size_t)it.batch * it.desc.n_out * (it.y_dtype == GOQ_F32 ? 4 : 2);
        const uintptr_t x = (uintptr_t)it.x_bf16, y = (uintptr_t)it.y;
        const bool x_in_x = x >= xs && x + xb <= xs + x_bytes, x_in_y = x >= ys && x + xb <= ys + y_bytes;
        if (!(x_in_x || (x_in_y && i > 0)) || !(y >= ys && y + yb <= ys + y_bytes)) return GOQ_ERR_INVALID_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemcpyAsync(x_stage, x_host, x_bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return from_cuda(cudaGetLastError());
    goq_status s = goq_gemv_sequence(items, n_items, ws, ws_bytes, stream);
    if (s != GOQ_OK) return s;
    if (cudaMemcpyAsync(y_host, y_stage, y_bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess) return from_cuda(cudaGetLastError());
    return GOQ_OK;
}

goq_status goq_gemv_host(const goq_desc* desc, const void* packed, const void* x_host, int batch, void* y_host,
                         int y_dtype, void* x_stage, void* y_stage, void* ws, size_t ws_bytes, void* stream) {
    Geometry g;
    if (!goq::make_geometry(desc, &g) || !x_host || !y_host || !x_stage || !y_stage) return GOQ_ERR_INVALID_ARG;
    if (batch < 1 || batch > 16) return GOQ_ERR_INVALID_ARG;
    if (y_dtype != GOQ_BF16 && y_dtype != GOQ_F32) return GOQ_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t xb = (size_t)batch * g.k_in * 2, yb = (size_t)batch * g.n_out * (y_dtype == GOQ_F32 ? 4 : 2);
    if (cudaMemcpyAsync(x_stage, x_host, xb, cudaMemcpyHostToDevice, st) != cudaSuccess) return GOQ_ERR_CUDA;
    goq_status s = goq_gemv(desc, packed, x_stage, batch, y_stage, y_dtype, ws, ws_bytes, stream);
    if (s != GOQ_OK) return s;
    if (cudaMemcpyAsync(y_host, y_stage, yb, cudaMemcpyDeviceToHost, st) != cudaSuccess) return GOQ_ERR_CUDA;
    return GOQ_OK;
}

goq_status goq_workspace_init(void* ws, size_t ws_bytes, void* stream) {
    if (!ws || ws_bytes == 0) return GOQ_ERR_INVALID_ARG;
    return from_cuda(cudaMemsetAsync(ws, 0, ws_bytes, (cudaStream_t)stream));
}

goq_status goq_workspace_status(const void* ws, void* stream, int* status_out) {
    if (!ws || !status_out) return GOQ_ERR_INVALID_ARG;
    int v = 0;
    if (cudaMemcpyAsync(&v, ws, sizeof(int), cudaMemcpyDeviceToHost, (cudaStream_t)stream) != cudaSuccess)
        return GOQ_ERR_CUDA;
    if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return GOQ_ERR_CUDA;
    *status_out = v;
    return GOQ_OK;
}

int goq_last_cuda_error(void) { return g_last_cuda_error.load(std::memory_order_relaxed); }

int goq_set_gemv_variant(int variant) { return g_gemv_variant.exchange(variant); }

int goq_set_wait_limit(int polls) { return g_wait_limit.exchange(polls > 0 ? polls : 0); }

}  // extern "C"
