// Internal launcher declarations shared by the translation units of libgoq.
#pragma once
#include <cuda_runtime.h>
#include "goq_common.cuh"
#include "goq_device.h"

namespace goq {

// GOQ_OK, or GOQ_ERR_CUDA after remembering the error for goq_last_cuda_error and clearing a non-sticky one.
goq_status status_from_cuda(cudaError_t e);

cudaError_t launch_pack(const Geometry& g, const uint8_t* codes, const uint8_t* meta, const uint16_t* coef,
                        void* packed, cudaStream_t st);
cudaError_t launch_unpack(const Geometry& g, const void* packed, uint8_t* b1, uint8_t* b2, uint16_t* coef,
                          cudaStream_t st);

// Float-activation layer, scalar exponent-add kernel (any group size, batch <= 16).
cudaError_t launch_gemv_scalar(const Geometry& g, const void* packed, const void* x_bf16, int batch, void* y,
                               int y_dtype, cudaStream_t st);
// Float-activation layer, tensor-core fragment kernel (group >= 32); m may exceed 16.
cudaError_t launch_linear_mma(const Geometry& g, const void* packed, const void* x_bf16, int m, void* y,
                              int y_dtype, cudaStream_t st);
bool linear_mma_supported(const Geometry& g);

// Decode GEMV on bf16 fragments straight from global memory (group >= 32, wbits 2..4, m <= 16); no scratch (goq_gemv_mma.cu).
// early: the first weights may be read before earlier kernels of the stream are complete.
bool gemv_mma_supported(const Geometry& g, int m);
cudaError_t launch_gemv_mma(const Geometry& g, const void* packed, const void* x_bf16, int m, void* y, int y_dtype, bool early, cudaStream_t st);

// Decode GEMV, streaming kernel (group >= 32, wbits <= 3, m <= 16). `ws` holds gemv_stream_workspace(g)
// bytes whose tile counters are zero on entry (goq_workspace_init) and are left zero on return.
bool gemv_stream_supported(const Geometry& g);
size_t gemv_stream_workspace(const Geometry& g);
size_t gemv_stream_zeroed_prefix(const Geometry& g);  // leading bytes of the scratch that must be zero on entry
bool stream_hash_is_bijective();
cudaError_t launch_gemv_stream(const Geometry& g, const void* packed, const void* x_bf16, int m, void* y, int y_dtype,
                               void* ws, cudaStream_t st);

// A chain of decode GEMVs in one persistent cooperative kernel (group >= 32, wbits <= 3, batch <= 8, the staged
// activations of each linear fit in shared memory; every linear has the same wbits and group). `ws` holds
// gemv_seq_workspace(n) bytes whose first gemv_seq_zeroed_prefix(n) bytes are zero on entry and left zero on return.
// spin_limit > 0 replaces the bound of every device-side wait (tests make waits run out with it).
constexpr int kSeqMaxItems = 256;
struct SeqCall {
    Geometry g;
    const void* packed;
    const void* x;
    void* y;
    int m, y_dtype, depends;
};
// Ordering of one item of a sequence launch, decided on the host from the address ranges
enum { kSeqOrderNone = 0, kSeqOrderData = 1, kSeqOrderBarrier = 2 };
struct SeqOrder {
    int kind;               // kSeqOrder...
    int source;             // kSeqOrderData: the earlier item whose output holds this item's activations
    unsigned word_offset;   // ... and where they start in that item's tagged copy (64-bit words)
};
void plan_sequence(const SeqCall* calls, int n, SeqOrder* out);
bool gemv_seq_supported(const Geometry& g, int m);
size_t gemv_seq_workspace(int n_items);
size_t gemv_seq_zeroed_prefix(int n_items);
cudaError_t launch_gemv_seq(const SeqCall* calls, int n, int wbits, int group, int unit_bytes, void* ws, int spin_limit,
                            cudaStream_t st);

// One decode GEMV of at most 4 tokens with the chain kernel's arithmetic, as a programmatic dependent launch (goq_gemv_one.cu).
// `ws` as for launch_gemv_stream (only the status word and the zero-kept counter area are used).
bool gemv_one_supported(const Geometry& g, int m);
cudaError_t launch_gemv_one(const Geometry& g, const void* packed, const void* x_bf16, int m, void* y, int y_dtype, void* ws,
                            int spin_limit, cudaStream_t st);

// Prefill GEMM on tcgen05 tensor cores (any wbits and group whose records fit the ring). `ws` holds gemm_tc_workspace(g, m) bytes: status word and
// (split-K) tile counters in the common areas, then the per-token scales, the fp16 copy of the m x k_in activations
// and the split-K partial tiles.
bool gemm_tc_supported(const Geometry& g);
size_t gemm_tc_workspace(const Geometry& g, int m);
float gemm_tc_us(const Geometry& g, int m);   // estimated time, more than 256 tokens
cudaError_t launch_gemm_tc(const Geometry& g, const void* packed, const void* x_bf16, int m, void* y, int y_dtype,
                           void* ws, int spin_limit, cudaStream_t st);

// Its main kernel on pairs of SMs, more than 256 tokens (goq_gemm_pair.cu): xh, inv_scale, row_scale, row_inv as the pre-pass leaves them.
bool gemm_pair_supported(const Geometry& g, int m);
float gemm_pair_us(const Geometry& g, int m);   // estimated time, pre-pass included
cudaError_t launch_gemm_pair(const Geometry& g, const void* packed, const void* xh, const float* inv_scale, const uint32_t* row_scale, const float* row_inv,
                             int m, void* y, int y_dtype, int* status, int spin_limit, cudaStream_t st);

// The same layer for a few to a few hundred tokens (goq_gemm_mid.cu), any group, wbits 2..4. exact: the two bases as separate
// operands without rounding (fp32 accuracy), else w_hat rounded once to fp16. `ws` holds gemm_mid_workspace bytes.
bool gemm_mid_supported(const Geometry& g, int m, bool exact);
float gemm_mid_us(const Geometry& g, int m);   // estimated time, more than 256 tokens
int gemm_mid_ctas();                           // CTAs of a full grid: one per SM
size_t gemm_mid_workspace(const Geometry& g, int m, bool exact);
size_t gemm_mid_workspace_upto(const Geometry& g, int m);   // enough for every call of up to m rows, either form
cudaError_t launch_gemm_mid(const Geometry& g, const void* packed, const void* x_bf16, int m, void* y, int y_dtype, void* ws,
                            bool exact, int spin_limit, cudaStream_t st);

// The same layer for a few tokens up to about 128 (goq_gemm_f8.cu): both bases and the activations as exact e4m3 operands; group >= 32.
bool gemm_f8_supported(const Geometry& g, int m);
float gemm_f8_us(const Geometry& g, int m);   // estimated time
size_t gemm_f8_workspace(const Geometry& g, int m);
size_t gemm_f8_workspace_upto(const Geometry& g, int m);
cudaError_t launch_gemm_f8(const Geometry& g, const void* packed, const void* x_bf16, int m, void* y, int y_dtype, void* ws, int spin_limit, cudaStream_t st);

// ... its summing kernel, which also computes the tokens of which the pre-pass has left a mark (goq_gemm_f8_finish.cu). tile_tokens: of a token tile
cudaError_t launch_f8_finish(const Geometry& g, const void* packed, const void* x, int m, void* y, int y_dtype, const float* partial, const float* inv_scale,
                             const int* marks, int tile_tokens, int tiles_x, int t_tiles, int units, int n_ctas, cudaStream_t st);

// Integer-activation layer.
// amax (optional, with y): per-token largest |y|, combined into the array with an integer max (zero it before the launch); NaN after a
// give-up. spin_limit > 0 replaces the bound of every device-side wait (tests).
cudaError_t launch_gemm_a8(const Geometry& g, const void* packed, const int8_t* x, int m, const float* sx,
                           const int8_t* cq, const float* sc, void* y, int y_dtype, int32_t* acc, float* amax, int* status,
                           int spin_limit, cudaStream_t st);

// The same on tcgen05 (goq_gemm_i8tc.cu), group >= 32, any wbits.
bool gemm_i8tc_supported(const Geometry& g, int m);
cudaError_t launch_gemm_i8tc(const Geometry& g, const void* packed, const int8_t* x, int m, const float* sx, const int8_t* cq, const float* sc,
                             void* y, int y_dtype, int32_t* acc, float* amax, int* status, int spin_limit, cudaStream_t st);

// The steps before the inner product (goq_quant.cu).
cudaError_t launch_quantize_geo(const Geometry& g, const float* w, uint8_t* codes, uint8_t* meta, uint16_t* coef, cudaStream_t st);
cudaError_t launch_solve_ref(const Geometry& g, const float* w, const uint8_t* codes, const uint8_t* meta, const float* x_calib,
                             int m, double lambda, uint16_t* coef, double* c_out, cudaStream_t st);
// The same on int8 tensor cores (goq_ref_tc.cu): groups of 32 and more, more observations than half a group, aligned inputs. Without a status
// word: a give-up of a bounded wait leaves NaN coefficients.
bool solve_ref_tc_supported(const Geometry& g, const float* w, const float* x_calib, int m);
cudaError_t launch_solve_ref_tc(const Geometry& g, const float* w, const uint8_t* codes, const uint8_t* meta, const float* x_calib, int m,
                                double lambda, uint16_t* coef, double* c_out, int spin_limit, cudaStream_t st);
cudaError_t launch_quantize_act(const void* x, int x_dtype, int m, int k, int abits, const float* amax, int8_t* xq, float* sx,
                                cudaStream_t st);

}  // namespace goq
