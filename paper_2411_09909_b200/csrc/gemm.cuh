// Internal launchers of the two GEMM kernels.
#pragma once

#include "amx_common.cuh"

namespace amx {

// Codes of an operand as one plane or as two sign planes whose nibbles are or-ed (a prepared operand keeps no other copy).
struct CodePlanes {
    const uint8_t* a;
    const uint8_t* b = nullptr;
};
int gemm_simt(CodePlanes a_codes, const uint8_t* a_scales, CodePlanes w_codes, const uint8_t* w_scales, int64_t M, int64_t N,
              int64_t K, int gs, float* C, int64_t ld_c, cudaStream_t st,
              const int* run_if_nonzero = nullptr /* device word: nothing is done when zero */);

// The same kernel on operands with binary16 shared scales ([rows, K/gs, 2] uint16).
int gemm_simt_f16s(const uint8_t* a_codes, const uint16_t* a_scales, const uint8_t* w_codes,
                   const uint16_t* w_scales, int64_t M, int64_t N, int64_t K, int gs, float* C,
                   int64_t ld_c, cudaStream_t st);

// Tensor-core (tcgen05) kernel: shapes it accepts, scratch it needs, launcher.
bool gemm_tc_supported(int64_t M, int64_t N, int64_t K, int gs);
size_t gemm_tc_workspace_bytes(int64_t M, int64_t N, int64_t K);
// run_if_nonzero (optional, device word): the launch does nothing when that word is zero.  status_word
// (optional): a status word the caller has cleared, used instead of the workspace's first word.
int gemm_tc(CodePlanes a_codes, const uint8_t* a_scales, CodePlanes w_codes,
            const uint8_t* w_scales, int64_t M, int64_t N, int64_t K, float* C, int64_t ld_c,
            void* workspace, cudaStream_t st, const int* run_if_nonzero = nullptr, int* status_word = nullptr);
// The same product with the cast of the bf16 activation X [M, ld_a] done inside the kernel.
int gemm_tc_cast(const void* x, int64_t ld_a, const uint8_t* w_codes, const uint8_t* w_scales, int64_t M,
                 int64_t N, int64_t K, float* C, int64_t ld_c, void* workspace, cudaStream_t st);
int gemm_tc_status(const void* workspace, cudaStream_t st);

// Weight-streaming kernel for few rows of A (mma.sync on exactly decoded f16, K ranges over a cluster; any fixed group
// size, K % 128 == 0).  Up to kRowsMaxM rows: blocks of at most 64 rows re-read the weight.  The workspace holds the
// status words and room for the decoded rows; gemm_rows_cast casts the bf16 rows X [M, ld_x] itself.
constexpr int64_t kRowsMaxM = 256;
bool gemm_rows_supported(int64_t M, int64_t N, int64_t K, int gs);
size_t gemm_rows_workspace_bytes(int64_t M, int64_t N, int64_t K);
double gemm_rows_estimated_us(int64_t M, int64_t N, int64_t K);
// amx_quant_gemm with the kernel that AUTO stands for given (0: AUTO's own choice), and its workspace with a quantized weight
// on the streaming kernel (0: that kernel does not take the shape).  api.cu
int quant_gemm(const void* A, int64_t ld_a, const uint8_t* w_codes, const uint8_t* w_scales, const void* W_bf16, int64_t ld_w, int64_t M,
               int64_t N, int64_t K, int group_size, uint32_t flags, uint32_t auto_kernel, float* C, int64_t ld_c, void* workspace,
               size_t workspace_bytes, void* stream);
size_t quant_gemm_rows_bytes(int64_t M, int64_t N, int64_t K, int gs);
int gemm_rows(const uint8_t* a_codes, const uint8_t* a_scales, const uint8_t* w_codes, const uint8_t* w_scales,
              int64_t M, int64_t N, int64_t K, int gs, float* C, int64_t ld_c, void* workspace, cudaStream_t st);
int gemm_rows_cast(const void* x, int64_t ld_x, const uint8_t* w_codes, const uint8_t* w_scales, int64_t M, int64_t N,
                   int64_t K, int gs, float* C, int64_t ld_c, void* workspace, cudaStream_t st);

// FP4-pipe kernel (four block-scaled MMAs per tile pair): same contract; the workspace also holds
// the prepared operands (sign planes, UE4M3 scale-factor blocks, row offsets).
bool gemm_fp4_supported(int64_t M, int64_t N, int64_t K, int gs);
size_t gemm_fp4_workspace_bytes(int64_t M, int64_t N, int64_t K);
int gemm_fp4(const uint8_t* a_codes, const uint8_t* a_scales, const uint8_t* w_codes,
             const uint8_t* w_scales, int64_t M, int64_t N, int64_t K, float* C, int64_t ld_c,
             void* workspace, cudaStream_t st, bool gate_on_flushed = false, int gs = 32);
// The same in two phases, so that an operand (typically the weight) is prepared once and reused.
size_t gemm_fp4_prepared_bytes(int64_t rows, int64_t K, bool is_weight);
size_t gemm_fp4_plane_bytes(int64_t rows, int64_t K);
// One operand to prepare (quantize.cu): a bf16 matrix x to cast, or a canonical one (x == nullptr).
struct PrepOperand {
    const uint4* x;              // bf16 rows, ld_vec 16-byte pieces apart
    int64_t ld_vec;
    const uint4* in_codes;       // canonical operand
    const uint16_t* in_scales;
    int64_t R;                   // operand rows
    unsigned seg_rows, seg_blocks;   // seg_blocks != 0: x holds segments of seg_rows rows, each padded to seg_blocks blocks of 128
                                     // operand rows with zero scale factors and row words
    uint4* codes;                // out, of a cast: canonical codes (optional) and scales
    uint16_t* scales;
    uint4 *pos, *neg;            // out: planes, scale factors, row words
    uint8_t *sf_pos, *sf_neg;
    int* row_exp;
    int64_t padded_rows;
};
// flushed_total (optional, device): incremented by the number of nonzero scales that fell below the UE4M3 range
// of their row and were flushed; the per-row counts are in the row words either way.
int prepare_operands(const PrepOperand* op, int n, int64_t K, int gs, int nk64, cudaStream_t st, int format = AMX_FMT_AMXFP4,
                     int* flushed_total = nullptr);
// Descriptions of an operand laid out for layout_rows rows (0: rows) as the left-hand or right-hand one: a cast (ld in
// elements), or the preparation of a canonical operand; and the launch for one or two of them.
PrepOperand gemm_fp4_cast_operand(const void* x, int64_t ld, int64_t rows, int64_t K, bool is_weight, uint8_t* codes, uint8_t* scales,
                                  void* prepared, int64_t layout_rows = 0, int64_t seg_rows = 0, int64_t seg_pad = 0);
PrepOperand gemm_fp4_split_operand(const uint8_t* codes, const uint8_t* scales, int64_t rows, int64_t K, bool is_weight,
                                   void* prepared, int64_t layout_rows = 0);
int gemm_fp4_prepare_operands(const PrepOperand* op, int n, int64_t K, int gs, cudaStream_t st, int format = AMX_FMT_AMXFP4,
                              int* flushed_total = nullptr);
// The casts of an attention call in one launch: two operands described above, and V ([kv_heads][L][d], contiguous) as V^T, 128
// operand rows per head, laid out for layout_rows rows; its canonical scales (and no codes) are written beside.
int gemm_fp4_prepare_attention(const PrepOperand (&qk)[2], const void* v, int64_t kv_heads, int64_t L, int64_t d, int64_t layout_rows,
                               uint8_t* v_scales, void* v_prepared, cudaStream_t st, int* flushed_total);
struct VtOperand {
    const uint4* x;
    int64_t L;
    int d, nk64;
    uint4 *pos, *neg;
    uint16_t* scales;
    uint8_t *sf_pos, *sf_neg;
    int* row_exp;
};
int prepare_attention(const PrepOperand (&qk)[2], int64_t d, int nk64, const VtOperand& vt, int64_t kv_heads, cudaStream_t st, int* flushed_total);
const int* gemm_fp4_row_words(const void* prepared, int64_t rows, int64_t K, bool is_weight);
// Softmax of the rows of S, rounded to bf16 and cast in one launch (cols % 32 == 0); pos == nullptr: canonical
// output only.  gemm_fp4_softmax_prepared lays the prepared operand out like gemm_fp4_quantize_prepared.
int softmax_cast_rows(const float* S, int64_t rows, int64_t cols, int64_t ld_s, float alpha, uint8_t* codes,
                      uint8_t* scales, void* pos, void* neg, uint8_t* sf_pos, uint8_t* sf_neg, int* row_exp, int nk64,
                      int64_t padded_rows, cudaStream_t st,
                      int64_t causal = 0 /* rows per matrix: row i of a matrix sees columns 0 .. i */);
int gemm_fp4_softmax_prepared(const float* S, int64_t rows, int64_t cols, int64_t ld_s, float alpha, bool is_weight,
                              uint8_t* codes, uint8_t* scales, void* prepared, cudaStream_t st, int64_t causal = 0);
// A prepared operand that stacks several matrices row-wise (rows_total rows, laid out for layout_rows >=
// rows_total rows) and the first row of the one to multiply; row0 % 128 == 0.  A right-hand operand whose 256-row
// tiles can reach past rows_total needs layout_rows >= rows_total + 128.
struct Fp4Operand {
    const void* prepared;
    int64_t rows_total, layout_rows, row0;
};
int gemm_fp4_prepared_at(const Fp4Operand& a, const Fp4Operand& w, int64_t M, int64_t N, int64_t K, float* C,
                         int64_t ld_c, void* workspace, cudaStream_t st, size_t workspace_bytes = 256,
                         const int* gate = nullptr /* device word: the kernel does nothing when it is nonzero */,
                         const float* scale_a = nullptr, const float* scale_w = nullptr /* device: one factor per
                         operand; every result is multiplied by their product (NVFP4 tensor scales) */,
                         bool one_plane = false /* the caller states that neither operand has a second sign plane:
                         full-width tiles run the deeper one-plane pipeline, which reports AMX_ERR_FLAGS in the status
                         word when a tile has a second plane after all */,
                         bool out_bf16 = false /* C points to bf16 [M, ld_c]: results rounded to nearest even */);
// workspace that lets the kernel cut K into ranges for products with few output tiles (256 bytes otherwise)
size_t gemm_fp4_prepared_workspace_bytes(int64_t M, int64_t N, int64_t K);
// C[m][n] = sum over `slices` partial products [slices][M][N], in slice order (defined with the bf16-decode kernel)
int reduce_slices(const float* part, int slices, int64_t M, int64_t N, float* C, int64_t ld_c, cudaStream_t st,
                  const int* run_if_nonzero = nullptr);
// Fused attention for head dimensions 128 and 64 (attention_fp4.cu): both products and the softmax in one or two launches,
// logits and attention map never in global memory.  Operands prepared ahead, heads stacked row-wise, padded to whole blocks
// of 128.
bool attn_fused_supported(int64_t L, int64_t d);
int64_t attn_fused_padded(int64_t L);
size_t attn_fused_scratch_bytes(int64_t heads, int64_t L, bool ordered);
int attn_fused(const Fp4Operand& q, const Fp4Operand& k, const Fp4Operand& vt, int heads, int64_t L, int64_t d, float alpha,
               int causal, bool ordered /* the softmax kernel's statistics bit for bit; otherwise online ones, d = 128 and L a
               multiple of 128 only */,
               void* scratch, float* O, void* workspace /* 256 B: status word, cleared by the caller */, cudaStream_t st, void* dbg_bits = nullptr, uint8_t* dbg_codes = nullptr, uint8_t* dbg_scales = nullptr,
               void* dbg_prepared = nullptr, int kv_group = 1 /* query heads per head of keys and values */,
               const int* gate = nullptr /* device word: the kernels do nothing when it is nonzero */);
// The same attention on CUDA cores from the planes (or-ed: the codes) and canonical scales of those operands, any scale
// range; nothing is done when *run_if_nonzero is zero.  attention_exact.cu
struct ExactOperand {
    const uint8_t *pos, *neg, *scales;
};
bool attn_exact_supported(int64_t L, int64_t d);
int attn_exact(const ExactOperand& q, const ExactOperand& k, const ExactOperand& vt, int heads, int64_t L, int64_t d, int kv_group,
               float alpha, int causal, float* O, const int* run_if_nonzero, cudaStream_t st);
// Batched bf16-decode products (gemm_tc.cu): `batch` left operands one after another, right operand (first + b) / group for
// product b.  causal: tiles that lie entirely above the diagonal are left out (C there is not written).
size_t gemm_tc_batched_workspace_bytes(int64_t batch, int64_t M, int64_t N, int64_t K);
int gemm_tc_batched(const uint8_t* a_codes, const uint8_t* a_scales, const uint8_t* w_codes, const uint8_t* w_scales, int64_t batch,
                    int64_t first, int64_t group, int64_t M, int64_t N, int64_t K, float* C, bool causal, void* workspace,
                    cudaStream_t st);
int quantize_cols_batched(const void* x, int64_t batch, int64_t R, int64_t C, uint8_t* codes, uint8_t* scales,
                          cudaStream_t st);
int gemm_fp4_prepared(const void* a_prepared, const void* w_prepared, int64_t M, int64_t N, int64_t K,
                      float* C, int64_t ld_c, void* workspace /* 256 B: status word */, cudaStream_t st,
                      size_t workspace_bytes = 256, const int* gate = nullptr);

}  // namespace amx
