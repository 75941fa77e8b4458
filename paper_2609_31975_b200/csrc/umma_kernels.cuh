// Launchers of the tcgen05 (TMEM accumulator) kernels of the batched path (see umma_kernels.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sffn {

// Value of UmmaRowsParams::act that stores the raw products (no bias is usually given, no activation).
constexpr int kUmmaActIdentity = 3;

// Token columns one pass of these kernels takes (the N of their MMAs).
constexpr int kUmmaMaxCols = 256;
constexpr int kUmmaExactTokens = 64;  // tokens of a pass with exact sums (see umma_kernels.cu) ...
constexpr int kUmmaExactCols = 128;   // ... and token columns, terms included, of one launch of it

struct UmmaRowsParams {
  const void* W;         // [*, K] bf16 (or int8 / packed int4 codes, see qbits), rows selected by idx (or 0..R-1)
  int R, K;
  int qbits;             // 0: bf16 rows; 8 / 4: rows of weight codes, K * qbits / 8 bytes each, expanded to bf16 in
                         // shared memory; 1: int8 rows multiplied as int8 -- X then holds the tokens as int8 limbs (four
                         // rows per token, launch_token_limbs) and tok_scale their scales; 2: the same for int4 rows,
                         // whose nibbles are expanded to int8 (16 x the code) in shared memory
  const float* tok_scale;  // qbits = 1: scale of each token's limbs
  const float* w_scale;  // quantised rows: scale of row j of W (applied to its accumulator row), or null
  const float* out_scale;  // UP, quantised rows: scale of row j of the down matrix, folded into Hm, or null
  const int32_t* idx;    // UP: list of rows, or null
  const int32_t* count;  // UP: device length of the list, or null (= R)
  const uint32_t* words_in;  // UP, instead of idx / count: the gate kernel's "fired" bit masks (n_words of
  int n_words;               //   them, 4 per gate tile of gate_tile_rows rows); the kernel compacts them itself
  int gate_tile_rows;
  int gate_rows_per_word;    //   rows covered by one mask word (umma_gate_rows_per_word)
  int32_t* idx_out;          //   ... and writes the ascending list
  int32_t* count_out;        //   ... and its length
  int32_t* walk_all;         //   ... and 1 here when it walked every row instead of the list (the down kernel must too), else 0
  const void* X;         // token operand [cols][K] bf16, row stride x_stride (elements)
  int x_stride;
  int ncols_valid;
  int B;                 // tokens
  int x_cols;            // GATE: nonzero (a multiple of 8) = token b's vector is the sum of columns b and x_cols + b
                         //   (exact: and 2 x_cols + b)
  int exact;             // sums that round as fp32 does: chains of few MMAs added in registers; h in three terms
  const float* b_g;
  const int32_t* g_idx;
  const int8_t* g_sign;
  const void* xtok;      // tokens [B][.] bf16 for the fixed-matrix term
  int xtok_stride;
  int act;
  float* a_out;          // GATE: gate values a_out[b * a_stride + j]
  int k_splits, k_tiles; // GATE, raw products only (0: not cut): runs of K and tiles of rows (umma_k_splits); run i writes
  size_t split_stride;   //   at a_out + i * split_stride; limbs (qbits = 1 / 2): all add their integers to rows 4 b + l of a_out
  int run_blocks, longer_runs, equal_max;  // filled by the launcher
  uint8_t* flag;         // GATE: [R] any token fires, or null
  uint32_t* words_out;   // GATE: the same as bit masks, word 4 * tile + epilogue warp, or null
  const float* a;        // UP: gate values
  int a_stride;
  void* hmT;             // UP: bf16 [h_terms * h_cols][hm_stride]: h of token b is the sum of rows b and (2 terms) h_cols + b
  int hm_stride;
  int h_terms, h_cols;   //   2 terms: quantised rows only (0: 1); exact: 3
  int act_up;            // UP: activation on the up projection (double activation), kUmmaActIdentity = none
  int32_t* status;       // device status word
  int npad, ring_bytes, pair;  // filled by the launcher
  long long wait_cycles; // budget of every device-side wait (filled by the launcher)
  int drop_stage;        // test hook: CTA 0 of the gate kernel never copies the weights of this stage (-1: none)
};

struct UmmaDownParams {
  const void* W_down;    // [R, D] bf16 (or codes, see qbits; their row scales are already folded into hmT)
  int R, D;
  int qbits;             // 0: bf16 rows; 8 / 4: rows of weight codes
  const int32_t* idx;    // list of rows (readable up to the next multiple of 64 past its length), or null = all R rows
  const int32_t* count;  // device length of the list, or null (= R)
  const void* hmT;       // bf16 [terms * h_cols][hm_stride] (see UmmaRowsParams); entries from the list's end to the next
                         // multiple of 64 are zero
  int hm_stride;         // multiple of 64
  int terms, h_cols;     // terms of h (0: 1) and the rows between them
  int exact;             // see UmmaRowsParams
  int tok0, B;           // tokens [tok0, tok0 + B) of those rows
  int cols;              // B rounded up to a multiple of 8 (token columns of one term)
  int splits;            // the list is cut into this many runs of 64-row blocks (umma_down_splits)
  const int32_t* walk_all;  // device word: nonzero = walk every row of W_down instead of the list (set by the up kernel), or null
  float* y;              // [B][D]: the splits are clusters (umma_down_splits), or null:
  float* partial;        //   [splits][B][D]
  int32_t* status;
  int npad, stages, expand, ring_bytes;  // filled by the launcher
  long long wait_cycles; // budget of every device-side wait (filled by the launcher)
};

// How the list (of up to R rows) is split; true: `y`, in clusters, false: `partial` (at most max_splits).  cols: token columns of all
// terms.  at_once[n]: clusters of n CTAs that the device runs at once (null: it is asked).
bool umma_down_splits(int D, int R, int qbits, int cols, bool exact, int sm_count, int max_splits, int* splits, const int* at_once = nullptr);
bool umma_down_supported(int D, int cols);
cudaError_t launch_umma_down(UmmaDownParams p, cudaStream_t s);
bool umma_rows_supported(int K, int cols);
// Batches wide enough for the up kernel to consider walking every row instead of the union list.
bool umma_may_walk(int B);
// R gate rows of K elements or codes (qbits as in UmmaRowsParams) against B tokens
bool umma_own_list_supported(int R, int K, int qbits, int B, int sm_count);
void umma_gate_tiling(int R, int K, int qbits, int B, int sm_count, int* tile_rows, int* n_tiles);
// Rows that a word of that gate's "fired" masks covers (`cols`: its token columns, limbs or terms included).
int umma_gate_rows_per_word(int R, int K, int qbits, int B, int cols, bool exact, int sm_count);
// Whether that gate, or an up projection that may walk every row, runs in pairs of CTAs.
bool umma_rows_pairs(int R, int K, int qbits, int B, int cols, bool exact, int sm_count);
cudaError_t launch_umma_rows(bool up, UmmaRowsParams p, int cols, int sm_count, cudaStream_t s);
bool umma_rows_native_i8_supported(int K, int tokens);
// Tokens [B][K] bf16 as four int8 limbs each ([4 B][K], most significant first, 7 bits apart) and one scale per token;
// zeroes B * zero_bytes (a multiple of 16) beside it.
cudaError_t launch_token_limbs(const void* x, int B, int K, int x_stride, void* limbs, float* scale, void* zero, int zero_bytes,
                               cudaStream_t s);
// How v = V x (R rows of K elements, or codes against limbs; B tokens) is cut: `splits` runs of K (1: not), each over `tiles` tiles
// of rows.
void umma_k_splits(int R, int K, bool codes, int B, int sm_count, int max_splits, int* tiles, int* splits);
// The same for the LoPA vector n = RMSNorm(v) (or v): from fp32 (`sums` null), or from integer sums, four rows of v_stride a token.
struct UmmaLimbSums {
  const float *row_scale, *tok_scale;  // of V's rows and of the tokens' limbs
  float code_scale;                    // 1, or 1 / 16 (4-bit codes, whose products are of 16 x the code)
};
cudaError_t launch_rmsnorm_limbs(float* v, int B, int r, int v_stride, const UmmaLimbSums* sums, const float* gain, float eps,
                                 bool use_rms, void* limbs, float* scale, cudaStream_t s);
// The bf16 pairs (or triples) of n.  v is the sum of `runs` vectors, `step` floats apart.
cudaError_t launch_rmsnorm_split(float* v, int B, int r, int v_stride, int runs, size_t step, const float* gain, float eps,
                                 bool use_rms, int cols, bool exact, void* x2, cudaStream_t s);

}  // namespace sffn
