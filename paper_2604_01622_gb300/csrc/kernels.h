// Internal launchers of the EC-MoE library. Not part of the C ABI.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <cuda_bf16.h>

#include "launch.h"

namespace ecmoe {

// ---------------------------------------------------------------- router + selection
// fp32 router: logits X.Wr (+ br) and their row softmax in one kernel, S [N][E] (NULL: not
// written) and S^T [E][N]; sets the slot map slot [N][E] (if given) to -1, the state launch_topk
// expects. X [N][d], Wr [d][E].
cudaError_t launch_router_f32(const float* X, const float* Wr, const float* br, float* S,
                              float* ST, int* slot, int N, int d, int E, LaunchStream st);
// Expert-choice top-k per (expert, group) over the scores ST [E][N]: idx/gate [E][M], and where
// given a second copy of both (idx2, gate2), a copy of the scores (S_copy [E][N]) and, for the
// selected pairs only, the token->slot map slot [N][E] (= m), whose other entries must already
// hold -1. group_off/k_g/k_off: device tables of the G groups, the longest of max_group tokens;
// aligned: every column starts on a 16-byte boundary of ST. No output overlaps ST.
struct TopkArgs {
  const float* ST = nullptr;
  int N = 0, E = 0, M = 0;
  const int *group_off = nullptr, *k_g = nullptr, *k_off = nullptr;
  int *idx = nullptr, *idx2 = nullptr;
  float *gate = nullptr, *gate2 = nullptr, *S_copy = nullptr;
  int* slot = nullptr;
};
cudaError_t launch_topk(const TopkArgs& p, int G, int max_group, bool aligned, LaunchStream st);

// Capacity update from device memory (one CTA): if 0 <= k_new[g] <= L_g for every group and
// sum k_new == M, writes k_g [G] and its prefix sums k_off [G+1]; otherwise leaves both and
// records DEV_BAD_CAPACITY in the status word.
cudaError_t launch_set_capacity(const int* k_new, const int* group_off, int G, int M, int* k_g,
                                int* k_off, int* status, LaunchStream st);

// ---------------------------------------------------------------- token-choice routing
// Token-choice routing of the scores S [N][E] (k <= 32, E <= 256; cap < 0: no cap):
// choice/tgate/kept [N][k] (experts best first, normalised gates, kept flags), Z [N] (sum of
// the k chosen scores), count [E+1] (kept rows per expert; count[E] = padded rows in use),
// tiles [E+1] (cumulative 256-row blocks), row_gate [P] of each kept pair's row (padding rows
// untouched), slot [N][E] absolute padded row of each kept pair, else -1.
// scratch: tc_route_scratch_ints(N, E) ints. Four kernels.
cudaError_t launch_tc_route(const float* S, int N, int E, int k, int cap, int* choice,
                            float* tgate, float* Z, int* count, int* tiles, float* row_gate,
                            int* slot, int* kept, int* scratch, LaunchStream st);
int64_t tc_route_scratch_ints(int N, int E);
// Router gradient of token choice: dZ [N][E] (and optionally the bf16 hi/lo planes
// dZb [2][N][Ep]) from the per-row gate-gradient partials row_dgate [parts][P].
cudaError_t launch_tc_softmax_bwd(const float* S, const int* choice, const float* tgate,
                                  const float* Z, const int* slot, const float* row_dgate, int parts,
                                  int64_t P, float* dZ, __nv_bfloat16* dZb, int N, int E, int Ep,
                                  int k, LaunchStream st);

// ---------------------------------------------------------------- data movement
// Token-major form of the gather: for each token t, X row t is copied to row e*M + slot[t][e]
// of H for every expert e with slot[t][e] >= 0 (M = 0: slot holds absolute rows). With count [E]
// and tiles [E+1] (in 256-row blocks, device arrays) the unused rows of the variable-row expert
// regions are zeroed as well.
template <typename T>
cudaError_t launch_scatter_rows(const T* X, const int* slot, T* H, int N, int E, int M, int d,
                                LaunchStream st, const int* count = nullptr,
                                const int* tiles = nullptr);
// Y_t = R_t + R2_t (each if given) + sum over the experts that chose t of gate * O row
// (gate NULL: 1, for O rows already scaled by their gates).
template <typename T>
cudaError_t launch_combine(const T* O, const float* gate, const int* slot, const T* R, const T* R2,
                           T* Y, int N, int E, int M, int d, LaunchStream st);
// dO row r = gate[r] dY row idx[r], dgate[r] = <dY row idx[r], O row r>, for the P rows (fp32
// path).
template <typename T>
cudaError_t launch_bwd_gather_scale(const T* dY, const T* O, const int* idx, const float* gate,
                                    T* dO, float* dgate, int64_t P, int d, LaunchStream st);
// Router softmax Jacobian: dS[t][e] = dgate of the pair (t chosen by e) else 0,
// dZ = S (dS - <dS, S>_row). dgate [E*M] summed beforehand; writes dZ [N][E] and, with dZb,
// the bf16 hi/lo planes [2][N][Ep] (any E <= 512).
cudaError_t launch_softmax_bwd(const float* S, const int* slot, const float* dgate, float* dZ,
                               __nv_bfloat16* dZb, int N, int E, int Ep, int M, LaunchStream st);
// The same, fused with the sum of the gate-gradient partials dg_part [parts][E*M] (in part
// order) and, with dbr, with the router bias gradient dbr[e] = sum_t dZ[t][e] (per-CTA
// column sums in scratch, then summed in a fixed order: deterministic). dZ and dZb are each
// optional. For E % 4 == 0, E <= 128 and E*M < 2^31 (router_bwd_fused); one kernel, two
// with dbr. scratch: router_bwd_scratch_floats(N, E) floats.
bool router_bwd_fused(int E, int64_t P);
int64_t router_bwd_scratch_floats(int N, int E);
cudaError_t launch_router_softmax_bwd(const float* S, const int* slot, const float* dg_part,
                                      int parts, float* dZ, __nv_bfloat16* dZb, float* dbr,
                                      float* scratch, int N, int E, int Ep, int M,
                                      LaunchStream st);
cudaError_t launch_reduce_partials(const float* part, float* out, int rows, int cols, int ld,
                                   int splits, LaunchStream st);
// dX_t = dXr_t + R_t + R2_t (each if given) + sum of the token's dH rows, summed in fp32;
// dXr (the router's part of the input gradient) is in the layer's dtype.
template <typename T>
cudaError_t launch_dx_combine(const T* dH, const int* slot, const T* dXr, const T* R,
                              const T* R2, T* dX, int N, int E, int M, int d, LaunchStream st);
// out[e] = sum over the N rows of Z [N][E]; scratch: colsum_scratch_floats(N, E) floats.
// Two kernels.
cudaError_t launch_colsum(const float* Z, float* out, int N, int E, float* scratch,
                          LaunchStream st);
int64_t colsum_scratch_floats(int N, int E);
// out = sum of part [splits][n] in order; with out1 and out2 (both) three such arrays after one
// another.
cudaError_t launch_reduce_splits(const float* part, float* out, int64_t n, int splits,
                                 LaunchStream st, float* out1 = nullptr, float* out2 = nullptr);

// ---------------------------------------------------------------- fp32 SIMT GEMM
// C[b] = A[b].B[b], A logical [M][K], B logical [K][N], C [M][N] (row stride c_ld). Each operand
// is contiguous along K (kfast: rows of A, columns of B, `ld` apart) or along its other
// dimension (k rows `ld` apart). With idx, A's rows (kfast) or k rows (else) are gathered:
// row i is row idx[b*idx_bs + i] of A. Forms, by the pointers given:
//   segs == 2       C = A.B + A2.B2 (two K loops, each rounded as its own sum)
//   C2 (no C3, E1)  C = A.B (N columns), C2 = A.B2 (N2 <= N columns, N by default); pairs only
//   C3              a = A.B, b = A.B2: C = a, C2 = b, C3 = silu(a) b
//   E1              dU = A.B with a = E1, b = E2 (layout of C): C = dU b silu'(a), C2 = dU silu(a)
//   splits > 1      (plain) split s of K writes C + s * c_split
struct SimtGemmArgs {
  const float *A = nullptr, *A2 = nullptr;
  int64_t a_bs = 0, a_ld = 0;
  const float *B = nullptr, *B2 = nullptr;
  int64_t b_bs = 0, b_ld = 0;
  const int* idx = nullptr;
  int64_t idx_bs = 0;
  float *C = nullptr, *C2 = nullptr, *C3 = nullptr;
  const float *E1 = nullptr, *E2 = nullptr;
  int64_t c_bs = 0, c_ld = 0, c_split = 0;
  int M = 0, N = 0, N2 = -1, K = 0, batch = 1, splits = 1, segs = 1;
  bool a_kfast = true, b_kfast = false;
  // set by the launcher
  int kchunk = 0;
  bool vec_a = false, vec_b = false, vec_c = false;
};
cudaError_t launch_simt_gemm(SimtGemmArgs a, LaunchStream st);
// Two problems of the C2 form with both operands contiguous off K (the weight gradients), one
// launch.
cudaError_t launch_simt_gemm_pair(SimtGemmArgs a, SimtGemmArgs b, LaunchStream st);

}  // namespace ecmoe
