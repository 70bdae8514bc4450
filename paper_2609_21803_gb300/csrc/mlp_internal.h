// Internal interface of the learned proposal's kernels: the BF16 tensor-core
// GEMM (tcgen05 + TMA + TMEM) and its fused epilogues.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "comet.h"
#include "comet_proposal.h"

namespace comet {
namespace mlp {

// What the GEMM epilogue does with the FP32 accumulator tile D = A B^T
// (A [M][K], B [N][K], both bf16 row-major, i.e. K-major operands).
enum EpiKind : int {
    kEpiStore = 0,      // out_f32[m][n] = D + bias[n]
    kEpiBiasGelu = 1,   // Z = D + bias -> z_f32, H = gelu(Z) -> h (bf16) and h_t (bf16, transposed)
    kEpiGeluGrad = 2,   // G = D * gelu'(z_in) -> h (bf16) and h_t (bf16, transposed)
    kEpiAtomicAdd = 3,  // out_f32[m][n] += D (split-K partial sums)
    kEpiLoss = 4,       // Y = D + bias, G = (2/B) Omega (Y - T) -> h, h_t; loss += Omega (Y - T)^2 / B (training;
                        // aligned rows, N a multiple of 16)
};

struct Epilogue {
    int kind;
    const float* bias;      // [N] (kEpiStore, kEpiBiasGelu; nullable)
    float* out_f32;         // [M][ld_out] (kEpiStore, kEpiAtomicAdd), z (kEpiBiasGelu)
    int64_t ld_out;
    uint16_t* h;            // [M][ld_h] bf16 (kEpiBiasGelu, kEpiGeluGrad; nullable)
    int64_t ld_h;
    uint16_t* h_t;          // [N][ld_ht] bf16, transposed (nullable)
    int64_t ld_ht;
    const float* z_in;      // [M][ld_z] pre-activation (kEpiGeluGrad)
    int64_t ld_z;
    int* err;               // device flag: a bounded wait ran out (nullable)
    // internal uses (zero otherwise)
    float* bias_grad;       // kEpiAtomicAdd: sums of column N - 1 go here instead, one per row
    const float* target;    // kEpiLoss: T, Omega [M][ld_z]
    const float* weight;
    float* loss;            // kEpiLoss: loss sum
    int64_t* step;          // kEpiLoss: the optimiser's step count, advanced once
    float inv_b;            // kEpiLoss: 1 / B
};

// A row-major bf16 matrix [rows][cols] with leading dimension ld (elements);
// the GEMM reduces over cols.
struct Mat {
    const uint16_t* ptr;
    int64_t rows, cols, ld;
};

// D[M][N] = A[M][K] B[N][K]^T over K split into `k_splits` chunks (each a
// multiple of 64; with k_splits > 1 the epilogue must be kEpiAtomicAdd).
// Requirements: ptr 16-byte aligned, ld a multiple of 8, N <= 256 per
// column tile (larger N is tiled), K >= 1.  Returns a CUDA error code.
cudaError_t gemm_bf16(const Mat& A, const Mat& B, int64_t M, int N, int K, int k_splits, const Epilogue& ep,
                      cudaStream_t s);

// Whether kernels on `device` may read the array at v (attributes `at`) where
// it lies, by 16-byte rows: memory of that device itself.  Another GPU's is
// not mapped there without peer access, and managed memory migrates; both are
// copied, as host arrays are.
inline bool usable_in_place(const cudaPointerAttributes& at, int device, const void* v) {
    return at.type == cudaMemoryTypeDevice && at.device == device && (reinterpret_cast<uintptr_t>(v) & 15u) == 0;
}

// Weight and bias gradients of up to kDwMax layers in one launch, added to dw
// and db: dw = G^T H, db = column sums of G, from the transposed copies g_t
// [dout][ld] and h_t [din + 1][ld], whose last row holds ones.  The batch is
// split; split s has places of its own for its bias sums, db + s ld_db, and
// the reader adds the splits up in order, so that a bias gradient does not
// depend on which CTA ends first (a weight's does: its splits are atomic sums).
// dw_splits() is the number of splits of K rows, and splits x the sum of dout
// stays within dw_parts_max().
constexpr int kDwMax = 4;
struct DwLayer {
    const uint16_t* g_t;
    const uint16_t* h_t;
    int64_t ld;
    int dout, din;
    float* dw;
    float* db;
};
int dw_splits(const DwLayer* layers, int n, int64_t K, int num_sms);
int64_t dw_parts_max(int64_t sum_dout, int num_sms);
cudaError_t dw_bf16(const DwLayer* layers, int n, int64_t K, int64_t ld_db, int num_sms, int* err, cudaStream_t s);

// The tensor-map encoder from the driver (resolved once); false if absent.
bool tensor_maps_available();

// Fused forward pass of the 4-layer MLP (width 256): x [M][in_dim] BF16
// (in_dim 64, 128, 192 or 256), w[l] BF16 row-major [out][in] (K-major),
// biases FP32, y [M][ld_y] FP32 (out_dim a multiple of 16, 16-byte rows).
// One persistent CTA per SM (at most num_sms CTAs).
bool fused_forward_fits(int in_dim, int width, int out_dim);
cudaError_t mlp_forward_fused(const uint16_t* x, int64_t M, int in_dim, const uint16_t* const w[4], int out_dim,
                              const float* const bias[4], float* y, int64_t ld_y, int* err, int num_sms,
                              cudaStream_t s);
cudaError_t fused_prepare();

// Raise the GEMM kernel's shared-memory limit to its largest configuration
// on the current device (once; not a stream operation, so later launches
// stay capturable).
cudaError_t gemm_prepare();

}  // namespace mlp

// The proposal's device-side steps used by the learned planner (mlp.cu).
comet_status proposal_reserve_prune(comet_proposal* q, int64_t cap, int keep);
comet_status proposal_prune_device(comet_proposal* q, comet_frontier* f, int keep, float* warm, int* row_scratch,
                                   cudaStream_t s);
comet_status proposal_predict_device(comet_proposal* q, const comet_mode_seq* seqs, int64_t n, float* merit,
                                     float* warm, cudaStream_t s);
// The problem a proposal was created for.
comet_problem* proposal_problem(const comet_proposal* q);

}  // namespace comet
