// Dense same-spin products on tcgen05 tensor cores (see gemm_tc.cu).
#pragma once
#include "common.cuh"

namespace kpm {

// Row pitch (elements) of an FP16 matrix with `cols` columns: 16-byte rows.
int64_t half_pitch(int64_t cols);

// Columns of a block that the tensor-core sigma takes in one set of launches: three (x, y
// and z of a request) up to 2^24 determinants, where one column's tiles leave a last wave
// half empty or (below 13 orbitals) most SMs idle; their split copies take 8 bytes per
// column and determinant (12 for BF16).
inline int batch_columns(int64_t dim) { return dim <= ((int64_t)1 << 24) ? 3 : 1; }

// sigma += F_b-part + F_a-part of H applied to x (FP32 [N_a][N_b]); see gemm_tc.cu.
struct DenseSS {
    int64_t na = 0, nb = 0, pa = 0, pb = 0;   // strings and FP16 row pitches per spin
    double wscale_a = 1.0, wscale_b = 1.0;    // power-of-two scales of the split matrices
    DevBuf fa_hi_own, fa_lo_own;              // alpha matrices (own copy if N_a != N_b)
    DevBuf fb_hi, fb_lo;                      // beta matrices
    DevBuf* fa_hi = nullptr;
    DevBuf* fa_lo = nullptr;
    int64_t xpitch = 0;                       // row pitch of xh/xl: N_b rounded up to 128
    DevBuf xh, xl, th, tl;                    // split copies of x and x^T (TcSigma::hold)
    DevBuf fmax;                              // scratch for max |F_off|
    // per tile of the split matrix, the k-blocks that hold a nonzero (CSR; see
    // block_lists): F_b by pairs of 128-row tiles, F_a by 256-row tiles
    DevBuf kbs_b, kbl_b, kbs_a, kbl_a;
    int64_t kb_nonzero[2] = {0, 0}, kb_total[2] = {0, 0};
    int nsm = 0;                              // SMs of the device
    int* err = nullptr;
    // exact diagonal H_II of the whole H (same-spin diagonals and the opposite-spin
    // Coulomb sum, FP64 stored as float hi + lo, [N_a][N_b]), added by the
    // product's epilogue; the split matrices and the row pass leave it out
    const float2* diag_full = nullptr;

    // Builds the split matrices; `same`: alpha and beta strings are identical.
    void init(const SpinTables& A, const SpinTables& B, bool same, int* err_flag,
              cudaStream_t st);
    // Split copies of the operand, scaled FP16 pieces with zero padding, written by the
    // caller (k_prepare): rows of x [nc][N_a][xpitch] in xh/xl, of x^T [nc][N_b][pa] in th/tl.
    size_t x_bytes(int nc) const { return (size_t)nc * na * xpitch * 2; }   // each of xh, xl
    size_t t_bytes(int nc) const { return (size_t)nc * nb * pa * 2; }       // each of th, tl
    // y += (F_a (x) 1 + 1 (x) F_b) x with the off-diagonal parts of F_a, F_b, plus
    // diag_full * x (the whole exact diagonal of H); amax = device max|x|.
    // Reads xh/xl and th/tl, not x's own entries, in the products.
    void apply(const float* x, float* y, const float* amax, int nc, cudaStream_t st);
    // Rasterisation group (row tiles per group), chosen by autotune() at set-up; 16 by
    // default.
    int group_m = 16;
    void autotune(cudaStream_t st);
    void launch(const float* x, float* y, const float* amax, int nc, int group, cudaStream_t st);
    // Columns (N) of the GEMM's tiles for nc columns of a block: 256, 128 or 64.
    int tile_columns(int nc) const;
};

}  // namespace kpm
