// nqs_fx.cuh -- FP64-accurate matrix steps on the tensor cores in fixed point
// (see nqs_fx.cu).
#pragma once

#include "nqs_tree.cuh"

namespace nqs {

constexpr int kFxDigits = 7;              // base-256 digits of a 56-bit fixed-point number
constexpr int kFxMaxD = 64;

// chains the fixed-point steps take
inline bool fx_fits(int D) { return D % 16 == 0 && D >= 16 && D <= kFxMaxD; }

// Digit images of a chain's site matrices: per (side, site, local state) -- side
// 0: y = M x, side 1: y = x^T M -- kFxDigits FP16 matrices of D x D (K-major
// core matrices, most significant first), and the powers of two of its columns,
// then of its rows ([2][D]; kFxNotFinite: the row holds an infinity or a NaN), then
// a mask per row of its large and of its nonzero entries ([2][D] words of 64 bits).
constexpr int kFxNotFinite = 1 << 28;
__host__ __device__ constexpr int fx_exp_stride(int D) { return 6 * D; }
// sides = 1: side 0 alone (a graph's edges).
inline size_t fx_image_bytes(int n_mats, int D, int sides) { return (size_t)sides * n_mats * kFxDigits * 2 * D * D; }
int launch_fx_images(const double* A, int n_mats, int D, int sides, unsigned char* img, int* exps, cudaStream_t st);

// One product per item: row `src` times the group's matrix into row `dst`,
// renormalised to a largest magnitude in [0.5, 1), its power of two added to the
// source's. Groups 0..3 are side 0 and 4..7 side 1, by local state.
struct FxStep {
    int K;
    int mat[2];                           // matrix block (side * K + site) * 4 of each side
    const unsigned char* img; const int* exps;
    const double* at[2];                  // the FP64 matrices, by side: AT (y_c = sum_k x_k at[k][c]), A
    double* pool[2]; int* pool_e[2];      // by side: rows of D, their exponents
    // items of a group: (src, dst) rows ...
    const uint2* items;
    int64_t gbeg[8], gend[8];
    // ... or (items NULL) samples list[side][off[side][g] ..], whose rows are
    // sample * stride + src[side] and + dst[side]
    const int32_t* list[2]; const int64_t* off[2];
    int64_t stride, src[2], dst[2];
    int64_t n;                            // samples of a list (bounds the grid)
    int sides;                            // list form: 1 (side 0 only) or 2
    DevError* err;
};
int launch_fx_step(const FxStep& s, int D, int n_sm, cudaStream_t st);

// vertex t of the nodes of level t (FP64 graph states, see TreeGraph64)
int launch_fx_graph(const TreeGraph64& a, const unsigned char* img, const int* exps, DevError* err, int t, int deg,
                    const TreeLevels& lv, const int64_t* bounds, int n_sm, cudaStream_t st);

// the normalised readout's candidate cells (see TreeRnn): images of a site's four
// matrices, widths whose tile fits shared memory
constexpr int kFxRnnMaxD = 24;
inline size_t fx_rnn_image_bytes(int K, int D)
{
    return (size_t)K * ((4 * D + 31) / 32) * kFxDigits * 64 * (D <= 16 ? 16 : 32);
}
__host__ __device__ constexpr int fx_rnn_exp_stride(int KP) { return KP + 128 + 2 * 2 * 128; }
inline size_t fx_rnn_exps(int K, int D) { return (size_t)K * fx_rnn_exp_stride(D <= 16 ? 16 : 32); }
int launch_fx_rnn_images(const double* A, const double* v, int K, int D, unsigned char* img, int* exps, cudaStream_t st);
int launch_fx_rnn(const TreeRnn& a, const unsigned char* img, const int* exps, DevError* err, int t, const TreeLevels& lv,
                  const int64_t* bounds, int n_sm, cudaStream_t st);

// outer-product partial sums of the gradient (k_grad_tn's, for the widths of fx_fits)
int launch_fx_grad(const GradArgs& a, int64_t chunks, int chunk_samples, DevError* err, cudaStream_t st);

// row `at` of every sample (stride rows each) set to e_0 with power 0
int launch_fx_unit_rows(double* rows, int* exps, int64_t n, int64_t stride, int64_t at, int D, cudaStream_t st);
// first entries and powers of those rows
int launch_fx_first(const double* rows, const int* exps, int64_t n, int64_t stride, int64_t at, int D, double* mant, int* ex,
                    cudaStream_t st);
// log|psi| and sign of n determinants from psi_TN = mant 2^ex and the correlator
int launch_fx_log_psi(const AnsatzView& an, const uint64_t* dets, int64_t n, const double* mant, const int* ex,
                      double* log_abs, int8_t* sign, cudaStream_t st);

}  // namespace nqs
