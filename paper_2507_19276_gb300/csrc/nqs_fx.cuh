// nqs_fx.cuh -- FP64-accurate matrix steps on the tensor cores in fixed point
// (see nqs_fx.cu).
#pragma once

#include "nqs_kernels.cuh"

namespace nqs {

constexpr int kFxDigits = 7;              // base-256 digits of a 56-bit fixed-point number
constexpr int kFxMaxD = 64;

// chains the fixed-point steps take
inline bool fx_fits(int D) { return D % 16 == 0 && D >= 16 && D <= kFxMaxD; }

// Digit images of a chain's site matrices: per (side, site, local state) -- side
// 0: y = M x, side 1: y = x^T M -- kFxDigits FP16 matrices of D x D (K-major
// core matrices, most significant first), and per output row its power of two
// (kFxNotFinite: the row holds an infinity or a NaN).
constexpr int kFxNotFinite = 1 << 28;
inline size_t fx_image_bytes(int n_mats, int D) { return (size_t)2 * n_mats * kFxDigits * 2 * D * D; }
int launch_fx_images(const double* A, int n_mats, int D, unsigned char* img, int* exps, cudaStream_t st);

// One product per item: row `src` times the group's matrix into row `dst`,
// renormalised to a largest magnitude in [0.5, 1), its power of two added to the
// source's. Groups 0..3 are side 0 and 4..7 side 1, by local state.
struct FxStep {
    int K;
    int mat[2];                           // matrix block (side * K + site) * 4 of each side
    const unsigned char* img; const int* exps;
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

// row `at` of every sample (stride rows each) set to e_0 with power 0
int launch_fx_unit_rows(double* rows, int* exps, int64_t n, int64_t stride, int64_t at, int D, cudaStream_t st);
// first entries and powers of those rows
int launch_fx_first(const double* rows, const int* exps, int64_t n, int64_t stride, int64_t at, int D, double* mant, int* ex,
                    cudaStream_t st);
// log|psi| and sign of n determinants from psi_TN = mant 2^ex and the correlator
int launch_fx_log_psi(const AnsatzView& an, const uint64_t* dets, int64_t n, const double* mant, const int* ex,
                      double* log_abs, int8_t* sign, cudaStream_t st);

}  // namespace nqs
