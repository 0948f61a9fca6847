// nqs_ansatz.cu -- the working forms of an ansatz's parameters, made on the
// device from the FP64 site tensors each time they are set: transposed, FP32
// and (hi, lo) float-pair copies, the split-FP16 operand images of the
// tensor-core paths (chain and graph) and the transposed FP32 correlator
// weights. A training loop sets the ansatz on every step, so this is on its
// path: formed on the host (single thread, D2H and H2D copies around it) the
// forms of H50's D = 64 chain took 34 ms of a 46 ms log|psi| step; the two
// kernels below read 6.5 MB and write ~40 MB, DRAM- and launch-bound (~20 us).
#include "nqs_kernels.cuh"
#include "nqs_family.cuh"
#include "nqs_tc.cuh"

namespace nqs {

namespace {

// Power of two of every matrix: e with max|entry| 2^-e in [0.5, 1) (0 for a
// zero matrix), one block per matrix; out1 (may be NULL) gets a second copy.
__global__ void __launch_bounds__(256) k_mat_exps(const double* __restrict__ A, int DD, int* out0, int* out1)
{
    __shared__ double sh[8];
    const double* M = A + (size_t)blockIdx.x * DD;
    double m = 0.0;
    for (int i = threadIdx.x; i < DD; i += 256) m = fmax(m, fabs(__ldg(M + i)));
    m = warp_max_f64(m);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) m = fmax(m, sh[w]);
        int e = 0;
        if (m > 0.0) frexp(m, &e);
        out0[blockIdx.x] = e;
        if (out1) out1[blockIdx.x] = e;
    }
}

__device__ __forceinline__ float2 pair_of(double x)
{
    const float h = (float)x;                    // 48 of the entry's 53 bits
    return make_float2(h, (float)(x - (double)h));
}

// split half images: element (row n, reduction index k) of an operand whose
// rows are `C` columns wide, hi at `hi`, lo at `lo` (K-major core matrices)
__device__ __forceinline__ void put_split(unsigned char* hi, unsigned char* lo, int n, int k, int C, float v)
{
    __half h, l;
    tc::split_half(v, h, l);
    const uint32_t off = tc::op_offset(n, k, C);
    *(__half*)(hi + off) = h;
    *(__half*)(lo + off) = l;
}

// One 32 x 32 tile of one matrix per block, the transposed forms through
// shared memory so that both directions store whole lines.
__global__ void __launch_bounds__(256) k_mat_forms(AnsatzForms f)
{
    __shared__ double t[32][33];
    const int D = f.D, m = blockIdx.z;
    const size_t mo = (size_t)m * D * D;
    const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int x = f.exps ? f.exps[m] : 0;
    for (int k = ty; k < 32; k += 8) {
        const int r = r0 + k, c = c0 + tx;
        if (r >= D || c >= D) continue;
        const double v = __ldg(f.A + mo + (size_t)r * D + c);
        t[k][tx] = v;
        f.Af[mo + (size_t)r * D + c] = (float)v;
        if (f.Adf) f.Adf[mo + (size_t)r * D + c] = pair_of(v);
        if (f.chain_img) {                       // side 0: B[n][k] = M[n][k]
            const int ck = c / f.kc, kk = c - ck * f.kc;
            unsigned char* hi = f.chain_img + (size_t)m * 4 * D * D + (size_t)ck * 4 * D * f.kc;
            put_split(hi, hi + (size_t)2 * D * f.kc, r, kk, f.kc, (float)ldexp(v, -x));
        }
        if (f.graph_img) {                       // per edge, rows sigma D + n
            const int e = m >> 2, sg = m & 3;
            unsigned char* hi = f.graph_img + (size_t)e * 16 * D * D + (size_t)sg * 2 * D * D;
            put_split(hi, hi + (size_t)8 * D * D, r, c, D, (float)ldexp(v, -x));
            if (c == 0) f.col0[(size_t)m * D + r] = (float)v;
        }
    }
    __syncthreads();
    for (int k = ty; k < 32; k += 8) {
        const int r = r0 + tx, c = c0 + k;       // element (r, c), written at [c][r]
        if (r >= D || c >= D) continue;
        const double v = t[tx][k];
        f.AT[mo + (size_t)c * D + r] = v;
        f.ATf[mo + (size_t)c * D + r] = (float)v;
        if (f.ATdf) f.ATdf[mo + (size_t)c * D + r] = pair_of(v);
        if (f.chain_img) {                       // side 1: B[n][k] = M[k][n]
            const int ck = r / f.kc, kk = r - ck * f.kc;
            unsigned char* hi = f.chain_img + ((size_t)f.n_mats + m) * 4 * D * D + (size_t)ck * 4 * D * f.kc;
            put_split(hi, hi + (size_t)2 * D * f.kc, c, kk, f.kc, (float)ldexp(v, -x));
        }
    }
}

// W [n_hidden][2K] in FP32 transposed, [2K][np] with zero columns past n_hidden
__global__ void k_corr_transpose(const double* __restrict__ W, int n_hidden, int np, int K2, float* WTf)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= K2 * np) return;
    const int s = q / np, k = q - s * np;
    WTf[q] = k < n_hidden ? (float)__ldg(W + (size_t)k * K2 + s) : 0.f;
}

}  // namespace

int launch_ansatz_forms(const AnsatzForms& f, cudaStream_t st)
{
    int n = 0;
    if (f.exps) {
        k_mat_exps<<<(unsigned)f.n_mats, 256, 0, st>>>(f.A, f.D * f.D, f.exps, f.exps2);
        ++n;
    }
    const unsigned nt = (unsigned)((f.D + 31) / 32);
    k_mat_forms<<<dim3(nt, nt, (unsigned)f.n_mats), 256, 0, st>>>(f);
    return n + 1;
}

int launch_corr_transpose(const double* W, int n_hidden, int np, int K2, float* WTf, cudaStream_t st)
{
    k_corr_transpose<<<(unsigned)((K2 * np + 255) / 256), 256, 0, st>>>(W, n_hidden, np, K2, WTf);
    return 1;
}

}  // namespace nqs
