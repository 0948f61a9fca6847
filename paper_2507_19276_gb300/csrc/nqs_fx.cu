// nqs_fx.cu -- FP64-accurate matrix steps on the tensor cores in fixed point.
//
// GB300 executes two FP64 FMAs per clock and SM; its tensor cores ~3600 FP16
// products. A step y = M x on vectors scaled to a largest magnitude in [0.5, 1)
// is therefore formed from exact integer products, the error-free splitting of
// Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012): every entry becomes
// a 56-bit fixed-point number (per vector, and per output row of the matrix),
// cut into seven signed base-256 digits. Digits are exact in FP16, a product of
// two is at most 2^14, and the sum over D <= 64 terms and the up to seven digit
// pairs of one significance stays below 2^23, so the FP32 accumulators of
// tensor memory hold exact integers. The 28 digit products down to significance
// 2^-62 are kept; the seven sums of a result are joined in 64-bit integers (unit
// 2^-56 of the scale) and rounded to FP64 once. The dropped products and the
// input rounding are ~2^-53 of the scale; a chain of FP64 FMAs over D = 64
// terms rounds its partial sums 64 times.
//
// A tile is 128 items of one matrix (256 threads, two per row): gather and cut
// the rows into digits (bytes of x + 0x80..80, turned into FP16 by PRMT and one
// packed subtraction), 28 x D/16 MMAs, then the integer epilogue. Per tile at
// D = 64 that is ~20 k warp instructions and 112 MMAs, against 301 k cycles of
// the FP64 pipe for the same products.
#include "nqs_fx.cuh"
#include "nqs_tc.cuh"

#include <algorithm>

namespace nqs {

namespace {

constexpr int kFxRows = 128;
constexpr int kFxThreads = 256;

// x 2^55 rounded to an integer, |x| < 1, plus 0x80 in each of the seven bytes:
// byte i (the top one nine bits wide) is digit i + 128.
__device__ __forceinline__ uint64_t fx_code(double x)
{
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FF);
    uint64_t m = (b & 0xFFFFFFFFFFFFFull) | (e ? 1ull << 52 : 0ull);
    const int sh = 1020 - e;                  // x 2^55 = m 2^-sh
    if (sh <= 0) m <<= (-sh) & 3;
    else m = sh > 54 ? 0ull : (m + (1ull << (sh - 1))) >> sh;
    const int64_t v = (int64_t)b < 0 ? -(int64_t)m : (int64_t)m;
    return (uint64_t)(v + 0x80808080808080ll);
}

// digit `i` (0 = least significant) of two codes as FP16
__device__ __forceinline__ __half2 fx_digit2(uint64_t c0, uint64_t c1, int i)
{
    uint32_t w;
    if (i < 6) {
        const uint32_t a = i < 4 ? (uint32_t)c0 : (uint32_t)(c0 >> 32), b = i < 4 ? (uint32_t)c1 : (uint32_t)(c1 >> 32);
        const uint32_t p = __byte_perm(a, b, (uint32_t)((i & 3) | ((4 + (i & 3)) << 8)));   // a's byte, x, b's byte, x
        w = (p & 0x00FF00FFu) | 0x64006400u;
    } else {
        w = (uint32_t)(c0 >> 48) | ((uint32_t)(c1 >> 48) << 16) | 0x64006400u;
    }
    const __half2 k = __half2half2(__ushort_as_half((unsigned short)0x6480));               // 1024 + 128
    return __hsub2(*reinterpret_cast<const __half2*>(&w), k);
}

// One block per (side, matrix): the rows' powers of two, then their digits.
__global__ void __launch_bounds__(256) k_fx_images(const double* __restrict__ A, int n_mats, int D, unsigned char* img,
                                                   int* exps)
{
    __shared__ int se[kFxMaxD];
    const int m = blockIdx.x, side = blockIdx.y, lane = threadIdx.x & 31;
    const double* M = A + (size_t)m * D * D;
    const size_t id = (size_t)side * n_mats + m;
    for (int n = threadIdx.x >> 5; n < D; n += 8) {
        double mx = 0.0;
        int bad = 0;
        for (int k = lane; k < D; k += 32) {
            const double v = fabs(side == 0 ? __ldg(M + (size_t)n * D + k) : __ldg(M + (size_t)k * D + n));
            mx = fmax(mx, v);
            bad |= !(v <= 1.7976931348623157e308);
        }
        mx = warp_max_f64(mx);
        bad = __any_sync(kFull, bad);
        int e = 0;
        if (mx > 0.0) frexp(mx, &e);
        if (lane == 0) {
            se[n] = bad ? 0 : e;
            exps[id * D + n] = bad ? kFxNotFinite : e;
        }
    }
    __syncthreads();
    unsigned char* out = img + id * kFxDigits * 2 * D * D;
    for (int q = threadIdx.x; q < D * (D / 2); q += 256) {
        const int n = q / (D / 2), k = 2 * (q - n * (D / 2));
        const double v0 = side == 0 ? __ldg(M + (size_t)n * D + k) : __ldg(M + (size_t)k * D + n);
        const double v1 = side == 0 ? __ldg(M + (size_t)n * D + k + 1) : __ldg(M + (size_t)(k + 1) * D + n);
        const uint64_t c0 = fx_code(ldexp(v0, -se[n])), c1 = fx_code(ldexp(v1, -se[n]));
        #pragma unroll
        for (int i = 0; i < kFxDigits; ++i)
            *(__half2*)(out + (size_t)(kFxDigits - 1 - i) * 2 * D * D + tc::op_offset(n, k, D)) = fx_digit2(c0, c1, i);
    }
}

// an FP32 accumulator that holds an integer; small: |v| <= 2^22
__device__ __forceinline__ int fx_int(uint32_t w, bool small)
{
    const float v = __uint_as_float(w);
    return small ? __float_as_int(v + 12582912.f) - 0x4B400000 : __float2int_rn(v);
}

template <int D>
__global__ void __launch_bounds__(kFxThreads, D <= 32 ? 2 : 1) k_fx_step(FxStep st)
{
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ uint32_t tmem_slot;
    __shared__ __align__(8) uint64_t mb_mma, mb_b;
    __shared__ int64_t s_src[kFxRows], s_dst[kFxRows];
    __shared__ int64_t s_gb[8], s_ge[8];
    __shared__ int s_tile[9];
    __shared__ int s_eb[D];
    __shared__ int s_max[2][kFxRows];
    __shared__ int s_bad[kFxRows];
    constexpr int H = D / 2;                          // columns per thread in the epilogue
    constexpr uint32_t kA = kFxRows * D * 2;          // one digit of the rows
    constexpr uint32_t kB = 2 * D * D;                // one digit of the matrix
    constexpr uint32_t kCols = kFxDigits * D <= 128 ? 128 : kFxDigits * D <= 256 ? 256 : 512;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned char* const Bs = smraw + kFxDigits * kA;
    if (warp == 0) { tc::tmem_alloc(&tmem_slot, kCols); tc::tmem_relinquish(); }
    if (tid == 0) {
        tc::mbar_init(&mb_mma, 1);
        tc::mbar_init(&mb_b, 1);
        int tiles = 0;
        for (int g = 0; g < 8; ++g) {
            int64_t b, e;
            if (st.items) { b = st.gbeg[g]; e = st.gend[g]; }
            else if ((g >> 2) < st.sides) { b = st.off[g >> 2][g & 3]; e = st.off[g >> 2][(g & 3) + 1]; }
            else b = e = 0;
            s_gb[g] = b;
            s_ge[g] = e;
            s_tile[g] = tiles;
            tiles += (int)((e - b + kFxRows - 1) / kFxRows);
        }
        s_tile[8] = tiles;
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_slot;
    const int r = 32 * (warp & 3) + lane, h = warp >> 2;
    const uint32_t tlane = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(h * H);
    const uint32_t idesc = tc::idesc_f16(kFxRows, D);
    uint32_t ph_mma = 0, ph_b = 0;
    bool ok = true;
    int held = -1;
    constexpr uint32_t kPoll = 1u << 24;
    const int nt = s_tile[8];
    const int tile0 = (int)((int64_t)nt * blockIdx.x / gridDim.x);
    const int tile1 = (int)((int64_t)nt * (blockIdx.x + 1) / gridDim.x);
    for (int tile = tile0; tile < tile1; ++tile) {
        int g = 0;
        while (g < 7 && tile >= s_tile[g + 1]) ++g;
        const int side = g >> 2;
        const int64_t i0 = s_gb[g] + (int64_t)(tile - s_tile[g]) * kFxRows;
        const int n = (int)min((int64_t)kFxRows, s_ge[g] - i0);
        if (tid < kFxRows) {
            int64_t a, b;
            const int64_t i = i0 + (tid < n ? tid : 0);          // rows past n repeat the first
            if (st.items) {
                const uint2 it = __ldg(st.items + i);
                a = it.x;
                b = it.y;
            } else {
                const int64_t s = (int64_t)__ldg(st.list[side] + i) * st.stride;
                a = s + st.src[side];
                b = s + st.dst[side];
            }
            s_src[tid] = a;
            s_dst[tid] = b;
            s_bad[tid] = 0;
        }
        const size_t mat = (size_t)st.mat[side] + (g & 3);
        if (held != g) {
            if (tid == 0) {
                tc::mbar_expect_tx(&mb_b, kFxDigits * kB);
                tc::bulk_g2s(Bs, st.img + mat * kFxDigits * kB, kFxDigits * kB, &mb_b);
            }
            if (tid < D) s_eb[tid] = __ldg(st.exps + mat * D + tid);
        }
        __syncthreads();
        // the rows' digits: eight entries of a row per task, eight rows x four tasks
        // per warp (shared memory in whole core matrices)
        {
            const double* pool = st.pool[side];
            constexpr int TASKS = D / 16;             // per thread: 128 D / 8 / 256
            #pragma unroll
            for (int u = 0; u < TASKS; ++u) {
                const int q = warp + 8 * u;           // (row group, 4 pieces)
                constexpr int PG = D / 8 < 4 ? 1 : D / 32;                   // groups of four pieces per row
                int row, pc;
                if constexpr (D == 16) {              // two pieces per row: sixteen rows per warp
                    row = q * 16 + (lane & 7) + 8 * (lane >> 4);
                    pc = (lane >> 3) & 1;
                } else if constexpr (D == 48) {       // six pieces per row, row-major over the tasks
                    const int x = q * 32 + lane;      // 768 tasks
                    row = (x / 48) * 8 + (x & 7);
                    pc = (x % 48) >> 3;
                } else {
                    row = (q / PG) * 8 + (lane & 7);
                    pc = (q % PG) * 4 + (lane >> 3);
                }
                const double* src = pool + (size_t)s_src[row] * D + 8 * pc;
                uint64_t c[8];
                int bad = 0;
                #pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const double2 v = *(const double2*)(src + 2 * k);
                    bad |= ((__double2hiint(v.x) & 0x7FF00000) == 0x7FF00000) | ((__double2hiint(v.y) & 0x7FF00000) == 0x7FF00000);
                    c[2 * k] = fx_code(v.x);
                    c[2 * k + 1] = fx_code(v.y);
                }
                if (bad) s_bad[row] = 1;
                const uint32_t off = tc::op_offset(row, 8 * pc, D);
                #pragma unroll
                for (int i = 0; i < kFxDigits; ++i) {
                    __align__(16) __half2 d[4];
                    #pragma unroll
                    for (int k = 0; k < 4; ++k) d[k] = fx_digit2(c[2 * k], c[2 * k + 1], i);
                    *(uint4*)(smraw + (kFxDigits - 1 - i) * kA + off) = *(const uint4*)d;
                }
            }
        }
        tc::fence_proxy_async();
        tc::fence_before_sync();
        __syncthreads();
        if (tid == 0) {
            tc::fence_after_sync();
            if (held != g) ok = tc::mbar_wait(&mb_b, ph_b, kPoll) && ok;
            const uint64_t d0 = tc::desc(0, 128, 16 * D);
            const uint64_t dA = d0 + (tc::smem_addr(smraw) >> 4), dB = d0 + (tc::smem_addr(Bs) >> 4);
            for (int l = 0; l < kFxDigits; ++l)       // significance l: digits a of the row, l - a of the matrix
                for (int a = 0; a <= l; ++a)
                    #pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks)
                        tc::mma_f16(tmem + (uint32_t)(l * D), dA + (uint64_t)(a * (kA >> 4) + 16 * ks),
                                    dB + (uint64_t)((l - a) * (kB >> 4) + 16 * ks), idesc, (a | ks) ? 1u : 0u);
            tc::mma_commit(&mb_mma);
        }
        if (held != g) ph_b ^= 1u;
        held = g;
        ok = tc::mbar_wait(&mb_mma, ph_mma, kPoll) && ok;
        ph_mma ^= 1u;
        tc::fence_after_sync();
        // join the seven sums: V = y 2^56 / 2^eb, and the row's largest exponent
        int64_t V[H];
        int emax = -(1 << 29);
        #pragma unroll
        for (int c0 = 0; c0 < H; c0 += 8) {
            uint32_t w[kFxDigits][8];
            #pragma unroll
            for (int l = 0; l < kFxDigits; ++l) tc::tmem_ld8u(tlane + (uint32_t)(l * D + c0), w[l]);
            tc::tmem_wait_ld();
            #pragma unroll
            for (int c = 0; c < 8; ++c) {
                int s[kFxDigits];
                #pragma unroll
                for (int l = 0; l < kFxDigits; ++l) s[l] = fx_int(w[l][c], (l + 1) * D <= 256);
                const int64_t hi = (int64_t)(s[0] * 256 + s[1]) * 65536 + (s[2] * 256 + s[3]);
                const int64_t lo = (int64_t)(s[4] * 256 + s[5]) * 256 + s[6];
                const int64_t v = (hi << 18) + ((lo + 32) >> 6);
                V[c0 + c] = v;
                const int eb = s_eb[h * H + c0 + c];
                if (v != 0) emax = max(emax, 64 - __clzll(v < 0 ? -v : v) + eb);
                if (eb == kFxNotFinite) emax = kFxNotFinite;
            }
        }
        s_max[h][r] = emax;
        tc::fence_before_sync();
        __syncthreads();                              // the two halves of each row meet
        emax = max(s_max[0][r], s_max[1][r]);
        if (r < n) {
            double* dst = st.pool[side] + (size_t)s_dst[r] * D + h * H;
            const bool bad = s_bad[r] != 0 || emax >= kFxNotFinite;
            #pragma unroll
            for (int c = 0; c < H; c += 2) {
                double o[2];
                #pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int64_t v = V[c + k];
                    const uint64_t mag = (uint64_t)(v < 0 ? -v : v);
                    const int L = 64 - __clzll((long long)mag);
                    const int f = 1022 + L + s_eb[h * H + c + k] - emax;       // exponent field
                    uint64_t m = L <= 53 ? mag << (53 - L) : (mag + (1ull << (L - 54))) >> (L - 53);
                    uint64_t bits = ((uint64_t)(f - 1) << 52) + m;
                    if (mag == 0 || f <= 0) bits = 0;
                    bits |= (uint64_t)v & 0x8000000000000000ull;
                    o[k] = bad ? __longlong_as_double(0x7FF8000000000000ll) : __longlong_as_double((long long)bits);
                }
                *(double2*)(dst + c) = make_double2(o[0], o[1]);
            }
            if (h == 0) {
                const int* se = st.pool_e[side] + s_src[r];
                st.pool_e[side][s_dst[r]] = *se + (emax < -(1 << 28) || bad ? 0 : emax - 56);
            }
        }
        __syncthreads();                              // the lists, maxima and digits are free
    }
    if (!ok && tid == 0) report(st.err, 5, 4, (long long)blockIdx.x);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tmem, kCols);
}

// rows of the unit vector e_0 with power 0
__global__ void k_fx_unit_rows(double* rows, int* exps, int64_t n, int64_t stride, int64_t at, int D)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n * D) return;
    const int64_t s = q / D;
    const int c = (int)(q - s * D);
    rows[(s * stride + at) * D + c] = c == 0 ? 1.0 : 0.0;
    if (c == 0) exps[s * stride + at] = 0;
}

__global__ void k_fx_first(const double* rows, const int* exps, int64_t n, int64_t stride, int64_t at, int D, double* mant,
                           int* ex)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    mant[s] = rows[(s * stride + at) * D];
    ex[s] = exps[s * stride + at];
}

// log|psi| and its sign from psi_TN = mant 2^ex, a warp per determinant
__global__ void __launch_bounds__(256) k_fx_log_psi(AnsatzView an, const uint64_t* dets, int64_t n, const double* mant,
                                                    const int* ex, double* log_abs, int8_t* sign)
{
    const int64_t id = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (id >= n) return;
    const uint64_t na = dets[2 * id], nb = dets[2 * id + 1];
    double lf = 0.0;
    int odd = 0;
    for (int k = lane; k < an.n_hidden; k += 32) {
        const double th = corr_theta(an, k, na, nb);
        lf += corr_log_factor(an.corr, th);
        if (an.corr != 0) odd ^= cos(th) < 0.0;
    }
    lf = warp_sum_f64(lf);
    odd = (int)__popc(__ballot_sync(kFull, odd & 1)) & 1;
    if (lane == 0) {
        const double m = mant[id];
        if (m == 0.0 || lf == -INFINITY) { sign[id] = 0; log_abs[id] = -INFINITY; }
        else {
            sign[id] = ((m < 0) ^ odd) ? -1 : 1;
            log_abs[id] = log(fabs(m)) + (double)ex[id] * 0.69314718055994530942 + lf;
        }
    }
}

template <int D>
void fx_launch(const FxStep& s, int64_t tiles, int n_sm, cudaStream_t st)
{
    const size_t smem = (size_t)kFxDigits * (kFxRows * D * 2 + 2 * D * D);
    allow_max_smem(k_fx_step<D>);
    const int per = D <= 16 ? 2 : D <= 32 ? 2 : 1;    // 512 tensor-memory columns per SM
    k_fx_step<D><<<(unsigned)std::min<int64_t>(tiles, (int64_t)per * n_sm), kFxThreads, smem, st>>>(s);
}

}  // namespace

int launch_fx_images(const double* A, int n_mats, int D, unsigned char* img, int* exps, cudaStream_t st)
{
    k_fx_images<<<dim3((unsigned)n_mats, 2), 256, 0, st>>>(A, n_mats, D, img, exps);
    return 1;
}

int launch_fx_step(const FxStep& s, int D, int n_sm, cudaStream_t st)
{
    int64_t tiles = 0;
    if (s.items) {
        for (int g = 0; g < 8; ++g) tiles += (s.gend[g] - s.gbeg[g] + kFxRows - 1) / kFxRows;
    } else {
        tiles = s.sides * ((s.n + kFxRows - 1) / kFxRows + 3);       // at most: four groups, one part tile each
    }
    if (tiles == 0) return 0;
    switch (D) {
    case 16: fx_launch<16>(s, tiles, n_sm, st); break;
    case 32: fx_launch<32>(s, tiles, n_sm, st); break;
    case 48: fx_launch<48>(s, tiles, n_sm, st); break;
    default: fx_launch<64>(s, tiles, n_sm, st); break;
    }
    return 1;
}

int launch_fx_unit_rows(double* rows, int* exps, int64_t n, int64_t stride, int64_t at, int D, cudaStream_t st)
{
    k_fx_unit_rows<<<(unsigned)((n * D + 255) / 256), 256, 0, st>>>(rows, exps, n, stride, at, D);
    return 1;
}

int launch_fx_first(const double* rows, const int* exps, int64_t n, int64_t stride, int64_t at, int D, double* mant, int* ex,
                    cudaStream_t st)
{
    k_fx_first<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(rows, exps, n, stride, at, D, mant, ex);
    return 1;
}

int launch_fx_log_psi(const AnsatzView& an, const uint64_t* dets, int64_t n, const double* mant, const int* ex,
                      double* log_abs, int8_t* sign, cudaStream_t st)
{
    k_fx_log_psi<<<(unsigned)((n + 7) / 8), 256, 0, st>>>(an, dets, n, mant, ex, log_abs, sign);
    return 1;
}

}  // namespace nqs
