// nqs_fx.cu -- FP64-accurate matrix steps on the tensor cores in fixed point.
//
// GB300 executes two FP64 FMAs per clock and SM; its tensor cores ~3600 FP16
// products. A step y = M x is therefore formed from exact integer products, the
// error-free splitting of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59,
// 2012). The matrix is equilibrated by powers of two, first its columns, then
// its rows; the vector takes the column powers and is scaled to a largest
// magnitude in [0.5, 1) (so a power-of-two change of basis between two sites
// changes nothing). Every entry becomes a 56-bit fixed-point number, cut into
// seven signed base-256 digits. Digits are exact in FP16, a product of two is at
// most 2^14, and the sum over D <= 64 terms and the up to seven digit pairs of
// one significance stays below 2^23, so the FP32 accumulators of tensor memory
// hold exact integers. The 34 digit products down to significance 2^-70 are
// kept; the eight sums of a result are joined in 64-bit integers (unit 2^-56 of
// the scale) and rounded to FP64 once. The remaining error, the rounding of the
// entries and of the result, is ~2^-56 sqrt(D) of the scale (at most ~D 2^-55);
// a chain of FP64 FMAs rounds its partial sums D times at 2^-53. On dense random
// matrices that is the smaller error. Results whose terms may all lie far below the
// scale are found by bit masks and redone in FP64 (see kFxTerm).
//
// A tile is 128 items of one matrix (two or four threads per row): gather and cut
// the rows into digits (bytes of x + 0x80..80, turned into FP16 by PRMT and one
// packed subtraction), 34 x D/16 MMAs, then the integer epilogue. Per tile at
// D = 64 that is ~20 k warp instructions and 136 MMAs, against 301 k cycles of
// the FP64 pipe for the same products. H50 tables of 200 samples (5 M products):
// 45 ms on the FP64 pipe, 4.9 ms here; issue and latency of the digit and
// epilogue chains bound it (one block per SM at D = 64).
#include "nqs_fx.cuh"
#include "nqs_tc.cuh"

#include <algorithm>

namespace nqs {

namespace {

constexpr int kFxRows = 128;
constexpr int kFxSums = 8;                // significances kept
// threads per row: four at D = 64, where one block fills the SM
// (more warps hide the digit and epilogue chains), else two
constexpr int fx_split(int D) { return D == 64 ? 4 : 2; }

// x 2^(55 + off) rounded to an integer, |x 2^off| < 1, plus 0x80 in each of the
// seven bytes: byte i (the top one nine bits wide) is digit i + 128.
__device__ __forceinline__ uint64_t fx_code(double x, int off)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t e = (hi >> 20) & 0x7FFu;
    const uint32_t mh = (hi & 0xFFFFFu) | (min(e, 1u) << 20);
    // the mantissa left-justified, x = m 2^(e - 1086), then x 2^(56 + off) (0 where
    // the shift passes the word), rounded by its last bit
    const uint64_t m = ((uint64_t)__funnelshift_l(lo, mh, 11) << 32) | (lo << 11);
    uint64_t v;
    asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"(1030u - e - (uint32_t)off));
    v = (v + 1) >> 1;
    const uint64_t sg = (uint64_t)((int64_t)(int32_t)hi >> 31);
    return (v ^ sg) + (0x80808080808080ull - sg);
}

constexpr int kFxNoExp = -(1 << 20);          // power of two of a zero

// e with |x| in [2^(e-1), 2^e)
__device__ __forceinline__ int fx_exp(double x)
{
    const int e = (__double2hiint(x) >> 20) & 0x7FF;
    return e ? e - 1022 : kFxNoExp;
}

__device__ __forceinline__ bool fx_not_finite(double x) { return (__double2hiint(x) & 0x7FF00000) == 0x7FF00000; }
__device__ __forceinline__ bool fx_nonzero(double x) { return ((__double2hiint(x) & 0x7FFFFFFF) | __double2loint(x)) != 0; }

// The unit of a result is 2^-56 of (row scale) x (matrix row scale), so its digits
// hold it as well as FP64 would only if one of its terms is near that scale: where
// the large entries of a graded state meet the small ones of the matrix row, an FP64
// chain keeps 53 bits of what is there and the digits few or none. A term of at least
// 2^-kFxTerm of the scale is known to be there if entries of at least 2^-(kFxTerm / 2)
// meet in the state and the matrix row (a bit mask each; for dense rows, also beside a
// unit diagonal, that holds practically always), or if the result itself reaches
// 2^-kFxTerm. Any other result with a nonzero term (two more masks) is redone with
// FP64 FMAs, as are those that an infinity or a NaN takes part in. The masks cost four
// instructions per entry and per result; a small result is looked at by its thread alone.
// What stays errs by at most ~D 2^-55 of the scale, that is D 2^-47 of its largest
// term where FP64 FMAs err by up to D 2^-53 of the sum of the terms. Of the results of
// I + G / sqrt(D) matrices, kFxTerm = 4 redoes 5% (H50's log|psi| 4.2 -> 18 ms), 6
// 0.6% (6.4 ms), 8 none but those of the first site's e_0.
constexpr int kFxTerm = 8;
__device__ __forceinline__ bool fx_is_big(int e) { return e > -(kFxTerm / 2); }      // e as fx_exp's: |x| >= 2^(e-1)

// exponent as fx_exp's of any finite nonzero number, kFxNoExp of the others
__device__ __forceinline__ int fx_top(double y)
{
    const int f = (__double2hiint(y) >> 20) & 0x7FF;
    if (f > 0) return f < 0x7FF ? f - 1022 : kFxNoExp;
    int e = kFxNoExp;
    if (fx_nonzero(y)) frexp(y, &e);
    return e;
}

// |v| < 2^bits (bits > 32; -2^bits passes too): the high word alone
__device__ __forceinline__ bool fx_below(int64_t v, int bits)
{
    return (uint32_t)(v >> 32) + (1u << (bits - 32)) < 2u << (bits - 32);
}

// an entry's digits (see fx_code) are those of a large one, |x| >= 2^-(kFxTerm / 2) up to
// 2^-19 of that: its high word is out of -2^h .. 2^h, h = 55 - kFxTerm / 2 - 32
__device__ __forceinline__ bool fx_code_big(uint64_t c)
{
    constexpr uint32_t kBig = 1u << (55 - kFxTerm / 2 - 32);
    return (uint32_t)(c >> 32) - 0x808080u + kBig >= 2u * kBig;
}

// the candidates among a thread's H results (columns h H ..), small (`below`) or not finite,
// of a row with the masks mb and mz of its large and nonzero entries (the columns' in s_m,
// Z words apart): those that share a nonzero entry and no large one
template <int H, int Z>
__device__ __forceinline__ uint32_t fx_low(uint32_t below, bool not_finite, uint64_t mb, uint64_t mz, const uint64_t* s_m,
                                           const int* s_eb, int h)
{
    uint32_t low = 0;
    // (a warp nearly always has one small result, a thread seldom two: a loop over them)
    for (uint32_t m = not_finite ? (H < 32 ? (1u << (H & 31)) - 1u : ~0u) : below; m; m &= m - 1) {
        const int c = __ffs((int)m) - 1, col = h * H + c;
        if (!(s_m[col] & mb) && ((((below >> c) & 1u) && (s_m[col + Z] & mz)) || s_eb[col] == kFxNotFinite)) low |= 1u << c;
    }
    return low;
}

// entry c of M x in FP64 (M by columns, as dot_col4): nz and mz are the masks of the
// nonzero entries of x and of row c, `whole` where either holds an infinity or a NaN
__device__ __forceinline__ double fx_dot(const double* M, const double* x, int D, int c, uint64_t nz, uint64_t mz, bool whole)
{
    if (!whole && !(nz & mz)) return 0.0;
    if (whole || (nz & (nz - 1))) return dot_col4(M, x, D, c);
    const int k = __ffsll((long long)nz) - 1;         // a state of one entry (the first site's e_0)
    return __ldg(M + (size_t)k * D + c) * x[k];
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
        w = __byte_perm((uint32_t)(c0 >> 32), (uint32_t)(c1 >> 32), 0x7632) | 0x64006400u;
    }
    const __half2 k = __half2half2(__ushort_as_half((unsigned short)0x6480));               // 1024 + 128
    return __hsub2(*reinterpret_cast<const __half2*>(&w), k);
}

// One block per (matrix, side): the columns' powers of two, the rows' after them,
// then the digits. A column without entries has the power kFxNoExp, so that the
// vector's entry there, which meets only zeros, takes no part in its scale. The operand
// has `rows` rows of D entries (columns past D, up to C, and rows past `rows`, up to R,
// are zero) in blocks of R rows: entry(n, k) of the matrix.
template <class Entry>
__device__ void fx_image(const Entry& entry, int rows, int D, int R, int C, unsigned char* img, int* cexp, int* rexp,
                         uint64_t* big, uint64_t* nonzero, int* sc, int* sr)
{
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x; k < C; k += blockDim.x) {
        int e = kFxNoExp;
        if (k < D)
            for (int n = 0; n < rows; ++n) {
                const double v = entry(n, k);
                if (!fx_not_finite(v)) e = max(e, fx_exp(v));
            }
        sc[k] = e == kFxNoExp ? 0 : e;
        cexp[k] = e;                              // kFxNoExp: an empty column, out of the vector's scale
    }
    __syncthreads();
    const int RT = (rows + R - 1) / R * R;
    for (int n = threadIdx.x >> 5; n < RT; n += blockDim.x >> 5) {
        int e = kFxNoExp, bad = 0;
        for (int k = lane; k < D && n < rows; k += 32) {
            const double v = entry(n, k);
            if (fx_not_finite(v)) bad = 1;
            else if (v != 0.0) e = max(e, fx_exp(v) - sc[k]);
        }
        e = __reduce_max_sync(kFull, e);
        bad = __any_sync(kFull, bad);
        e = e <= kFxNoExp / 2 ? 0 : e;
        uint64_t mb = 0, mz = 0;
        for (int k0 = 0; k0 < C; k0 += 32) {
            const int k = k0 + lane;
            const double v = n < rows && k < D ? entry(n, k) : 0.0;
            const int x = k < C ? fx_exp(v) - sc[k] - e : kFxNoExp;
            mb |= (uint64_t)__ballot_sync(kFull, !bad && fx_is_big(x)) << k0;
            mz |= (uint64_t)__ballot_sync(kFull, fx_nonzero(v)) << k0;
        }
        if (lane == 0) {
            sr[n] = e;
            rexp[n] = bad ? kFxNotFinite : e;
            big[n] = mb;
            nonzero[n] = mz;
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < RT * (C / 2); q += blockDim.x) {
        const int n = q / (C / 2), k = 2 * (q - n * (C / 2));
        const double v0 = n < rows && k < D ? entry(n, k) : 0.0, v1 = n < rows && k + 1 < D ? entry(n, k + 1) : 0.0;
        const uint64_t c0 = fx_code(v0, -sc[k] - sr[n]), c1 = fx_code(v1, -sc[k + 1] - sr[n]);
        unsigned char* out = img + (size_t)(n / R) * kFxDigits * 2 * R * C;
        #pragma unroll
        for (int i = 0; i < kFxDigits; ++i)
            *(__half2*)(out + (size_t)(kFxDigits - 1 - i) * 2 * R * C + tc::op_offset(n % R, k, C)) = fx_digit2(c0, c1, i);
    }
}

__global__ void __launch_bounds__(256) k_fx_images(const double* __restrict__ A, int n_mats, int D, unsigned char* img,
                                                   int* exps)
{
    __shared__ int sc[kFxMaxD], sr[kFxMaxD];
    const int m = blockIdx.x, side = blockIdx.y;
    const double* M = A + (size_t)m * D * D;
    const size_t id = (size_t)side * n_mats + m;
    int* const x = exps + id * fx_exp_stride(D);
    uint64_t* const masks = (uint64_t*)(x + 2 * D);
    fx_image([&](int n, int k) { return side == 0 ? __ldg(M + (size_t)n * D + k) : __ldg(M + (size_t)k * D + n); }, D, D, D, D,
             img + id * kFxDigits * 2 * D * D, x, x + D, masks, masks + D, sc, sr);
}

// The eight sums of a result (FP32 accumulators that hold integers) as an integer
// of unit 2^-(56 - drop). A sum of at most 2^22 is read from the low bits of
// v + 1.5 2^23 (their common offset comes off once per pair), a larger one converted.
template <int RED>
__device__ __forceinline__ int64_t fx_join(const uint32_t* w, int drop)
{
    constexpr uint32_t kOff = 0x4B400000u;        // bits of 1.5 2^23
    uint32_t s[kFxSums];
    #pragma unroll
    for (int l = 0; l < kFxSums; ++l) {
        const float v = __uint_as_float(w[l]);
        // (l + 1, at most 7) digit pairs of RED terms of at most 2^14 each
        const bool small = (l < kFxDigits ? l + 1 : 2 * kFxDigits - 1 - l) * RED <= 256;
        s[l] = small ? (uint32_t)__float_as_int(v + 12582912.f) : (uint32_t)__float2int_rn(v) + kOff;
    }
    const int a = (int)(s[0] * 256u + s[1] - 257u * kOff), b = (int)(s[2] * 256u + s[3] - 257u * kOff);
    const int c = (int)(s[4] * 256u + s[5] - 257u * kOff), d = (int)(s[6] * 256u + s[7] - 257u * kOff);
    const int64_t hi = (int64_t)a * 65536 + b, lo = (int64_t)c * 65536 + d;
    return (hi << (18 - drop)) + ((lo + (1 << (13 + drop))) >> (14 + drop));
}

// V 2^q as a double with its exponent field f relative to the row's largest:
// f = 1022 + (bits of |V|) + power - emax
__device__ __forceinline__ double fx_double(int64_t v, int power, int emax)
{
    const uint64_t mag = (uint64_t)(v < 0 ? -v : v);
    const int L = 64 - __clzll((long long)mag);
    const int f = 1022 + L + power - emax;
    const uint64_t m = L <= 53 ? mag << (53 - L) : (mag + (1ull << (L - 54))) >> (L - 53);
    uint64_t bits = ((uint64_t)(f - 1) << 52) + m;
    if (mag == 0 || f <= 0) bits = 0;
    else if (f >= 2047) bits = 0x7FF0000000000000ull;
    return __longlong_as_double((long long)(bits | ((uint64_t)v & 0x8000000000000000ull)));
}

// A thread's H results of row r (column block h) into the staging rows (D + 2
// doubles apart: no bank conflicts), which reuse the digits' shared memory; those
// marked in `low` are there already, redone in FP64, and are scaled by 2^shift ...
template <int D, int H>
__device__ __forceinline__ void fx_put(const int64_t* V, const int* power, int emax, uint32_t low, int shift, double* rows,
                                       int r, int h)
{
    double* out = rows + (size_t)r * (D + 2) + h * H;
    #pragma unroll
    for (int c = 0; c < H; c += 2) {
        const double o0 = fx_double(V[c], power[c], emax), o1 = fx_double(V[c + 1], power[c + 1], emax);
        const uint32_t m = (low >> c) & 3u;
        if (m == 0) {
            *(double2*)(out + c) = make_double2(o0, o1);
        } else {
            if (!(m & 1u)) out[c] = o0;
            if (!(m & 2u)) out[c + 1] = o1;
        }
    }
    for (; low; low &= low - 1) {
        const int c = __ffs((int)low) - 1;
        out[c] = scale_pow2(out[c], shift);
    }
}

// ... and whole rows from there to dst(row) (16 bytes per lane: stored straight
// from the threads, 32 rows per instruction, they took a third of a tile's time)
template <int D, class Dst>
__device__ __forceinline__ void fx_store(const double* rows, int n, const Dst& dst)
{
    for (int q = threadIdx.x; q < n * (D / 2); q += blockDim.x) {
        const int row = q / (D / 2), c = 2 * (q - row * (D / 2));
        *(double2*)(dst(row) + c) = *(const double2*)(rows + (size_t)row * (D + 2) + c);
    }
}

// the digit products of significance 0..7 of one operand pair into eight
// accumulators of N columns (one thread)
template <int KS>
__device__ __forceinline__ void fx_mma(uint32_t tmem, uint32_t N, uint64_t dA, uint64_t dB, uint32_t kA, uint32_t kB,
                                       uint32_t idesc)
{
    for (int l = 0; l < kFxSums; ++l)             // digits a of the rows, l - a of the matrix
        for (int a = max(0, l - kFxDigits + 1); a <= min(l, kFxDigits - 1); ++a)
            #pragma unroll
            for (int ks = 0; ks < KS; ++ks)
                tc::mma_f16(tmem + (uint32_t)l * N, dA + (uint64_t)(a * (kA >> 4) + 16 * ks),
                            dB + (uint64_t)((l - a) * (kB >> 4) + 16 * ks), idesc,
                            (a != max(0, l - kFxDigits + 1) || ks) ? 1u : 0u);
}

// The digits of a tile's rows (row r at pool + src[r] * D, times the column powers
// cm, scaled by 2^-ea[r]) into the operand buffers: eight entries of a row per
// task, eight rows x four tasks per warp (shared memory in whole core matrices).
// ea[r] must hold kFxNoExp; contains a block barrier. big and nonzero get each row's
// masks of entries that are large after the scaling, and not zero (bits below D).
template <int D, int SP>
__device__ __forceinline__ void fx_rows(const double* __restrict__ pool, const int64_t* src_row, const int* cm, int* ea_row,
                                        int* bad_row, uint64_t* big, uint64_t* nonzero, unsigned char* A)
{
    constexpr int NW = kFxRows * SP / 32;
    constexpr uint32_t kA = kFxRows * D * 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int TASKS = D / 8 / SP;         // per thread: 128 D / 8 in all
    double v[TASKS][8];
    int rows[TASKS], pcs[TASKS];
    #pragma unroll
    for (int u = 0; u < TASKS; ++u) {
        const int q = warp + NW * u;          // (row group, 4 pieces)
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
        rows[u] = row;
        pcs[u] = pc;
        const double* src = pool + (size_t)src_row[row] * D + 8 * pc;
        #pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double2 w = *(const double2*)(src + 2 * k);
            v[u][2 * k] = w.x;
            v[u][2 * k + 1] = w.y;
        }
    }
    #pragma unroll
    for (int u = 0; u < TASKS; ++u) {
        int e = kFxNoExp;
        bool bad = false;
        #pragma unroll
        for (int k = 0; k < 8; ++k) {
            e = max(e, fx_exp(v[u][k]) + cm[8 * pcs[u] + k]);
            bad |= fx_not_finite(v[u][k]);
        }
        atomicMax(&ea_row[rows[u]], e);
        if (bad) bad_row[rows[u]] = 1;
    }
    __syncthreads();
    #pragma unroll
    for (int u = 0; u < TASKS; ++u) {
        const int ea = ea_row[rows[u]];
        uint64_t c[8];
        uint32_t mb = 0, mz = 0;
        #pragma unroll
        for (int k = 0; k < 8; ++k) {
            c[k] = fx_code(v[u][k], cm[8 * pcs[u] + k] - ea);
            mb |= (fx_code_big(c[k]) ? 1u : 0u) << k;
            mz |= (fx_nonzero(v[u][k]) ? 1u : 0u) << k;
        }
        ((unsigned char*)(big + rows[u]))[pcs[u]] = (unsigned char)mb;
        ((unsigned char*)(nonzero + rows[u]))[pcs[u]] = (unsigned char)mz;
        const uint32_t off = tc::op_offset(rows[u], 8 * pcs[u], D);
        #pragma unroll
        for (int i = 0; i < kFxDigits; ++i) {
            __align__(16) __half2 d[4];
            #pragma unroll
            for (int k = 0; k < 4; ++k) d[k] = fx_digit2(c[2 * k], c[2 * k + 1], i);
            *(uint4*)(A + (kFxDigits - 1 - i) * kA + off) = *(const uint4*)d;
        }
    }
}

template <int D>
__global__ void __launch_bounds__(kFxRows * fx_split(D), D <= 32 ? 2 : 1) k_fx_step(FxStep st)
{
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ uint32_t tmem_slot;
    __shared__ __align__(8) uint64_t mb_mma, mb_b;
    __shared__ int64_t s_src[kFxRows], s_dst[kFxRows];
    __shared__ int64_t s_gb[8], s_ge[8];
    __shared__ int s_tile[9];
    __shared__ __align__(8) int s_x[fx_exp_stride(D)];         // the matrix's powers of two and masks
    __shared__ int s_ea[kFxRows];                     // power of two taken out of each scaled row
    constexpr int SP = fx_split(D);                   // threads per row
    __shared__ int s_max[SP][kFxRows];
    __shared__ int s_bad[kFxRows], s_inf;             // rows, and the matrix, with an infinity or a NaN
    __shared__ uint64_t s_big[kFxRows], s_nz[kFxRows];
    int* const s_cm = s_x;
    int* const s_eb = s_x + D;
    const uint64_t* const s_m = (const uint64_t*)(s_x + 2 * D);
    constexpr int H = D / SP;                         // columns per thread in the epilogue
    constexpr uint32_t kA = kFxRows * D * 2;          // one digit of the rows
    constexpr uint32_t kB = 2 * D * D;                // one digit of the matrix
    constexpr uint32_t kCols = kFxSums * D <= 128 ? 128 : kFxSums * D <= 256 ? 256 : 512;
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
            s_ea[tid] = kFxNoExp;
        }
        const size_t mat = (size_t)st.mat[side] + (g & 3);
        if (held != g) {
            if (tid == 0) {
                tc::mbar_expect_tx(&mb_b, kFxDigits * kB);
                tc::bulk_g2s(Bs, st.img + mat * kFxDigits * kB, kFxDigits * kB, &mb_b);
            }
            for (int q = tid; q < fx_exp_stride(D); q += kFxRows * SP) s_x[q] = __ldg(st.exps + mat * fx_exp_stride(D) + q);
            if (warp == 0) {
                bool inf = false;
                for (int q = lane; q < D; q += 32) inf |= __ldg(st.exps + mat * fx_exp_stride(D) + D + q) == kFxNotFinite;
                inf = __any_sync(kFull, inf);
                if (lane == 0) s_inf = inf;
            }
        }
        __syncthreads();
        fx_rows<D, SP>(st.pool[side], s_src, s_cm, s_ea, s_bad, s_big, s_nz, smraw);
        tc::fence_proxy_async();
        tc::fence_before_sync();
        __syncthreads();
        if (tid == 0) {
            tc::fence_after_sync();
            if (held != g) ok = tc::mbar_wait(&mb_b, ph_b, kPoll) && ok;
            const uint64_t d0 = tc::desc(0, 128, 16 * D);
            const uint64_t dA = d0 + (tc::smem_addr(smraw) >> 4), dB = d0 + (tc::smem_addr(Bs) >> 4);
            fx_mma<D / 16>(tmem, D, dA, dB, kA, kB, idesc);
            tc::mma_commit(&mb_mma);
        }
        if (held != g) ph_b ^= 1u;
        held = g;
        if (tile + 1 < tile1) {                       // the next tile's rows towards L2 meanwhile
            int g2 = g;
            while (g2 < 7 && tile + 1 >= s_tile[g2 + 1]) ++g2;
            const int64_t i = s_gb[g2] + (int64_t)(tile + 1 - s_tile[g2]) * kFxRows + (tid & (kFxRows - 1));
            if (i < s_ge[g2]) {
                const int64_t row = st.items ? (int64_t)__ldg(st.items + i).x
                                             : (int64_t)__ldg(st.list[g2 >> 2] + i) * st.stride + st.src[g2 >> 2];
                const double* src = st.pool[g2 >> 2] + (size_t)row * D;
                for (int c = 16 * (tid / kFxRows); c < D; c += 16 * SP)
                    asm volatile("prefetch.global.L2 [%0];" :: "l"(src + c));
            }
        }
        if (tid == 0) ok = tc::mbar_wait(&mb_mma, ph_mma, kPoll) && ok;
        ph_mma ^= 1u;
        __syncthreads();
        tc::fence_after_sync();
        // join the sums: V = y 2^(56 - ea - eb), and the row's largest exponent
        int64_t V[H];
        int emax = -(1 << 29);
        uint32_t below = 0;
        #pragma unroll
        for (int c0 = 0; c0 < H; c0 += 8) {
            uint32_t w[kFxSums][8];
            #pragma unroll
            for (int l = 0; l < kFxSums; ++l) tc::tmem_ld8u(tlane + (uint32_t)(l * D + c0), w[l]);
            tc::tmem_wait_ld();
            #pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint32_t x[kFxSums] = {w[0][c], w[1][c], w[2][c], w[3][c], w[4][c], w[5][c], w[6][c], w[7][c]};
                const int64_t v = fx_join<D>(x, 0);
                V[c0 + c] = v;
                if (v != 0) emax = max(emax, 64 - __clzll(v < 0 ? -v : v) + s_eb[h * H + c0 + c]);
                below |= (fx_below(v, 56 - kFxTerm) ? 1u : 0u) << (c0 + c);
            }
        }
        uint32_t low = fx_low<H, D>(below, s_inf != 0, s_big[r], s_nz[r], s_m, s_eb, h);
        if (s_bad[r]) low = H < 32 ? (1u << (H & 31)) - 1u : ~0u;
        if (r >= n) low = 0;
        if (low) {                                    // the others' largest, and these in FP64
            emax = -(1 << 29);
            #pragma unroll
            for (int c = 0; c < H; ++c)
                if (V[c] != 0 && !((low >> c) & 1u)) emax = max(emax, 64 - __clzll(V[c] < 0 ? -V[c] : V[c]) + s_eb[h * H + c]);
            const double* M = st.at[side] + (mat - (size_t)side * 4 * st.K) * D * D;
            const double* x = st.pool[side] + (size_t)s_src[r] * D;
            const uint64_t nz = s_nz[r] & (D < 64 ? (1ull << (D & 63)) - 1 : ~0ull);
            for (uint32_t m = low; m; m &= m - 1) {
                const int c = h * H + __ffs((int)m) - 1;
                const double y = fx_dot(M, x, D, c, nz, s_m[D + c], s_bad[r] || s_eb[c] == kFxNotFinite);
                ((double*)smraw)[(size_t)r * (D + 2) + c] = y;
                const int e = fx_top(y);
                if (e != kFxNoExp) emax = max(emax, e - s_ea[r] + 56);
            }
        }
        s_max[h][r] = emax;
        tc::fence_before_sync();
        __syncthreads();                              // the parts of each row meet
        #pragma unroll
        for (int k = 0; k < SP; ++k) emax = max(emax, s_max[k][r]);
        fx_put<D, H>(V, s_eb + h * H, emax, low, 56 - emax - s_ea[r], (double*)smraw, r, h);
        if (r < n && h == 0) {
            const int* se = st.pool_e[side] + s_src[r];
            st.pool_e[side][s_dst[r]] = *se + (emax < -(1 << 28) ? 0 : emax - 56 + s_ea[r]);
        }
        __syncthreads();
        fx_store<D>((const double*)smraw, n, [&](int row) { return st.pool[side] + (size_t)s_dst[row] * D; });
        __syncthreads();                              // the lists, maxima and digits are free
    }
    if (!ok && tid == 0) report(st.err, 5, 4, (long long)blockIdx.x);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tmem, kCols);
}

// ---------------------------------------------------------------------------
// Graph states over the prefix trees: vertex t of a level's nodes. Per in-edge
// with a vertex source the tile's rows are cut and multiplied as above; the
// edges' 64-bit results are aligned by their powers of two and added as
// integers (log2 of the in-degree bits of the unit are given up for the sum).
// H18 (D = 32, 2.5 in-edges): 128 nodes took 188 k cycles of the FP64 pipe.
// ---------------------------------------------------------------------------

// v 2^-d rounded, d >= 0
__device__ __forceinline__ int64_t fx_shift(int64_t v, int d)
{
    if (d <= 0) return v;
    return d > 62 ? 0 : (v + (1ll << (d - 1))) >> d;
}

// Results `low` (from column c0) of one node in FP64, into out[]: the power of two its
// sums are aligned to goes to *power (the same from every part of the row), the largest
// exponent is returned. AT: the matrices of the node's local state, four apart per edge.
// Out of line: the caller keeps its registers.
template <int D>
__device__ __noinline__ int fx_graph_redo(const uint32_t* it, uint32_t nl, const double* pool, const int* pool_e,
                                          const double* __restrict__ AT, const int* t_e, int nv, int deg, uint32_t low,
                                          int c0, double* out, int* power)
{
    int er = nv < deg ? 0 : -(1 << 30);               // an e_0 source has power 0
    for (int k = 0; k < nv; ++k) er = max(er, pool_e[__ldg(it + (size_t)(k + 1) * nl)]);
    int top = -(1 << 29);
    for (; low; low &= low - 1) {
        const int c = c0 + __ffs((int)low) - 1;
        double y = 0.0;
        for (int k = 0; k < deg; ++k) {
            const double* M = AT + (size_t)t_e[k] * 4 * D * D;
            if (k < nv) {
                const uint32_t sr = __ldg(it + (size_t)(k + 1) * nl);
                y += scale_pow2(dot_col4(M, pool + (size_t)sr * D, D, c), pool_e[sr] - er);
            } else {
                y += scale_pow2(__ldg(M + c), -er);
            }
        }
        out[c] = y;
        const int e = fx_top(y);
        if (e != kFxNoExp) top = max(top, e + er);
    }
    *power = er;
    return top;
}

template <int D>
__global__ void __launch_bounds__(kFxRows * fx_split(D), D <= 32 ? 2 : 1)
k_fx_graph(TreeGraph64 a, const unsigned char* __restrict__ img, const int* __restrict__ exps, DevError* err, int t, int deg,
           uint32_t at, uint32_t nl, TreeGroups gr, int drop)
{
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ uint32_t tmem_slot;
    __shared__ __align__(8) uint64_t mb_mma, mb_b;
    __shared__ int64_t s_src[kFxRows];
    __shared__ __align__(8) int s_x[fx_exp_stride(D)];
    __shared__ int s_ea[kFxRows], s_es[kFxRows], s_bad[kFxRows];
    constexpr int SP = fx_split(D), H = D / SP;
    __shared__ int s_max[SP][kFxRows];
    __shared__ int s_inf;
    __shared__ uint64_t s_big[kFxRows], s_nz[kFxRows];
    int* const s_cm = s_x;
    int* const s_eb = s_x + D;
    const uint64_t* const s_m = (const uint64_t*)(s_x + 2 * D);
    __shared__ int t_e[kGtMaxDeg];                    // edges with a vertex source, then the e_0 ones
    constexpr uint32_t kA = kFxRows * D * 2, kB = 2 * D * D;
    constexpr uint32_t kCols = kFxSums * D <= 128 ? 128 : kFxSums * D <= 256 ? 256 : 512;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned char* const Bs = smraw + kFxDigits * kA;
    if (warp == 0) { tc::tmem_alloc(&tmem_slot, kCols); tc::tmem_relinquish(); }
    if (tid == 0) { tc::mbar_init(&mb_mma, 1); tc::mbar_init(&mb_b, 1); }
    const int e0 = a.an.pred_ptr[t];
    int nv = 0;                                       // in-edges with a vertex source
    for (int e = e0; e < e0 + deg; ++e) nv += a.an.pred_idx[e] >= 0;
    if (tid < deg) {
        const bool vs = a.an.pred_idx[e0 + tid] >= 0;
        int before = 0;
        for (int e = e0; e < e0 + tid; ++e) before += (a.an.pred_idx[e] >= 0) == vs;
        t_e[(vs ? 0 : nv) + before] = e0 + tid;
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
    int64_t held = -1;
    constexpr uint32_t kPoll = 1u << 24;
    const int nt = gr.tile[4];
    const int tile0 = (int)((int64_t)nt * blockIdx.x / gridDim.x);
    const int tile1 = (int)((int64_t)nt * (blockIdx.x + 1) / gridDim.x);
    for (int tile = tile0; tile < tile1; ++tile) {
        int g = 0;
        while (g < 3 && tile >= gr.tile[g + 1]) ++g;
        const uint32_t i0 = gr.b[g] + (uint32_t)(tile - gr.tile[g]) * kFxRows;
        const int n = (int)min(gr.b[g + 1] - i0, (uint32_t)kFxRows);
        int64_t acc[H];
        int X[H];
        #pragma unroll
        for (int c = 0; c < H; ++c) { acc[c] = 0; X[c] = kFxNoExp; }
        uint32_t low = 0;                             // results to be redone in FP64, all edges
        for (int k = 0; k < nv; ++k) {
            const int64_t mat = (int64_t)t_e[k] * 4 + g;
            if (tid < kFxRows) {                      // rows past n repeat the first
                const uint32_t row = __ldg(a.items + at + (size_t)(k + 1) * nl + i0 + (tid < n ? tid : 0));
                s_src[tid] = row;
                s_es[tid] = a.pool_e[row];
                s_ea[tid] = kFxNoExp;
                s_bad[tid] = 0;
            }
            if (held != mat) {
                if (tid == 0) {
                    tc::mbar_expect_tx(&mb_b, kFxDigits * kB);
                    tc::bulk_g2s(Bs, img + (size_t)mat * kFxDigits * kB, kFxDigits * kB, &mb_b);
                }
                for (int q = tid; q < fx_exp_stride(D); q += kFxRows * SP) s_x[q] = __ldg(exps + (size_t)mat * fx_exp_stride(D) + q);
                if (warp == 0) {
                    bool inf = false;
                    for (int q = lane; q < D; q += 32) inf |= __ldg(exps + (size_t)mat * fx_exp_stride(D) + D + q) == kFxNotFinite;
                    inf = __any_sync(kFull, inf);
                    if (lane == 0) s_inf = inf;
                }
            }
            __syncthreads();
            fx_rows<D, SP>(a.pool, s_src, s_cm, s_ea, s_bad, s_big, s_nz, smraw);
            tc::fence_proxy_async();
            tc::fence_before_sync();
            __syncthreads();
            if (tid == 0) {
                tc::fence_after_sync();
                if (held != mat) ok = tc::mbar_wait(&mb_b, ph_b, kPoll) && ok;
                const uint64_t d0 = tc::desc(0, 128, 16 * D);
                fx_mma<D / 16>(tmem, D, d0 + (tc::smem_addr(smraw) >> 4), d0 + (tc::smem_addr(Bs) >> 4), kA, kB, idesc);
                tc::mma_commit(&mb_mma);
            }
            if (held != mat) ph_b ^= 1u;
            held = mat;
            if (tid == 0) ok = tc::mbar_wait(&mb_mma, ph_mma, kPoll) && ok;
            ph_mma ^= 1u;
            __syncthreads();
            tc::fence_after_sync();
            const int ex = s_ea[r] + s_es[r];
            uint32_t below = 0;
            if (s_bad[r]) low = H < 32 ? (1u << (H & 31)) - 1u : ~0u;
            #pragma unroll
            for (int c0 = 0; c0 < H; c0 += 8) {
                uint32_t w[kFxSums][8];
                #pragma unroll
                for (int l = 0; l < kFxSums; ++l) tc::tmem_ld8u(tlane + (uint32_t)(l * D + c0), w[l]);
                tc::tmem_wait_ld();
                #pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint32_t x8[kFxSums] = {w[0][c], w[1][c], w[2][c], w[3][c], w[4][c], w[5][c], w[6][c], w[7][c]};
                    const int64_t v = fx_join<D>(x8, drop);
                    below |= (fx_below(v, 56 - kFxTerm - drop) ? 1u : 0u) << (c0 + c);
                    if (v != 0) {
                        const int x = ex + s_eb[h * H + c0 + c];
                        int64_t& A = acc[c0 + c];
                        int& XA = X[c0 + c];
                        if (x > XA) { A = fx_shift(A, x - XA) + v; XA = x; }
                        else A += fx_shift(v, XA - x);
                    }
                }
            }
            low |= fx_low<H, D>(below, s_inf != 0, s_big[r], s_nz[r], s_m, s_eb, h);
            tc::fence_before_sync();
            __syncthreads();                          // accumulators, digits and lists are free
        }
        for (int k = nv; k < deg; ++k) {              // M e_0: column 0 of the matrix
            const double* col = a.an.AT + ((size_t)t_e[k] * 4 + g) * D * D + h * H;
            #pragma unroll
            for (int c = 0; c < H; ++c) {
                const double m = __ldg(col + c);
                const int x = fx_exp(m);
                if (fx_not_finite(m) || (x == kFxNoExp && fx_nonzero(m))) low |= 1u << c;
                int64_t v = (int64_t)fx_code(m, -x) - 0x80808080808080ll;             // unit 2^-55
                v = drop ? fx_shift(v, drop - 1) : v * 2;
                if (v != 0) {
                    if (x > X[c]) { acc[c] = fx_shift(acc[c], x - X[c]) + v; X[c] = x; }
                    else acc[c] += fx_shift(v, X[c] - x);
                }
            }
        }
        int emax = -(1 << 29);
        #pragma unroll
        for (int c = 0; c < H; ++c)
            if (acc[c] != 0 && !((low >> c) & 1u)) emax = max(emax, 64 - __clzll(acc[c] < 0 ? -acc[c] : acc[c]) + X[c]);
        if (r >= n) low = 0;
        if (low)                                      // these in FP64, all edges
            emax = max(emax, fx_graph_redo<D>(a.items + at + i0 + r, nl, a.pool, a.pool_e, a.an.AT + (size_t)g * D * D,
                                              t_e, nv, deg, low, h * H, (double*)smraw + (size_t)r * (D + 2), s_es + r) + 56 - drop);
        s_max[h][r] = emax;
        __syncthreads();                              // the parts of each row meet
        #pragma unroll
        for (int k = 0; k < SP; ++k) emax = max(emax, s_max[k][r]);
        const uint32_t out = __ldg(a.items + at + i0 + (r < n ? r : 0));
        fx_put<D, H>(acc, X, emax, low, low ? s_es[r] + 56 - drop - emax : 0, (double*)smraw, r, h);
        if (h == 0) {
            s_src[r] = out;                           // the result rows (the sources are done with)
            if (r < n) a.pool_e[out] = emax < -(1 << 28) ? 0 : emax - 56 + drop;
        }
        __syncthreads();
        fx_store<D>((const double*)smraw, n, [&](int row) { return a.pool + (size_t)s_src[row] * D; });
        __syncthreads();                              // s_max and the rows are free
    }
    if (!ok && tid == 0) report(err, 5, 4, (long long)blockIdx.x);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tmem, kCols);
}

template <int D>
void fx_graph_launch(const TreeGraph64& a, const unsigned char* img, const int* exps, DevError* err, int t, int deg,
                     const TreeLevels& lv, const TreeGroups& g, int n_sm, cudaStream_t st)
{
    const size_t smem = (size_t)kFxDigits * (kFxRows * D * 2 + 2 * D * D);
    allow_max_smem(k_fx_graph<D>);
    int drop = -6;                                    // D deg <= 2^(6 + drop) keeps the sums in 63 bits
    for (int x = 1; x < D; x <<= 1) ++drop;
    for (int x = 1; x < deg; x <<= 1) ++drop;
    k_fx_graph<D><<<(unsigned)std::min<int64_t>(g.tile[4], (int64_t)(D <= 32 ? 2 : 1) * n_sm), kFxRows * fx_split(D), smem, st>>>(
        a, img, exps, err, t, deg, lv.at[t], lv.n[t], g, std::max(0, drop));
}

// ---------------------------------------------------------------------------
// Outer-product sums of the gradient, sum_n (w_n g_n) h_n^T over a chunk of one
// local-state group (k_grad_tn's blocks), with the samples as the reduction:
// 64 samples at a time, the operands' rows (components) scaled by powers of two
// over those samples, the exact sums converted once and added in FP64; entries without a
// term near the scale (one sample's weight may set it) are redone as above. A
// 64-sample product of 64 x 64 takes 150 k cycles of the FP64 pipe (1.95 ms for
// H50, D = 64, 4096 samples).
// ---------------------------------------------------------------------------

constexpr int kGradRed = 64;              // samples per product

template <int D>
__global__ void __launch_bounds__(256) k_fx_grad(GradArgs a, int chunk_samples, DevError* err)
{
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ uint32_t tmem_slot;
    __shared__ __align__(8) uint64_t mb_mma;
    __shared__ const double* s_g[kGradRed];
    __shared__ const double* s_h[kGradRed];
    __shared__ double s_w[kGradRed];
    __shared__ int s_e[2 * D], s_bad[2 * D];
    __shared__ uint64_t s_big[2 * D], s_nz[2 * D];    // per component, masks of samples
    __shared__ int s_nlow;                            // entries to be redone in FP64: list, results
    unsigned short* const s_low = (unsigned short*)(smraw + 8 * D * D);
    double* const redone = (double*)smraw;            // [D][D] (both where the operands were)
    constexpr uint32_t kB = 2 * D * kGradRed;         // one digit of one operand
    constexpr uint32_t kCols = kFxSums * D <= 128 ? 128 : kFxSums * D <= 256 ? 256 : 512;
    constexpr int H = D / 2;
    const int K = a.an.K, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int e = blockIdx.y >> 2, sg = blockIdx.y & 3, chunk = blockIdx.x;
    int i, j;
    if (a.an.chain) { i = e; j = e - 1; }
    else {
        j = a.an.pred_idx[e];
        int lo = 0;
        while (a.an.pred_ptr[lo + 1] <= e) ++lo;
        i = lo;
    }
    const int64_t g0 = a.soff[(size_t)i * 5 + sg], g1 = a.soff[(size_t)i * 5 + sg + 1];
    const int64_t c0 = g0 + (int64_t)chunk * chunk_samples;
    if (c0 >= g1) return;                             // beyond this group's chunks
    const int64_t c1 = c0 + chunk_samples < g1 ? c0 + chunk_samples : g1;
    if (warp == 0) { tc::tmem_alloc(&tmem_slot, kCols); tc::tmem_relinquish(); }
    if (tid == 0) tc::mbar_init(&mb_mma, 1);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tmem_slot;
    // M = 128 rows of which the first D are components (the others read what
    // follows in shared memory and are not used)
    const int r = 32 * (warp & 3) + lane, h = warp >> 2;
    const bool act = 32 * (warp & 3) < D;             // uniform over the warp
    const uint32_t tlane = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(h * H);
    const uint32_t idesc = tc::idesc_f16(kFxRows, D);
    uint32_t ph = 0;
    bool ok = true;
    double acc[H];
    #pragma unroll
    for (int c = 0; c < H; ++c) acc[c] = 0.0;
    for (int64_t k0 = c0; k0 < c1; k0 += kGradRed) {
        const int nk = (int)(c1 - k0 < kGradRed ? c1 - k0 : kGradRed);
        if (tid < kGradRed) {
            const double *gp = nullptr, *hp = nullptr;
            double w = 0.0;
            if (tid < nk) {
                const int64_t s = a.sidx[(size_t)i * a.Ns + k0 + tid];
                int eg, eh;
                if (a.an.chain) {
                    gp = a.Renv + ((size_t)s * (K + 1) + i + 1) * D;
                    eg = a.Rexp[(size_t)s * (K + 1) + i + 1];
                    hp = a.Lenv + ((size_t)s * (K + 1) + i) * D;
                    eh = a.Lexp[(size_t)s * (K + 1) + i];
                } else {
                    gp = a.Gst + ((size_t)s * K + i) * D;
                    eg = a.Gexp[(size_t)s * K + i];
                    hp = j < 0 ? nullptr : a.Hst + ((size_t)s * K + j) * D;
                    eh = j < 0 ? 0 : a.Hexp[(size_t)s * K + j];
                }
                w = ldexp(a.u[s] / a.psi_mant[s], eg + eh - a.psi_exp[s]);
            }
            s_g[tid] = gp;
            s_h[tid] = hp;
            s_w[tid] = w;
        }
        if (tid < 2 * D) { s_e[tid] = kFxNoExp; s_bad[tid] = 0; }
        if (tid == 0) s_nlow = 0;
        __syncthreads();
        // component c of operand o (0: w g, 1: h) over eight samples per task, the
        // components across the lanes
        constexpr int TASKS = 2 * D * (kGradRed / 8) / 256;
        double v[TASKS][8];
        #pragma unroll
        for (int u = 0; u < TASKS; ++u) {
            const int q = tid + 256 * u, c = q % (2 * D), n8 = q / (2 * D);
            int ex = kFxNoExp;
            bool bad = false;
            #pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int n = 8 * n8 + k;
                double x = 0.0;
                if (n < nk) {
                    if (c < D) x = s_w[n] * s_g[n][c];
                    else x = s_h[n] ? s_h[n][c - D] : (c == D ? 1.0 : 0.0);
                }
                v[u][k] = x;
                ex = max(ex, fx_exp(x));
                bad |= fx_not_finite(x);
            }
            if (ex != kFxNoExp) atomicMax(&s_e[c], ex);
            if (bad) s_bad[c] = 1;
        }
        __syncthreads();
        #pragma unroll
        for (int u = 0; u < TASKS; ++u) {
            const int q = tid + 256 * u, c = q % (2 * D), n8 = q / (2 * D);
            const int ex = s_e[c] == kFxNoExp ? 0 : s_e[c];
            uint64_t cd[8];
            uint32_t mb = 0, mz = 0;
            #pragma unroll
            for (int k = 0; k < 8; ++k) {
                cd[k] = fx_code(v[u][k], -ex);
                mb |= (fx_code_big(cd[k]) ? 1u : 0u) << k;
                mz |= (fx_nonzero(v[u][k]) ? 1u : 0u) << k;
            }
            ((unsigned char*)(s_big + c))[n8] = (unsigned char)mb;
            ((unsigned char*)(s_nz + c))[n8] = (unsigned char)mz;
            unsigned char* op = smraw + (c < D ? 0u : kFxDigits * kB);
            const uint32_t off = tc::op_offset(c < D ? c : c - D, 8 * n8, kGradRed);
            #pragma unroll
            for (int d = 0; d < kFxDigits; ++d) {
                __align__(16) __half2 w[4];
                #pragma unroll
                for (int k = 0; k < 4; ++k) w[k] = fx_digit2(cd[2 * k], cd[2 * k + 1], d);
                *(uint4*)(op + (kFxDigits - 1 - d) * kB + off) = *(const uint4*)w;
            }
        }
        tc::fence_proxy_async();
        tc::fence_before_sync();
        __syncthreads();
        if (tid == 0) {
            tc::fence_after_sync();
            const uint64_t d0 = tc::desc(0, 128, 16 * kGradRed);
            fx_mma<kGradRed / 16>(tmem, D, d0 + (tc::smem_addr(smraw) >> 4),
                                  d0 + (tc::smem_addr(smraw + kFxDigits * kB) >> 4), kB, kB, idesc);
            tc::mma_commit(&mb_mma);
            ok = tc::mbar_wait(&mb_mma, ph, 1u << 24) && ok;
        }
        ph ^= 1u;
        __syncthreads();
        tc::fence_after_sync();
        uint32_t low = 0;
        if (act) {
            const int ea = r < D ? s_e[r] : 0;
            const bool bad = r < D && s_bad[r];
            const uint64_t mb = s_big[r < D ? r : 0], mz = s_nz[r < D ? r : 0];
            #pragma unroll
            for (int q0 = 0; q0 < H; q0 += 8) {
                uint32_t w[kFxSums][8];
                #pragma unroll
                for (int l = 0; l < kFxSums; ++l) tc::tmem_ld8u(tlane + (uint32_t)(l * D + q0), w[l]);
                tc::tmem_wait_ld();
                #pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint32_t x[kFxSums] = {w[0][c], w[1][c], w[2][c], w[3][c], w[4][c], w[5][c], w[6][c], w[7][c]};
                    const int col = D + h * H + q0 + c;
                    const int64_t V = fx_join<kGradRed>(x, 0);
                    double y = fx_double(V, ea + s_e[col] - 56, 0);
                    if ((fx_below(V, 56 - kFxTerm) && !(s_big[col] & mb) && (s_nz[col] & mz)) || bad || s_bad[col]) {
                        low |= 1u << (q0 + c);
                        y = 0.0;
                    }
                    acc[q0 + c] += y;
                }
            }
            if (r >= D) low = 0;
            if (low) {
                int at = atomicAdd(&s_nlow, __popc(low));
                for (uint32_t m = low; m; m &= m - 1) s_low[at++] = (unsigned short)(r * D + h * H + __ffs((int)m) - 1);
            }
        }
        tc::fence_before_sync();
        __syncthreads();                              // operands, accumulators and lists are free
        if (s_nlow) {
            const int nl = s_nlow;
            for (int k = tid; k < nl; k += 256) {
                const int q = s_low[k], row = q / D, c = q - row * D;
                double y = 0.0;
                #pragma unroll 4
                for (int n = 0; n < nk; ++n)
                    y = fma(s_w[n] * s_g[n][row], s_h[n] ? s_h[n][c] : (c == 0 ? 1.0 : 0.0), y);
                redone[q] = y;
            }
            __syncthreads();
            if (act && r < D) {
                #pragma unroll
                for (int c = 0; c < H; ++c)
                    if ((low >> c) & 1u) acc[c] += redone[(size_t)r * D + h * H + c];
            }
            __syncthreads();
        }
    }
    if (act && r < D) {
        double* out = a.part + (((size_t)chunk * a.an.n_edges + e) * 4 + sg) * D * D + (size_t)r * D + h * H;
        #pragma unroll
        for (int c = 0; c < H; c += 2) *(double2*)(out + c) = make_double2(acc[c], acc[c + 1]);
    }
    if (!ok && tid == 0) report(err, 5, 4, (long long)blockIdx.x);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tmem, kCols);
}

template <int D>
void fx_grad_launch(const GradArgs& a, int64_t chunks, int chunk_samples, DevError* err, cudaStream_t st)
{
    allow_max_smem(k_fx_grad<D>);
    // the MMAs read 128 rows of the last digit too: D and a spare 128 - D rows behind the operands
    const size_t smem = (size_t)2 * kFxDigits * 2 * D * kGradRed + (size_t)2 * (128 - D) * kGradRed;
    k_fx_grad<D><<<dim3((unsigned)chunks, (unsigned)(a.an.n_edges * 4)), 256, smem, st>>>(a, chunk_samples, err);
}

// ---------------------------------------------------------------------------
// Normalised chain readout over the prefix trees (the steps of k_tree_rnn): the
// 4 D candidate entries of 128 nodes as one product of the nodes' cells with the
// vertex's four matrices, 32 rows of them at a time. FP64 work is what is left:
// adding v, P and the choice (~3 operations per entry instead of D + 3).
// ---------------------------------------------------------------------------

template <int KP>
__global__ void __launch_bounds__(256) k_fx_rnn(TreeRnn a, const unsigned char* __restrict__ img, const int* __restrict__ exps,
                                                DevError* err, int t, uint32_t at, uint32_t nl, TreeGroups gr)
{
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ uint32_t tmem_slot;
    __shared__ __align__(8) uint64_t mb_mma, mb_b;
    __shared__ const double* s_src[kFxRows];
    __shared__ double s_prod[kFxRows];
    __shared__ int s_pex[kFxRows], s_sig[kFxRows], s_ea[kFxRows], s_bad[kFxRows];
    __shared__ uint32_t s_flag[kFxRows], s_node[kFxRows];
    __shared__ int s_cm[KP], s_eb[128];
    __shared__ uint64_t s_m[2 * 128];                 // masks of the operand rows, the cells' below
    __shared__ uint64_t s_big[kFxRows], s_nz[kFxRows];
    __shared__ short s_pos[128];                      // candidate entry n at s DP + component
    constexpr uint32_t kA = kFxRows * KP * 2, kB = 32 * KP * 2;
    constexpr uint32_t kCols = kFxSums * 32;
    const AnsatzView& an = a.an;
    const int K = an.K, D = an.D, DP = D | 1, nch = (4 * D + 31) / 32;
    const bool fold = D < KP;                         // v as one more column, against a cell entry of 1
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned char* const Bs = smraw + kFxDigits * kA;                       // [nch][digits][32][KP]
    double* rv = (double*)(Bs + (size_t)nch * kFxDigits * kB);              // [4][D]
    double* eta = rv + 4 * D;
    double* rw = eta + D;
    double* cand = rw + D;                                                  // [rows][4][DP]
    double* Pv = cand + (size_t)kFxRows * 4 * DP;                           // [rows][4]
    if (warp == 0) { tc::tmem_alloc(&tmem_slot, kCols); tc::tmem_relinquish(); }
    if (tid == 0) { tc::mbar_init(&mb_mma, 1); tc::mbar_init(&mb_b, 1); }
    for (int q = tid; q < 4 * D; q += 256) rv[q] = __ldg(an.rv + (size_t)t * 4 * D + q);
    for (int q = tid; q < D; q += 256) { eta[q] = __ldg(an.reta + (size_t)t * D + q); rw[q] = __ldg(an.rw + (size_t)t * D + q); }
    bool inf = false;                                 // in the site's matrices or v
    {
        const int* x = exps + (size_t)t * fx_rnn_exp_stride(KP);
        for (int q = tid; q < KP + 128; q += 256) {
            const int e = __ldg(x + q);
            (q < KP ? s_cm : s_eb - KP)[q] = e;
            inf |= q >= KP && q < KP + 32 * nch && e == kFxNotFinite;
        }
        s_m[tid] = __ldg((const uint64_t*)(x + KP + 128) + tid);
    }
    for (int q = tid; q < 4 * D; q += 256) s_pos[q] = (short)((q / D) * DP + q % D);
    const double rc = __ldg(an.rc + t);
    tc::fence_before_sync();
    const bool any_inf = __syncthreads_or(inf);
    tc::fence_after_sync();
    const uint32_t tmem = tmem_slot;
    const uint32_t b_bytes = (uint32_t)nch * kFxDigits * kB;
    bool ok = true;
    constexpr uint32_t kPoll = 1u << 24;
    if (tid == 0) {
        tc::mbar_expect_tx(&mb_b, b_bytes);
        tc::bulk_g2s(Bs, img + (size_t)t * b_bytes, b_bytes, &mb_b);
        ok = tc::mbar_wait(&mb_b, 0, kPoll);
    }
    const int r = 32 * (warp & 3) + lane, h = warp >> 2;                    // row and half of a 32-entry chunk
    const uint32_t tlane = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(h * 16);
    const uint32_t idesc = tc::idesc_f16(kFxRows, 32);
    uint32_t ph_mma = 0;
    const size_t cur = (size_t)(t & 1) * a.n_nodes, prv = (size_t)((t & 1) ^ 1) * a.n_nodes;
    const uint32_t nt = (nl + kFxRows - 1) / kFxRows;
    for (uint32_t tile = blockIdx.x; tile < nt; tile += gridDim.x) {
        const uint32_t i0 = tile * (uint32_t)kFxRows;
        const int n = (int)min(nl - i0, (uint32_t)kFxRows);
        __syncthreads();
        if (tid < kFxRows) {
            const uint32_t i = i0 + (tid < n ? tid : 0), node = __ldg(a.t.items + at + i);
            s_node[tid] = node;
            s_sig[tid] = (i >= gr.b[1]) + (i >= gr.b[2]) + (i >= gr.b[3]);
            s_ea[tid] = kFxNoExp;
            s_bad[tid] = 0;
            uint32_t src = node;
            if ((int)(a.t.start[node] & 255u) == t) src = a.t.parent[node];
            if (src < a.t.id1) {                      // n itself up to here
                const int64_t s = a.t.s0 + src;
                const uint64_t na = a.t.samples[2 * s], nb = a.t.samples[2 * s + 1];
                s_src[tid] = t > 0 ? a.cells + ((size_t)s * K + t - 1) * D : nullptr;
                s_prod[tid] = 1.0;
                s_pex[tid] = 0;
                s_flag[tid] = (uint32_t)__popcll(na & low_mask(t)) | ((uint32_t)__popcll(nb & low_mask(t)) << 8);
            } else {
                s_src[tid] = a.cell + (prv + src) * D;
                s_prod[tid] = a.prod[prv + src];
                s_pex[tid] = a.pex[prv + src];
                s_flag[tid] = a.flag[prv + src];
            }
        }
        __syncthreads();
        {
            // the cells' digits, eight entries per task (zeros past D)
            constexpr int TASKS = KP / 16;
            double v[TASKS][8];
            int rows[TASKS], pcs[TASKS];
            #pragma unroll
            for (int u = 0; u < TASKS; ++u) {
                const int q = warp + 8 * u;
                const int row = KP == 16 ? q * 16 + (lane & 7) + 8 * (lane >> 4) : q * 8 + (lane & 7);
                const int pc = KP == 16 ? (lane >> 3) & 1 : lane >> 3;
                rows[u] = row;
                pcs[u] = pc;
                const double* src = s_src[row];
                int e = kFxNoExp;
                bool bad = false;
                #pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int c = 8 * pc + k;
                    v[u][k] = c < D ? (src ? src[c] : (c == 0 ? 1.0 : 0.0)) : (c == D ? 1.0 : 0.0);   // h_{-1} = e_0
                    e = max(e, fx_exp(v[u][k]) + s_cm[c]);
                    bad |= fx_not_finite(v[u][k]);
                }
                e = max(e, __shfl_xor_sync(kFull, e, 8));
                if constexpr (KP == 32) e = max(e, __shfl_xor_sync(kFull, e, 16));
                if (KP == 16 ? !(lane & 8) : lane < 8) atomicMax(&s_ea[row], e);
                if (bad) s_bad[row] = 1;
            }
            __syncthreads();
            #pragma unroll
            for (int u = 0; u < TASKS; ++u) {
                const int ea = s_ea[rows[u]];
                uint64_t c[8];
                uint32_t mb = 0, mz = 0;
                #pragma unroll
                for (int k = 0; k < 8; ++k) {
                    c[k] = fx_code(v[u][k], s_cm[8 * pcs[u] + k] - ea);
                    mb |= (fx_code_big(c[k]) ? 1u : 0u) << k;
                    mz |= (fx_nonzero(v[u][k]) ? 1u : 0u) << k;
                }
                ((unsigned char*)(s_big + rows[u]))[pcs[u]] = (unsigned char)mb;
                ((unsigned char*)(s_nz + rows[u]))[pcs[u]] = (unsigned char)mz;
                const uint32_t off = tc::op_offset(rows[u], 8 * pcs[u], KP);
                #pragma unroll
                for (int i = 0; i < kFxDigits; ++i) {
                    __align__(16) __half2 d[4];
                    #pragma unroll
                    for (int k = 0; k < 4; ++k) d[k] = fx_digit2(c[2 * k], c[2 * k + 1], i);
                    *(uint4*)(smraw + (kFxDigits - 1 - i) * kA + off) = *(const uint4*)d;
                }
            }
        }
        const int ea = s_ea[r];
        const bool row_bad = s_bad[r] != 0;
        uint64_t mb = 0, mz = 0;
        for (int ch = 0; ch < nch; ++ch) {
            tc::fence_proxy_async();
            tc::fence_before_sync();
            __syncthreads();                          // digits written (first chunk), accumulators read (later ones)
            if (tid == 0) {
                tc::fence_after_sync();
                const uint64_t d0 = tc::desc(0, 128, 16 * KP);
                fx_mma<KP / 16>(tmem, 32, d0 + (tc::smem_addr(smraw) >> 4),
                                d0 + (tc::smem_addr(Bs + (size_t)ch * kFxDigits * kB) >> 4), kA, kB, idesc);
                tc::mma_commit(&mb_mma);
            }
            if (tid == 0) ok = tc::mbar_wait(&mb_mma, ph_mma, kPoll) && ok;
            ph_mma ^= 1u;
            __syncthreads();
            tc::fence_after_sync();
            if (ch == 0) { mb = s_big[r]; mz = s_nz[r]; }
            uint32_t below = 0;
            #pragma unroll
            for (int c0 = 0; c0 < 16; c0 += 8) {
                const int col = 32 * ch + 16 * h + c0;
                if (col >= 4 * D) break;              // uniform over the warp
                uint32_t w[kFxSums][8];
                #pragma unroll
                for (int l = 0; l < kFxSums; ++l) tc::tmem_ld8u(tlane + (uint32_t)(l * 32 + c0), w[l]);
                tc::tmem_wait_ld();
                #pragma unroll
                for (int c = 0; c < 8; ++c) {
                    if (col + c >= 4 * D) break;
                    const uint32_t x[kFxSums] = {w[0][c], w[1][c], w[2][c], w[3][c], w[4][c], w[5][c], w[6][c], w[7][c]};
                    const int64_t v = fx_join<KP>(x, 0);
                    double y = fx_double(v, ea + s_eb[col + c] - 56, 0);
                    below |= (fx_below(v, 56 - kFxTerm) ? 1u : 0u) << (c0 + c);
                    if (!fold) y += rv[col + c];
                    cand[(size_t)r * 4 * DP + s_pos[col + c]] = y;
                }
            }
            uint32_t low = fx_low<16, 128>(below, any_inf, mb, mz, s_m + 32 * ch, s_eb + 32 * ch, h);
            if (row_bad) low = 0xFFFFu;
            for (; low; low &= low - 1) {             // in FP64
                const int e = 32 * ch + 16 * h + __ffs((int)low) - 1;
                if (e >= 4 * D) break;
                const int sg = e / D, c = e - sg * D;
                const double* M = an.AT + ((size_t)t * 4 + sg) * D * D;
                const double* x = s_src[r];
                cand[(size_t)r * 4 * DP + s_pos[e]] = rv[e] + (x ? dot_col4(M, x, D, c) : __ldg(M + c));
            }
        }
        tc::fence_before_sync();
        __syncthreads();
        for (int q = tid; q < n * 4; q += 256) {
            const double* x = cand + (size_t)q * DP;
            double p = 0.0;
            for (int c = 0; c < D; ++c) p = fma(eta[c] * x[c], x[c], p);
            Pv[q] = p;
        }
        __syncthreads();
        if (tid < n) tree_rnn_pick(a, t, tid, s_sig[tid], s_flag[tid], s_prod[tid], s_pex[tid], cur + s_node[tid], cand, DP, Pv, rw, rc);
        if (t + 1 < K)
            for (int q = tid; q < n * D; q += 256) {
                const int it = q / D, c = q - it * D;
                a.cell[(cur + s_node[it]) * D + c] = cand[(size_t)(it * 4 + s_sig[it]) * DP + c];
            }
    }
    if (!ok && tid == 0) report(err, 5, 4, (long long)blockIdx.x);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tmem, kCols);
}

// per site: row s D + r of the operand is row r of M^s and, where a column is free,
// v^s[r], in blocks of 32 rows
__global__ void __launch_bounds__(256) k_fx_rnn_images(const double* __restrict__ A, const double* __restrict__ v, int D, int KP,
                                                       unsigned char* img, int* exps)
{
    __shared__ int sc[32], sr[128];
    const int t = blockIdx.x, nch = (4 * D + 31) / 32;
    const double* M = A + (size_t)t * 4 * D * D;
    const double* vt = v + (size_t)t * 4 * D;
    int* const x = exps + (size_t)t * fx_rnn_exp_stride(KP);
    uint64_t* const masks = (uint64_t*)(x + KP + 128);
    fx_image([&](int n, int k) { return k < D ? __ldg(M + (size_t)n * D + k) : __ldg(vt + n); }, 4 * D, D < KP ? D + 1 : D, 32, KP,
             img + (size_t)t * nch * kFxDigits * 64 * KP, x, x + KP, masks, masks + 128, sc, sr);
}

size_t fx_rnn_smem(int D)
{
    const size_t KP = D <= 16 ? 16 : 32, nch = (4 * D + 31) / 32;
    return kFxDigits * (kFxRows * KP * 2 + nch * 64 * KP) + (6 * D + (size_t)kFxRows * 4 * (D | 1) + 4 * kFxRows) * 8;
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
    k_fx_step<D><<<(unsigned)std::min<int64_t>(tiles, (int64_t)per * n_sm), kFxRows * fx_split(D), smem, st>>>(s);
}

}  // namespace

int launch_fx_images(const double* A, int n_mats, int D, int sides, unsigned char* img, int* exps, cudaStream_t st)
{
    k_fx_images<<<dim3((unsigned)n_mats, (unsigned)sides), 256, 0, st>>>(A, n_mats, D, img, exps);
    return 1;
}

int launch_fx_graph(const TreeGraph64& a, const unsigned char* img, const int* exps, DevError* err, int t, int deg,
                    const TreeLevels& lv, const int64_t* bounds, int n_sm, cudaStream_t st)
{
    const TreeGroups g = tree_groups(t, bounds, kFxRows);
    if (g.tile[4] == 0) return 0;
    switch (a.an.D) {
    case 16: fx_graph_launch<16>(a, img, exps, err, t, deg, lv, g, n_sm, st); break;
    case 32: fx_graph_launch<32>(a, img, exps, err, t, deg, lv, g, n_sm, st); break;
    case 48: fx_graph_launch<48>(a, img, exps, err, t, deg, lv, g, n_sm, st); break;
    default: fx_graph_launch<64>(a, img, exps, err, t, deg, lv, g, n_sm, st); break;
    }
    return 1;
}

int launch_fx_grad(const GradArgs& a, int64_t chunks, int chunk_samples, DevError* err, cudaStream_t st)
{
    switch (a.an.D) {
    case 16: fx_grad_launch<16>(a, chunks, chunk_samples, err, st); break;
    case 32: fx_grad_launch<32>(a, chunks, chunk_samples, err, st); break;
    case 48: fx_grad_launch<48>(a, chunks, chunk_samples, err, st); break;
    default: fx_grad_launch<64>(a, chunks, chunk_samples, err, st); break;
    }
    return 1;
}

int launch_fx_rnn_images(const double* A, const double* v, int K, int D, unsigned char* img, int* exps, cudaStream_t st)
{
    k_fx_rnn_images<<<(unsigned)K, 256, 0, st>>>(A, v, D, D <= 16 ? 16 : 32, img, exps);
    return 1;
}

int launch_fx_rnn(const TreeRnn& a, const unsigned char* img, const int* exps, DevError* err, int t, const TreeLevels& lv,
                  const int64_t* bounds, int n_sm, cudaStream_t st)
{
    if (lv.n[t] == 0) return 0;
    const size_t smem = fx_rnn_smem(a.an.D);
    const int64_t nt = (lv.n[t] + kFxRows - 1) / kFxRows;
    const int per = smem <= 100 * 1024 ? 2 : 1;       // 256 tensor-memory columns each
    const unsigned grid = (unsigned)std::min<int64_t>(nt, (int64_t)per * n_sm);
    if (a.an.D <= 16) {
        allow_max_smem(k_fx_rnn<16>);
        k_fx_rnn<16><<<grid, 256, smem, st>>>(a, img, exps, err, t, lv.at[t], lv.n[t], tree_groups(t, bounds, kFxRows));
    } else {
        allow_max_smem(k_fx_rnn<32>);
        k_fx_rnn<32><<<grid, 256, smem, st>>>(a, img, exps, err, t, lv.at[t], lv.n[t], tree_groups(t, bounds, kFxRows));
    }
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
