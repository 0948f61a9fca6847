// nqs_util.cu -- integral build, prefix scans, per-sample reductions and the
// energy summary (Sec. 2.1 weighted mean, Sec. 2.3 B and E~_loc).
#include "nqs_kernels.cuh"

#include <mutex>
#include <set>
#include <utility>

namespace nqs {

void allow_max_smem_fn(const void* kernel)
{
    static std::mutex mu;
    static std::set<std::pair<int, const void*>> done;
    int dev = 0, mx = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    std::lock_guard<std::mutex> lock(mu);
    if (done.count({dev, kernel})) return;
    cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, kernel) == cudaSuccess &&
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, mx - (int)fa.sharedSizeBytes) == cudaSuccess)
        done.insert({dev, kernel});
}

// (pq|rs) = sum_x L[x][p][q] L[x][r][s], ascending x, fused multiply-add,
// stored at [p][q][s][r] (the layout eri_at reads).
__global__ void k_build_eri(const double* L, int n_chol, int K, double* eri)
{
    const int64_t KK = (int64_t)K * K;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= KK * KK) return;
    const int64_t pq = idx / KK, sr = idx - pq * KK;
    const int64_t s = sr / K, r = sr - s * K, rs = r * K + s;
    double acc = 0.0;
    for (int x = 0; x < n_chol; ++x)
        acc = __fma_rn(__ldg(L + x * KK + pq), __ldg(L + x * KK + rs), acc);
    eri[idx] = acc;
}

int launch_build_eri(const double* L, int n_chol, int K, double* eri, cudaStream_t st)
{
    const int64_t n = (int64_t)K * K * K * K;
    k_build_eri<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(L, n_chol, K, eri);
    return 1;
}

// a full (pq|rs) table [p][q][r][s] into the layout eri_at reads, [p][q][s][r]
__global__ void k_swap_eri(const double* in, int K, double* eri)
{
    const int64_t KK = (int64_t)K * K;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= KK * KK) return;
    const int64_t pq = idx / KK, sr = idx - pq * KK;
    const int64_t s = sr / K, r = sr - s * K;
    eri[idx] = in[pq * KK + r * K + s];
}

int launch_swap_eri(const double* in, int K, double* eri, cudaStream_t st)
{
    const int64_t n = (int64_t)K * K * K * K;
    k_swap_eri<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(in, K, eri);
    return 1;
}

// Block-wide inclusive scan of one value per thread (blockDim multiple of 32).
template <typename T>
__device__ T block_incl_scan(T v, T* warp_tot)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        T t = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += t;
    }
    if (lane == 31) warp_tot[warp] = v;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nw ? warp_tot[lane] : T(0);
        for (int o = 1; o < 32; o <<= 1) {
            T t = __shfl_up_sync(kFull, w, o);
            if (lane >= o) w += t;
        }
        if (lane < nw) warp_tot[lane] = w;
    }
    __syncthreads();
    if (warp) v += warp_tot[warp - 1];
    __syncthreads();
    return v;
}

__global__ void k_scan_chunks_u32(const uint32_t* cnt, uint32_t* off, int64_t* total,
                                  uint32_t n_chunks)
{
    __shared__ uint32_t wt[32];
    const size_t row = (size_t)blockIdx.x * n_chunks;
    uint32_t carry = 0;
    for (uint32_t t0 = 0; t0 < n_chunks; t0 += blockDim.x) {
        const uint32_t i = t0 + threadIdx.x;
        const uint32_t v = i < n_chunks ? cnt[row + i] : 0u;
        const uint32_t inc = block_incl_scan<uint32_t>(v, wt);
        if (i < n_chunks) off[row + i] = carry + inc - v;
        carry += wt[(blockDim.x >> 5) - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

int launch_scan_chunks_u32(const uint32_t* cnt, uint32_t* off, int64_t* total, int64_t Ns,
                           uint32_t n_chunks, cudaStream_t st)
{
    if (Ns == 0) return 0;
    k_scan_chunks_u32<<<(unsigned)Ns, 256, 0, st>>>(cnt, off, total, n_chunks);
    return 1;
}

__global__ void k_scan_chunks_u64(uint64_t* w, uint64_t* total, uint32_t n_chunks)
{
    __shared__ uint64_t wt[32];
    const size_t row = (size_t)blockIdx.x * n_chunks;
    uint64_t carry = 0;
    for (uint32_t t0 = 0; t0 < n_chunks; t0 += blockDim.x) {
        const uint32_t i = t0 + threadIdx.x;
        const uint64_t v = i < n_chunks ? w[row + i] : 0ull;
        const uint64_t inc = block_incl_scan<uint64_t>(v, wt);
        if (i < n_chunks) w[row + i] = carry + inc;
        carry += wt[(blockDim.x >> 5) - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

int launch_scan_chunks_u64(uint64_t* w, uint64_t* total, int64_t Ns, uint32_t n_chunks,
                           cudaStream_t st)
{
    if (Ns == 0) return 0;
    k_scan_chunks_u64<<<(unsigned)Ns, 256, 0, st>>>(w, total, n_chunks);
    return 1;
}

// one block per job
__global__ void __launch_bounds__(1024) k_scan_i64(ScanJobs jobs)
{
    __shared__ int64_t wt[32];
    const ScanJob& s = jobs.job[blockIdx.x];
    int64_t carry = 0;
    for (int64_t t0 = 0; t0 < s.n; t0 += blockDim.x) {
        const int64_t i = t0 + threadIdx.x;
        int64_t v = i < s.n ? s.in[i] + (s.add ? s.add[i] : 0) : 0;
        if (s.rows > 0) v = (v + s.rows - 1) / s.rows;
        const int64_t inc = block_incl_scan<int64_t>(v, wt);
        if (i < s.n) s.out[i] = carry + inc - v;
        carry += wt[(blockDim.x >> 5) - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) s.out[s.n] = carry;
}

int launch_scan_jobs(const ScanJobs& jobs, cudaStream_t st)
{
    k_scan_i64<<<(unsigned)jobs.n, 1024, 0, st>>>(jobs);
    return 1;
}

int launch_scan_i64(const int64_t* in, int64_t* out, int64_t n, cudaStream_t st)
{
    return launch_scan_jobs({{{in, nullptr, out, n, 0}}, 1}, st);
}

// Multi-block exclusive scan: sums of 4096-element tiles, one block scans the
// sums, then every tile rescans its elements from its offset (integers: the
// result does not depend on the tiling).

__global__ void __launch_bounds__(1024) k_scan_tile_sums(const int64_t* in, int64_t n, int64_t* sums)
{
    __shared__ int64_t wt[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t v = 0;
    #pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int64_t i = base + k * 1024 + threadIdx.x;
        if (i < n) v += in[i];
    }
    v = block_incl_scan<int64_t>(v, wt);
    if (threadIdx.x == blockDim.x - 1) sums[blockIdx.x] = v;
}

__global__ void __launch_bounds__(1024) k_scan_tiles(const int64_t* in, int64_t* out, int64_t n,
                                                      const int64_t* tile_off)
{
    __shared__ int64_t wt[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + 4 * (int64_t)threadIdx.x;
    int64_t x[4], s = 0;
    #pragma unroll
    for (int k = 0; k < 4; ++k) {
        x[k] = base + k < n ? in[base + k] : 0;
        s += x[k];
    }
    const int64_t inc = block_incl_scan<int64_t>(s, wt);
    int64_t run = tile_off[blockIdx.x] + inc - s;
    #pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (base + k < n) out[base + k] = run;
        run += x[k];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1) out[n] = run;
}

int launch_scan_i64_wide(const int64_t* in, int64_t* out, int64_t n, int64_t* tmp, cudaStream_t st)
{
    if (n <= kScanOneBlock || !tmp) return launch_scan_i64(in, out, n, st);
    const int64_t nt = (n + kScanTile - 1) / kScanTile;
    int64_t* sums = tmp;
    int64_t* offs = tmp + nt + 1;
    k_scan_tile_sums<<<(unsigned)nt, 1024, 0, st>>>(in, n, sums);
    launch_scan_i64(sums, offs, nt, st);
    k_scan_tiles<<<(unsigned)nt, 1024, 0, st>>>(in, out, n, offs);
    return 3;
}

int launch_chunk_base(const int64_t* cnt, int rows, int64_t* out, int64_t Ns, cudaStream_t st)
{
    return launch_scan_jobs({{{cnt, nullptr, out, Ns, rows}}, 1}, st);
}

// ---------------------------------------------------------------------------
// E_loc per sample = H_nn + sum of det-row partials + sum of draw-row partials
// (in chunk order), then the weighted summary (fixed tree order). A heavy
// sample's E_loc - Ebar cancels in the energy gradient, so the orders are those
// of plain loops: a warp per sample loads 32 partials at a time and adds them
// one after the other; the summary's sums run in one block, and only the counts
// of the chunks (whole numbers, 1.2 M chunks on H18) are summed over the chip.
// ---------------------------------------------------------------------------

// v[b0] + v[b0 + 1] + ... in order, on every lane of the warp
__device__ double chunk_sum_warp(const double* v, int64_t b0, int64_t b1, int lane, double x)
{
    for (int64_t b = b0; b < b1; b += 32) {
        const double mine = b + lane < b1 ? v[b + lane] : 0.0;
        const int n = (int)(b1 - b < 32 ? b1 - b : 32);
        if (n == 32) {
            #pragma unroll
            for (int k = 0; k < 32; ++k) x += __shfl_sync(kFull, mine, k);
        } else {
            for (int k = 0; k < n; ++k) x += __shfl_sync(kFull, mine, k);
        }
    }
    return x;
}

__global__ void __launch_bounds__(256) k_final_samples(FinalArgs a)
{
    const int64_t s = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (s >= a.Ns) return;
    const int64_t d0 = a.base_det[s], d1 = a.base_det[s + 1];
    int64_t w0 = 0, w1 = 0;
    if (a.base_draw) { w0 = a.base_draw[s]; w1 = a.base_draw[s + 1]; }
    const double ed = chunk_sum_warp(a.part_det, d0, d1, lane, 0.0);
    const double es = chunk_sum_warp(a.part_draw, w0, w1, lane, 0.0);
    double ea = 0.0;
    if (a.e_abs) {
        ea = chunk_sum_warp(a.part_det_abs, d0, d1, lane, fabs(a.h_diag[s]));
        if (a.part_draw_abs) ea = chunk_sum_warp(a.part_draw_abs, w0, w1, lane, ea);
    }
    if (lane) return;
    a.e_loc[s] = a.h_diag[s] + ed + es;
    if (a.e_abs) a.e_abs[s] = ea;
    if (a.e_det) a.e_det[s] = ed;
    if (a.e_stoch) a.e_stoch[s] = es;
}

__device__ double block_reduce_sum(double v, double* sh)
{
    v = warp_sum_f64(v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += sh[w];
    __syncthreads();
    return r;   // valid in thread 0
}

// Block b's share of the chunks' vertex and product counts, at summary[8 + 2 b].
__global__ void __launch_bounds__(256) k_summary_counts(FinalArgs a)
{
    __shared__ double sh[32];
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    double sp = 0.0, mv = 0.0;
    const int64_t nd = a.base_det ? a.base_det[a.Ns] : 0, nw = a.base_draw ? a.base_draw[a.Ns] : 0;
    if (a.span_det) for (int64_t b = t0; b < nd; b += step) sp += (double)a.span_det[b];
    if (a.span_draw) for (int64_t b = t0; b < nw; b += step) sp += (double)a.span_draw[b];
    if (a.mv_det) for (int64_t b = t0; b < nd; b += step) mv += (double)a.mv_det[b];
    if (a.mv_draw) for (int64_t b = t0; b < nw; b += step) mv += (double)a.mv_draw[b];
    sp = block_reduce_sum(sp, sh);
    mv = block_reduce_sum(mv, sh);
    if (threadIdx.x == 0) {
        a.summary[8 + 2 * blockIdx.x] = sp;
        a.summary[8 + 2 * blockIdx.x + 1] = mv;
    }
}

__global__ void __launch_bounds__(256) k_summary(FinalArgs a, int count_blocks)
{
    __shared__ double sh[5][8];
    __shared__ double bc;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double m = -INFINITY;
    #pragma unroll 4
    for (int64_t s = threadIdx.x; s < a.Ns; s += 256) m = fmax(m, 2.0 * a.log_f[s]);
    m = warp_max_f64(m);
    if (lane == 0) sh[0][warp] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        double mm = -INFINITY;
        for (int w = 0; w < 8; ++w) mm = fmax(mm, sh[0][w]);
        bc = mm;
    }
    __syncthreads();
    m = bc;
    // sum c, sum c E, sum c f^2 e^-m, listed and drawn rows
    double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    #pragma unroll 4
    for (int64_t s = threadIdx.x; s < a.Ns; s += 256) {
        const double c = a.counts ? a.counts[s] : 1.0;
        v[0] += c;
        v[1] += c * a.e_loc[s];
        v[2] += c * exp(2.0 * a.log_f[s] - m);
        if (a.det_off) v[3] += (double)(a.det_off[s + 1] - a.det_off[s]);
        if (a.n_unique) v[4] += (double)a.n_unique[s];
    }
    __syncthreads();
    #pragma unroll
    for (int k = 0; k < 5; ++k) {
        v[k] = warp_sum_f64(v[k]);
        if (lane == 0) sh[k][warp] = v[k];
    }
    __syncthreads();
    double r = 0.0;                                   // threads 0..4: one sum each, warps in order
    if (threadIdx.x < 5)
        for (int w = 0; w < 8; ++w) r += sh[threadIdx.x][w];
    __syncthreads();
    if (threadIdx.x < 5) sh[threadIdx.x][0] = r;
    __syncthreads();
    const double sc = sh[0][0], sce = sh[1][0], scf = sh[2][0], ndet = sh[3][0], nu = sh[4][0];
    const double logB = m + log(scf / sc);
    double set = 0.0;
    #pragma unroll 4
    for (int64_t s = threadIdx.x; s < a.Ns; s += 256) {
        const double c = a.counts ? a.counts[s] : 1.0;
        set += c * exp(2.0 * a.log_f[s] - logB) * a.e_loc[s];
    }
    __syncthreads();
    set = block_reduce_sum(set, sh[0]);
    double sp = 0.0, mv = 0.0;
    if (warp == 0) {
        for (int b = lane; b < count_blocks; b += 32) { sp += a.summary[8 + 2 * b]; mv += a.summary[8 + 2 * b + 1]; }
        sp = warp_sum_f64(sp);
        mv = warp_sum_f64(mv);
    }
    if (threadIdx.x == 0) {
        a.summary[0] = sce / sc;
        a.summary[1] = sc;
        a.summary[2] = logB;
        a.summary[3] = set / sc;
        a.summary[4] = ndet;
        a.summary[5] = nu;
        a.summary[6] = sp;
        a.summary[7] = mv;
    }
}

int launch_summary(const FinalArgs& a, cudaStream_t st)
{
    if (a.Ns == 0 || !a.summary) return 0;
    const bool counts = a.span_det || a.mv_det;
    if (counts) k_summary_counts<<<kSummaryBlocks, 256, 0, st>>>(a);
    k_summary<<<1, 256, 0, st>>>(a, counts ? kSummaryBlocks : 0);
    return counts ? 2 : 1;
}

// samples picked for re-evaluation: their words, counts and global positions
__global__ void k_gather_picked(const int64_t* idx, int64_t n, const uint64_t* samples,
                                const double* counts, int64_t base, uint64_t* out_s, double* out_c,
                                int64_t* out_pos)
{
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const int64_t s = idx[j];
    out_s[2 * j] = samples[2 * s];
    out_s[2 * j + 1] = samples[2 * s + 1];
    out_c[j] = counts ? counts[s] : 1.0;
    out_pos[j] = base + s;
}

__global__ void k_scatter_picked(const int64_t* idx, int64_t n, const double* v, double* out)
{
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < n) out[idx[j]] = v[j];
}

int launch_gather_picked(const int64_t* idx, int64_t n, const uint64_t* samples, const double* counts,
                         int64_t base, uint64_t* out_s, double* out_c, int64_t* out_pos, cudaStream_t st)
{
    if (n == 0) return 0;
    k_gather_picked<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(idx, n, samples, counts, base, out_s,
                                                                 out_c, out_pos);
    return 1;
}

int launch_scatter_picked(const int64_t* idx, int64_t n, const double* v, double* out, cudaStream_t st)
{
    if (n == 0) return 0;
    k_scatter_picked<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(idx, n, v, out);
    return 1;
}

int launch_finalize(const FinalArgs& a, cudaStream_t st)
{
    if (a.Ns == 0) return 0;
    k_final_samples<<<(unsigned)((a.Ns + 7) / 8), 256, 0, st>>>(a);
    return 1 + launch_summary(a, st);
}

}  // namespace nqs
