// nqs_grad.cu -- the backward pass: sum_n u_n d log|psi(n)| / d theta (the
// vector-Jacobian product of Eq. egrad: with u_n = 2 c_n (E_loc(n) - E) / sum c
// it is the energy gradient; Sec. 2.3 gives the weights of the reweighted form).
//
// Tensor network (linear readout): with the forward cells h and the adjoints
// g = d psi_TN / d h of sample n, d psi_TN(n) / d M_e^s[a][b] = [s = s_i(n)]
// g_i(n)[a] h_j(n)[b] for the edge e = (j -> i) (chain: h_j = L_{i-1},
// g_i = R_{i+1}), so
//   grad_e^s = sum_{n : s_i(n) = s} w_n g_i(n) h_j(n)^T,   w_n = u_n / psi_TN(n),
// one outer-product sum (a GEMM with the samples as the reduction axis) per
// edge and local state. Per vertex the samples are grouped by local state with
// a stable counting sort; each block sums one chunk of one group into a 64 x 64
// output tile (4 x 4 accumulators per thread, operand rows staged in shared
// memory); the chunk partials are added in chunk order, so the result does not
// depend on the schedule. FP64 throughout (the check form of the gradient).
//
// Correlator: d log|f| / d b_k = t_k, d / d W[k][s] = t_k n_s, d / d W2[k][s][t]
// = t_k n_s n_t / 2, with t_k = tanh(theta_k) (2cosh) or -tan(theta_k) (cos,
// Ising); one thread per parameter sums over the samples in index order.
#include "nqs_fx.cuh"

namespace nqs {

namespace {

constexpr int kGradChunk = 256;   // samples per block (one chunk of a local-state group)
// samples from which the fixed-point products run. H18 energy gradient (D = 32),
// fixed-point / FP64: 32 samples 1.81 / 1.81 ms, 64 2.03 / 2.06, 128 2.52 / 2.59,
// 512 5.75 / 6.18
constexpr int64_t kFxGradMin = 64;
constexpr int kTile = 64;         // output tile edge
constexpr int kStage = 16;        // samples staged per round

int64_t grad_chunks(int64_t Ns) { return (Ns + kGradChunk - 1) / kGradChunk; }

// samples per block of the correlator gradient: at most 128 chunks, at least
// 32 samples each (about two blocks per SM for N_h = 100, 4096 samples)
int64_t corr_chunk(int64_t Ns)
{
    const int64_t c = (Ns + 127) / 128;
    return c < 32 ? 32 : c;
}

// bound on corr_chunks over every count up to Ns (a shorter last pass may have more chunks)
int64_t max_corr_chunks(int64_t Ns) { return (Ns + 31) / 32 < 128 ? (Ns + 31) / 32 : 128; }

int64_t corr_chunks(int64_t Ns) { return (Ns + corr_chunk(Ns) - 1) / corr_chunk(Ns); }

}  // namespace

size_t grad_scratch_bytes(const AnsatzView& an, int64_t Ns)
{
    return grad_corr_offset(an, Ns) + ((size_t)Ns + (size_t)max_corr_chunks(Ns) * (2 * an.K + 1)) * an.n_hidden * 8;
}

size_t grad_corr_offset(const AnsatzView& an, int64_t Ns)
{
    return (size_t)an.K * Ns * 4 + (size_t)an.K * 5 * 8 + 512 +     // two 256-byte alignments
           (size_t)grad_chunks(Ns) * an.n_edges * 4 * an.D * an.D * 8;
}

// Stable grouping of the sample indices of vertex i (blockIdx.x) by local state.
__global__ void __launch_bounds__(1024) k_group_by_state(const uint64_t* samples, int64_t Ns, int32_t* sidx, int64_t* soff)
{
    __shared__ int wsum[32];
    __shared__ int64_t base;
    const int i = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int32_t* out = sidx + (size_t)i * Ns;
    if (threadIdx.x == 0) base = 0;
    __syncthreads();
    for (int sg = 0; sg < 4; ++sg) {
        if (threadIdx.x == 0) soff[(size_t)i * 5 + sg] = base;
        for (int64_t t0 = 0; t0 < Ns; t0 += blockDim.x) {
            const int64_t s = t0 + threadIdx.x;
            const bool f = s < Ns && sigma_at(samples[2 * s], samples[2 * s + 1], i) == sg;
            const unsigned bal = __ballot_sync(kFull, f);
            if (lane == 0) wsum[warp] = __popc(bal);
            __syncthreads();
            int before = 0, total = 0;
            for (int w = 0; w < nw; ++w) { if (w < warp) before += wsum[w]; total += wsum[w]; }
            if (f) out[base + before + __popc(bal & ((1u << lane) - 1u))] = (int32_t)s;
            __syncthreads();
            if (threadIdx.x == 0) base += total;
            __syncthreads();
        }
    }
    if (threadIdx.x == 0) soff[(size_t)i * 5 + 4] = base;
}

// One (edge, local state, chunk, output tile): partial sum over the chunk's samples.
__global__ void __launch_bounds__(256) k_grad_tn(GradArgs a, int n_tiles)
{
    __shared__ double gS[kStage][kTile];
    __shared__ double hS[kStage][kTile];
    __shared__ int32_t sid[kStage];
    const int D = a.an.D, K = a.an.K;
    const int e = blockIdx.z >> 2, sg = blockIdx.z & 3;
    const int chunk = blockIdx.y;
    const int ta = blockIdx.x / n_tiles, tb = blockIdx.x - ta * n_tiles;
    int i, j;
    if (a.an.chain) { i = e; j = e - 1; }
    else {
        j = a.an.pred_idx[e];
        int lo = 0;
        while (a.an.pred_ptr[lo + 1] <= e) ++lo;
        i = lo;
    }
    const int64_t g0 = a.soff[(size_t)i * 5 + sg], g1 = a.soff[(size_t)i * 5 + sg + 1];
    const int64_t c0 = g0 + (int64_t)chunk * kGradChunk;
    if (c0 >= g1) return;                              // beyond this group's chunks
    const int64_t c1 = c0 + kGradChunk < g1 ? c0 + kGradChunk : g1;
    const int a0 = ta * kTile, b0 = tb * kTile;
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    double acc[4][4];
    #pragma unroll
    for (int u = 0; u < 4; ++u)
        #pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = 0.0;
    for (int64_t k0 = c0; k0 < c1; k0 += kStage) {
        const int nk = (int)(c1 - k0 < kStage ? c1 - k0 : kStage);
        if (threadIdx.x < kStage) sid[threadIdx.x] = threadIdx.x < nk ? a.sidx[(size_t)i * a.Ns + k0 + threadIdx.x] : 0;
        __syncthreads();
        for (int q = threadIdx.x; q < kStage * kTile; q += blockDim.x) {
            const int k = q / kTile, c = q - k * kTile;
            double gv = 0.0, hv = 0.0;
            if (k < nk) {
                const int64_t s = sid[k];
                const double* g;
                const double* h;
                int eg, eh;
                if (a.an.chain) {
                    g = a.Renv + ((size_t)s * (K + 1) + i + 1) * D;
                    eg = a.Rexp[(size_t)s * (K + 1) + i + 1];
                    h = a.Lenv + ((size_t)s * (K + 1) + i) * D;
                    eh = a.Lexp[(size_t)s * (K + 1) + i];
                } else {
                    g = a.Gst + ((size_t)s * K + i) * D;
                    eg = a.Gexp[(size_t)s * K + i];
                    h = j < 0 ? nullptr : a.Hst + ((size_t)s * K + j) * D;
                    eh = j < 0 ? 0 : a.Hexp[(size_t)s * K + j];
                }
                const double w = ldexp(a.u[s] / a.psi_mant[s], eg + eh - a.psi_exp[s]);
                if (a0 + c < D) gv = w * g[a0 + c];
                if (b0 + c < D) hv = h ? h[b0 + c] : (b0 + c == 0 ? 1.0 : 0.0);
            }
            gS[k][c] = gv;
            hS[k][c] = hv;
        }
        __syncthreads();
        for (int k = 0; k < nk; ++k) {
            double gr[4], hr[4];
            #pragma unroll
            for (int u = 0; u < 4; ++u) { gr[u] = gS[k][ty * 4 + u]; hr[u] = hS[k][tx * 4 + u]; }
            #pragma unroll
            for (int u = 0; u < 4; ++u)
                #pragma unroll
                for (int v = 0; v < 4; ++v) acc[u][v] = fma(gr[u], hr[v], acc[u][v]);
        }
        __syncthreads();
    }
    double* out = a.part + (((size_t)chunk * a.an.n_edges + e) * 4 + sg) * D * D;
    #pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int ra = a0 + ty * 4 + u;
        if (ra >= D) continue;
        #pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int cb = b0 + tx * 4 + v;
            if (cb < D) out[(size_t)ra * D + cb] = acc[u][v];
        }
    }
}

// grad[e][s] = sum over the group's chunks, in chunk order.
__global__ void k_grad_reduce(GradArgs a)
{
    const int D = a.an.D;
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t per = (int64_t)4 * D * D;
    if (q >= (int64_t)a.an.n_edges * per) return;
    const int e = (int)(q / per);
    const int sg = (int)((q - e * per) / ((int64_t)D * D));
    int i;
    if (a.an.chain) i = e;
    else { int lo = 0; while (a.an.pred_ptr[lo + 1] <= e) ++lo; i = lo; }
    const int64_t n = a.soff[(size_t)i * 5 + sg + 1] - a.soff[(size_t)i * 5 + sg];
    const int64_t nck = (n + kGradChunk - 1) / kGradChunk;
    double acc = a.accumulate ? a.grad_sites[q] : 0.0;
    for (int64_t c = 0; c < nck; ++c) acc += a.part[(size_t)c * a.an.n_edges * per + q];
    a.grad_sites[q] = acc;
}

// v[s][k] = u_s d log|f(s)| / d theta_k
__global__ void k_grad_corr_v(GradArgs a)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= a.Ns * a.an.n_hidden) return;
    a.vcorr[q] = a.u[q / a.an.n_hidden] * corr_dlog(a.an.corr, a.theta[q]);
}

// One chunk of samples and 32 hidden units per block (one per lane): warp w
// sums the columns w, w + 8, ... (spin orbitals 0..2K-1, then b at 2K). The
// samples' words are uniform over a warp, so an unoccupied column costs no FP64
// add. With one thread per parameter over all samples, each re-evaluating
// tanh, the same sums took 4.2 ms for H50 (4096 samples, N_h = 100); the FP64
// adds alone need 0.04 ms.
constexpr int kCorrCols = 2 * kMaxOrb / 8 + 1;

__global__ void __launch_bounds__(256) k_grad_rbm(GradArgs a, int64_t chunk)
{
    const int K2 = 2 * a.an.K, NH = a.an.n_hidden;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.y * 32 + lane;
    const int64_t s0 = (int64_t)blockIdx.x * chunk;
    const int64_t s1 = s0 + chunk < a.Ns ? s0 + chunk : a.Ns;
    double acc[kCorrCols];
    #pragma unroll
    for (int j = 0; j < kCorrCols; ++j) acc[j] = 0.0;
    for (int64_t s = s0; s < s1; ++s) {
        const uint64_t w0 = __ldg(a.samples + 2 * s), w1 = __ldg(a.samples + 2 * s + 1);
        const double v = k < NH ? a.vcorr[s * NH + k] : 0.0;
        #pragma unroll
        for (int j = 0; j < kCorrCols; ++j) {
            const int col = warp + 8 * j;
            if (col > K2) continue;
            if (col == K2 || (((col & 1) ? w1 : w0) >> (col >> 1)) & 1ull) acc[j] += v;
        }
    }
    if (k >= NH) return;
    double* out = a.cpart + ((size_t)blockIdx.x * (K2 + 1)) * NH + k;
    #pragma unroll
    for (int j = 0; j < kCorrCols; ++j) {
        const int col = warp + 8 * j;
        if (col <= K2) out[(size_t)col * NH] = acc[j];
    }
}

__global__ void k_grad_rbm_reduce(GradArgs a, int64_t chunks)
{
    const int K2 = 2 * a.an.K, NH = a.an.n_hidden;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (K2 + 1) * NH) return;
    const int col = q / NH, k = q - col * NH;
    double* g = col == K2 ? (a.grad_b ? a.grad_b + k : nullptr)
                          : (a.grad_W ? a.grad_W + (size_t)k * K2 + col : nullptr);
    if (!g) return;
    double acc = a.accumulate ? *g : 0.0;
    for (int64_t c = 0; c < chunks; ++c) acc += a.cpart[(size_t)c * (K2 + 1) * NH + q];
    *g = acc;
}

__global__ void k_grad_w2(GradArgs a)
{
    const int k = blockIdx.x, K = a.an.K, NH = a.an.n_hidden, N = 2 * K;
    for (int q = threadIdx.x; q < N * N; q += blockDim.x) {
        const int s1 = q / N, s2 = q - s1 * N;
        double acc = 0.0;
        for (int64_t s = 0; s < a.Ns; ++s) {
            const uint64_t w1 = a.samples[2 * s + (s1 & 1)], w2 = a.samples[2 * s + (s2 & 1)];
            if (((w1 >> (s1 >> 1)) & 1ull) && ((w2 >> (s2 >> 1)) & 1ull))
                acc += 0.5 * a.vcorr[s * NH + k];
        }
        double* g = a.grad_W2 + ((size_t)k * N + s1) * N + s2;
        *g = (a.accumulate ? *g : 0.0) + acc;
    }
}

// Per-sample weights of the energy gradient: u_n = 2 c_n (E_loc(n) - E) / sum c
// (Eq. egrad); reweighted (Sec. 2.3): u_n = 2 c_n f~_n^2 (E_loc(n) - E) / sum c
// with f~^2 = f^2 / B = exp(2 log|f(n)| - log B) and E the mean of E~_loc.
__global__ void k_energy_weights(const double* e_loc, const double* counts, const double* log_f,
                                 int64_t Ns, double e_mean, double sum_c, double log_B, int reweighted,
                                 double* u)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= Ns) return;
    const double cn = counts ? counts[s] : 1.0;
    double w = 2.0 * cn / sum_c;
    if (reweighted) w *= exp(2.0 * log_f[s] - log_B);
    u[s] = w * (e_loc[s] - e_mean);
}

int launch_energy_weights(const double* e_loc, const double* counts, const double* log_f, int64_t Ns,
                          double e_mean, double sum_c, double log_B, bool reweighted, double* u,
                          cudaStream_t st)
{
    if (Ns == 0) return 0;
    k_energy_weights<<<(unsigned)((Ns + 255) / 256), 256, 0, st>>>(e_loc, counts, log_f, Ns, e_mean, sum_c,
                                                                   log_B, reweighted ? 1 : 0, u);
    return 1;
}

int launch_group_by_state(const uint64_t* samples, int64_t Ns, int K, int32_t* sidx, int64_t* soff, cudaStream_t st)
{
    k_group_by_state<<<K, 1024, 0, st>>>(samples, Ns, sidx, soff);
    return 1;
}

int launch_grad_fp64(const GradArgs& a, cudaStream_t st)
{
    const int D = a.an.D;
    int n = 0;
    if (a.grad_sites && a.Ns > 0) {
        launch_group_by_state(a.samples, a.Ns, a.an.K, a.sidx, a.soff, st);
        // fixed-point products where the width allows and the groups fill their
        // 64-sample reductions (a quarter of the samples each)
        if (fx_fits(D) && a.Ns >= kFxGradMin && a.err) {
            launch_fx_grad(a, grad_chunks(a.Ns), kGradChunk, a.err, st);
        } else {
            const int nt = (D + kTile - 1) / kTile;
            dim3 grid((unsigned)(nt * nt), (unsigned)grad_chunks(a.Ns), (unsigned)(a.an.n_edges * 4));
            k_grad_tn<<<grid, 256, 0, st>>>(a, nt);
        }
        const int64_t tot = (int64_t)a.an.n_edges * 4 * D * D;
        k_grad_reduce<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(a);
        n += 3;
    }
    const int NH = a.an.n_hidden;
    const bool w2 = a.grad_W2 && a.an.corr == 2;
    if (NH > 0 && a.Ns > 0 && (a.grad_W || a.grad_b || w2)) {
        k_grad_corr_v<<<(unsigned)((a.Ns * NH + 255) / 256), 256, 0, st>>>(a);
        ++n;
    }
    if (NH > 0 && a.Ns > 0 && (a.grad_W || a.grad_b)) {
        const int64_t nc = corr_chunks(a.Ns);
        k_grad_rbm<<<dim3((unsigned)nc, (unsigned)((NH + 31) / 32)), 256, 0, st>>>(a, corr_chunk(a.Ns));
        k_grad_rbm_reduce<<<(unsigned)(((2 * a.an.K + 1) * NH + 255) / 256), 256, 0, st>>>(a, nc);
        n += 2;
    }
    if (NH > 0 && a.Ns > 0 && w2) {
        k_grad_w2<<<a.an.n_hidden, 256, 0, st>>>(a);
        ++n;
    }
    return n;
}

}  // namespace nqs
