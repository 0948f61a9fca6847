// nqs_rnn.cu -- the normalised MPS-RNN / BDG-RNN readout of Sec. 2.2 and the
// autoregressive sampling it allows (Sec. 2.1, Sec. 3), in FP64 on CUDA cores.
//
// Vertex i (= spatial orbital i, the computation order) forms four candidate
// memory cells h_i^s = sum_{e=(j->i)} M_e^s h_j + v_i^s from the cells of the
// local states already chosen (Eq. MPS-RNN-1D; Eq. bdg-rnn-update without the
// tensor term), h_{-1} = e_0. P_i(s) = sum_a eta_i[a] (h_i^s[a])^2 is
// normalised over the local states the N_alpha / N_beta constraint of Sec. 3
// still allows, and Phi(n) = prod_i sqrt(P~_i(s_i)) sign(w_i . h_i^{s_i} + c_i).
//
// Local energy: a connected m shares n's prefix up to its first changed
// vertex p, so its cells and conditionals agree with n's below p; vertices
// p..K-1 are re-run for m (chains up to D = 32 over prefix trees, k_tree_rnn;
// else one warp per row, k_rnn_amp) and divided by n's suffix
// of conditionals and signs. The normalisers depend on the whole prefix, so
// there is no right environment: the cost per amplitude is (K - p) x 4 cell
// products.
//
// Sampling: breadth first over the vertices. A node of level i is a distinct
// prefix holding `cnt` of the batch's draws at offsets off..off+cnt-1 (the
// nodes of a level tile the draws in prefix order). Draw j picks local state
// s at vertex i with u_j = Philox4x64-10(key (seed, 0), counter (j, i, 1, 0))
// as the first allowed s with u_j Z < sum_{allowed s' <= s} P_i(s') (the last
// allowed state when rounding leaves none); the children keep the offsets in
// the order of s, so the result does not depend on how nodes are scheduled.
#include "nqs_tree.cuh"

#include <algorithm>

namespace nqs {

namespace {

__device__ __forceinline__ double warp_allsum(double v)
{
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// One warp: the four candidate cells of vertex i into cand[4][D] (shared
// memory) and P_i(s) on every lane. src(j) gives the cell of vertex j >= 0;
// the boundary source j = -1 is e_0 (M e_0 = column 0 of M).
template <class Src>
__device__ void rnn_vertex_warp(const AnsatzView& an, int i, const Src& src, double* cand,
                                double P[4], int lane, double* tkz)
{
    const int D = an.D;
    const int e0 = an.chain ? i : an.pred_ptr[i];
    const int e1 = an.chain ? i + 1 : an.pred_ptr[i + 1];
    // tensor term (BDG-TensorRNN): the sources' projections once, the core of
    // every local state, z [d][r] then y [4][r] in the scratch
    const bool tk = tk_has(an, i);
    const int rk = tk ? an.tk_rank[i] : 0;
    const int dr = tk ? tk_degree(an, i) * rk : 0;
    if (tk) {
        tk_project(an, i, src, tkz, lane, 32);
        __syncwarp();
        for (int s = 0; s < 4; ++s) tk_core(an, i, s, tkz, tkz + dr + s * rk, lane, 32);
        __syncwarp();
    }
    // the 4 D candidate entries spread over the lanes (local state, component)
    for (int q = lane; q < 4 * D; q += 32) {
        const int s = q / D, r = q - s * D;
        double acc = __ldg(an.rv + ((size_t)i * 4 + s) * D + r);
        for (int e = e0; e < e1; ++e) {
            const int j = an.chain ? e - 1 : an.pred_idx[e];
            const double* AT = an.AT + ((size_t)e * 4 + s) * D * D;    // AT[c][r] = M[r][c]
            if (j < 0) {
                acc += __ldg(AT + r);
            } else {
                acc += dot_col4(AT, src(j), D, r);
            }
        }
        if (tk) acc += tk_out(an, i, r, tkz + dr + s * rk);
        cand[q] = acc;
    }
    __syncwarp();                       // cand visible to every lane
    for (int s = 0; s < 4; ++s) {
        double p = 0.0;
        for (int r = lane; r < D; r += 32) {
            const double h = cand[s * D + r];
            p = fma(__ldg(an.reta + (size_t)i * D + r) * h, h, p);
        }
        P[s] = warp_allsum(p);
    }
}

// The conditional of local state `sg` at vertex i and the sign of its phase:
// returns 1/2 log P~_i(sg), -inf where the state is not allowed or has zero
// weight; *neg = (w_i . h + c_i < 0).
__device__ __forceinline__ double rnn_pick(const AnsatzView& an, int i, int nad, int nbd, int sg,
                                           const double* cand, const double P[4], int lane, int* neg)
{
    const int D = an.D;
    double Z = 0.0;
    for (int q = 0; q < 4; ++q)
        if (rnn_allowed(an, i, nad, nbd, q)) Z += P[q];
    double ph = 0.0;
    for (int r = lane; r < D; r += 32) ph = fma(__ldg(an.rw + (size_t)i * D + r), cand[sg * D + r], ph);
    ph = warp_allsum(ph) + __ldg(an.rc + i);
    *neg = ph < 0.0;
    if (!rnn_allowed(an, i, nad, nbd, sg) || !(P[sg] > 0.0) || !(Z > 0.0)) return -INFINITY;
    return 0.5 * (log(P[sg]) - log(Z));
}

}  // namespace

// ---------------------------------------------------------------------------
// psi(n): cells, conditionals and phase signs of every vertex (one warp per sample)
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(256) k_rnn_env(RnnEnvArgs a)
{
    extern __shared__ double sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t s = (int64_t)blockIdx.x * 8 + warp;
    if (s >= a.Ns) return;
    const AnsatzView& an = a.an;
    const int K = an.K, D = an.D;
    double* cand = sm + (size_t)warp * (4 * D + an.tk_zy);
    double* tkz = cand + 4 * D;
    const uint64_t na = a.samples[2 * s], nb = a.samples[2 * s + 1];
    double* cells = a.cells + (size_t)s * K * D;
    int nad = 0, nbd = 0, sign = 1;
    for (int i = 0; i < K; ++i) {
        double P[4];
        rnn_vertex_warp(an, i, [&](int j) { return (const double*)(cells + (size_t)j * D); }, cand, P, lane, tkz);
        const int sg = sigma_at(na, nb, i);
        int neg;
        const double lp = rnn_pick(an, i, nad, nbd, sg, cand, P, lane, &neg);
        if (lane == 0) {
            a.lp[(size_t)s * K + i] = lp;
            a.sg[(size_t)s * K + i] = neg ? -1 : 1;
        }
        if (lp == -INFINITY) sign = 0;
        else if (neg) sign = -sign;
        for (int r = lane; r < D; r += 32) cells[(size_t)i * D + r] = cand[sg * D + r];
        __syncwarp();
        nad += sg & 1;
        nbd += sg >> 1;
    }
    if (lane == 0) {
        const double lf = a.log_f[s];
        a.psi_mant[s] = (lf == -INFINITY) ? 0.0 : (double)sign;
        a.psi_exp[s] = 0;
    }
}

int launch_rnn_env(const RnnEnvArgs& a, cudaStream_t st)
{
    if (a.Ns == 0) return 0;
    const size_t smem = (size_t)8 * (4 * a.an.D + a.an.tk_zy) * sizeof(double);
    allow_max_smem(k_rnn_env);
    k_rnn_env<<<(unsigned)((a.Ns + 7) / 8), 256, smem, st>>>(a);
    return 1;
}

// ---------------------------------------------------------------------------
// Connected amplitudes: vertices p..K-1 re-run for m, one warp per row
// ---------------------------------------------------------------------------

constexpr int kRnnRows = 32;      // rows per block (one chunk of the row set)

int rnn_rows_per_block() { return kRnnRows; }

static int rnn_warps(const AnsatzView& an)
{
    const size_t per = ((size_t)(an.K + 4) * an.D + an.tk_zy) * sizeof(double);
    int w = (int)((200u << 10) / per);
    return w < 1 ? 1 : (w > 8 ? 8 : w);
}

__global__ void __launch_bounds__(256) k_rnn_amp(RnnAmpArgs a)
{
    extern __shared__ double sm[];
    __shared__ OrbLists lists;
    __shared__ double s_term[kRnnRows];
    __shared__ int s_span[kRnnRows];
    const AnsatzView& an = a.an;
    const int K = an.K, D = an.D;
    const int64_t b = blockIdx.x;
    const int64_t* cb = a.rows.chunk_base;
    if (b >= cb[a.Ns]) return;
    int64_t lo = 0, hi = a.Ns - 1;                  // largest s with cb[s] <= b
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (cb[mid] <= b) lo = mid; else hi = mid - 1;
    }
    const int64_t s = lo;
    const int64_t j = b - cb[s];
    const int64_t beg = a.rows.begin ? a.rows.begin[s] : s * a.rows.stride;
    const int64_t cnt = a.rows.count[s];
    const int64_t r0 = beg + j * kRnnRows;
    const int nr = (int)((cnt - j * kRnnRows) < kRnnRows ? (cnt - j * kRnnRows) : kRnnRows);
    const uint64_t na = a.samples[2 * s], nb = a.samples[2 * s + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (warp == 0) build_lists_warp(na, nb, a.h.K, lists, lane);
    __syncthreads();
    double* wc = sm + (size_t)warp * ((K + 4) * D + an.tk_zy);   // this warp's cells of m, [K][D]
    double* cand = wc + (size_t)K * D;
    double* tkz = cand + 4 * D;
    const double* cn = a.cells + (size_t)s * K * D;  // n's cells
    for (int r = warp; r < nr; r += nw) {
        const Exc e = decode_rank<false>(a.h, lists, a.rows.rank[r0 + r]);   // sites only
        uint64_t ma = na, mb = nb;
        flip(ma, mb, e.i); flip(ma, mb, e.a);
        if (e.kind == 2) { flip(ma, mb, e.j); flip(ma, mb, e.b); }
        const int p = __ffsll((long long)((na ^ ma) | (nb ^ mb))) - 1;
        int nad = __popcll(na & low_mask(p)), nbd = __popcll(nb & low_mask(p));
        double lpm = 0.0;
        int odd = 0;
        bool ok = true;
        for (int i = p; i < K; ++i) {
            double P[4];
            rnn_vertex_warp(an, i, [&](int jj) { return (const double*)(jj < p ? cn + (size_t)jj * D : wc + (size_t)jj * D); },
                            cand, P, lane, tkz);
            const int sg = sigma_at(ma, mb, i);
            int neg;
            const double lp = rnn_pick(an, i, nad, nbd, sg, cand, P, lane, &neg);
            if (lp == -INFINITY) ok = false;
            else { lpm += lp; odd ^= neg; }
            for (int c = lane; c < D; c += 32) wc[(size_t)i * D + c] = cand[sg * D + c];
            __syncwarp();
            nad += sg & 1;
            nbd += sg >> 1;
        }
        // n's suffix of conditionals and signs
        double lpn = 0.0;
        int oddn = 0;
        for (int i = p + lane; i < K; i += 32) {
            lpn += a.lp[(size_t)s * K + i];
            oddn ^= a.sg[(size_t)s * K + i] < 0;
        }
        for (int o = 16; o; o >>= 1) {
            lpn += __shfl_xor_sync(kFull, lpn, o);
            oddn ^= __shfl_xor_sync(kFull, oddn, o);
        }
        int negf;
        const double lr = corr_log_ratio_warp(an, s, a.theta, a.lc, na, nb, ma, mb, lane, &negf);
        if (lane == 0) {
            double t = 0.0;
            if (ok) {
                t = a.rows.coef[r0 + r] * exp(lpm - lpn + lr);
                if (odd ^ oddn ^ negf) t = -t;
            }
            s_term[r] = t;
            s_span[r] = K - p;
        }
        __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double acc = 0.0;
        int64_t sp = 0;
        for (int r = 0; r < nr; ++r) { acc += s_term[r]; sp += s_span[r]; }
        a.partial[b] = acc;
        if (a.span) a.span[b] = sp;
    }
}

// ---------------------------------------------------------------------------
// Chain readout over the prefix trees (nqs_tree.cu): one launch per vertex
// advances every node of its level. The normalisers depend on the whole prefix,
// so every row is continued to the last vertex; what rows share is the part up
// to their third change (H50 at eps = 0.01: 444 000 instead of 908 000 vertex
// updates per sample). FP64 bounds it (4 D^2 + 8 D operations per update at two
// per clock and SM): the vertex's four matrices sit in shared memory, each
// thread holds one candidate entry of four nodes, a thread per (node, local
// state) forms P, a thread per node the normaliser and the choice. The weight
// is kept as a product of P / Z (one division per update) instead of a sum of
// logarithms (two logs, a tenth of the operations at D = 10). The 32-row blocks
// that re-ran every row took 420 ms for 300 H50 samples (chi = 10).
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(256) k_tree_rnn(TreeRnn a, int t, uint32_t at, uint32_t nl, TreeGroups gr, int IT)
{
    extern __shared__ double sm[];
    __shared__ const double* s_src[64];
    __shared__ double s_prod[64];
    __shared__ int s_pex[64], s_sig[64];
    __shared__ uint32_t s_flag[64], s_node[64];
    const AnsatzView& an = a.an;
    const int K = an.K, D = an.D, DP = D | 1;        // padded rows: no bank conflicts across nodes
    double* AT4 = sm;                                // [4][D][D]: AT4[s][k][c] = M^s[c][k]
    double* rv = AT4 + (size_t)4 * D * D;            // [4][D]
    double* eta = rv + 4 * D;                        // [D]
    double* rw = eta + D;                            // [D]
    double* xs = rw + D;                             // [IT][D] the nodes' previous cells
    double* cand = xs + (size_t)IT * D;              // [IT][4][DP]
    double* Pv = cand + (size_t)IT * 4 * DP;         // [IT][4]
    const int tid = threadIdx.x;
    for (int q = tid; q < 4 * D * D; q += 256) AT4[q] = __ldg(an.AT + (size_t)t * 4 * D * D + q);
    for (int q = tid; q < 4 * D; q += 256) rv[q] = __ldg(an.rv + (size_t)t * 4 * D + q);
    for (int q = tid; q < D; q += 256) { eta[q] = __ldg(an.reta + (size_t)t * D + q); rw[q] = __ldg(an.rw + (size_t)t * D + q); }
    const double rc = __ldg(an.rc + t);
    const size_t cur = (size_t)(t & 1) * a.n_nodes, prv = (size_t)((t & 1) ^ 1) * a.n_nodes;
    const uint32_t nt = (nl + IT - 1) / IT;
    for (uint32_t tile = blockIdx.x; tile < nt; tile += gridDim.x) {
        const uint32_t i0 = tile * (uint32_t)IT;
        const int n = (int)min(nl - i0, (uint32_t)IT);
        __syncthreads();
        if (tid < n) {
            const uint32_t i = i0 + tid, node = __ldg(a.t.items + at + i);
            s_node[tid] = node;
            s_sig[tid] = (i >= gr.b[1]) + (i >= gr.b[2]) + (i >= gr.b[3]);
            uint32_t src = node;
            if ((int)(a.t.start[node] & 255u) == t) src = a.t.parent[node];
            if (src < a.t.id1) {                     // n itself up to here
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
        for (int q = tid; q < n * D; q += 256) {
            const int it = q / D, c = q - it * D;
            const double* src = s_src[it];
            xs[q] = src ? src[c] : (c == 0 ? 1.0 : 0.0);       // h_{-1} = e_0
        }
        __syncthreads();
        for (int q = tid; q < (IT / 4) * 4 * D; q += 256) {
            const int it = 4 * (q / (4 * D)), sc = q - it * D, sg = sc / D, c = sc - sg * D;
            if (it >= n) continue;
            const double* M = AT4 + (size_t)sg * D * D + c;
            const double* x = xs + (size_t)it * D;   // (rows past n hold older numbers, not used)
            double acc[4] = {0.0, 0.0, 0.0, 0.0};
            for (int k = 0; k < D; ++k) {
                const double m = M[(size_t)k * D];
                #pragma unroll
                for (int v = 0; v < 4; ++v) acc[v] = fma(m, x[v * D + k], acc[v]);
            }
            const double v0 = rv[sc];
            #pragma unroll
            for (int v = 0; v < 4; ++v) cand[((size_t)(it + v) * 4 + sg) * DP + c] = v0 + acc[v];
        }
        __syncthreads();
        for (int q = tid; q < n * 4; q += 256) {
            const double* h = cand + (size_t)q * DP;
            double p = 0.0;
            for (int c = 0; c < D; ++c) p = fma(eta[c] * h[c], h[c], p);
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
}

int launch_tree_rnn(const TreeRnn& a, int t, const TreeLevels& lv, const int64_t* bounds, int n_sm, cudaStream_t st)
{
    if (lv.n[t] == 0) return 0;
    const int D = a.an.D, IT = D <= 16 ? 64 : 32;
    const size_t smem = ((size_t)4 * D * D + 6 * D + (size_t)IT * D + (size_t)IT * 4 * (D | 1) + 4 * IT) * sizeof(double);
    allow_max_smem(k_tree_rnn);
    const uint32_t nt = (lv.n[t] + IT - 1) / IT;
    const int per = std::max(1, std::min(6, (int)((200u << 10) / smem)));
    k_tree_rnn<<<std::min<uint32_t>(nt, (uint32_t)(per * n_sm)), 256, smem, st>>>(a, t, lv.at[t], lv.n[t],
                                                                              tree_groups(t, bounds, IT), IT);
    return 1;
}

// Terms of the rows: a row's node holds its weight since the first change p, n's
// is the sum of its conditionals from p on.
__global__ void __launch_bounds__(kTreeRows) k_tree_rows_rnn(TreeRowsRnn a)
{
    __shared__ int64_t s_s;
    __shared__ double s_lp[kMaxOrb + 1], s_lr[kTreeRows], wsum[4];
    __shared__ int s_odd[kMaxOrb + 1], s_neg[kTreeRows], wspan[4];
    const TreeArgs& t = a.r.t;
    const AnsatzView& an = a.r.an;
    const int K = an.K, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t b = t.chunk_base[t.s0] + blockIdx.x;
    if (tid == 0) s_s = tree_sample(t, b);
    __syncthreads();
    const int64_t s = s_s;
    if (s < 0) return;
    const uint64_t na = t.samples[2 * s], nb = t.samples[2 * s + 1];
    const int64_t r0 = (b - t.chunk_base[s]) * kTreeRows, g0 = t.row_base[s] - t.row_base[t.s0] + r0;
    const int64_t left = t.row_base[s + 1] - t.row_base[s] - r0;
    const int nr = (int)(left < kTreeRows ? left : kTreeRows);
    if (tid <= K) {
        double lp = 0.0;
        int odd = 0;
        for (int i = K - 1; i >= tid; --i) {
            lp += a.lp[(size_t)s * K + i];
            odd ^= a.sg[(size_t)s * K + i] < 0;
        }
        s_lp[tid] = lp;
        s_odd[tid] = odd;
    }
    if (an.n_hidden > 0)
        for (int rr = warp; rr < nr; rr += kTreeRows / 32) {
            uint64_t ma, mb;
            tree_det(tree_unpack(t.word[g0 + rr]), na, nb, ma, mb);
            int neg;
            const double lr = corr_log_ratio_warp(an, s, a.theta, a.lc, na, nb, ma, mb, lane, &neg);
            if (lane == 0) { s_lr[rr] = lr; s_neg[rr] = neg; }
        }
    __syncthreads();
    double term = 0.0;
    int sp = 0;
    if (tid < nr) {
        const int p = (int)(t.word[g0 + tid] & 255u) / 3;
        const size_t at = (size_t)((K - 1) & 1) * a.r.n_nodes + t.rnode[g0 + tid];
        const uint32_t f = a.r.flag[at];
        sp = K - p;
        if (!((f >> 17) & 1u)) {
            const double lpm = 0.5 * (log(a.r.prod[at]) + (500.0 * 0.69314718055994530942) * a.r.pex[at]);
            term = tree_coef(t, s, r0 + tid) * exp(lpm - s_lp[p] + (an.n_hidden > 0 ? s_lr[tid] : 0.0));
            const int neg = (int)((f >> 16) & 1u) ^ s_odd[p] ^ (an.n_hidden > 0 ? s_neg[tid] : 0);
            if (neg) term = -term;
        }
    }
    term = warp_sum_f64(term);
    sp = (int)__reduce_add_sync(kFull, (unsigned)sp);
    if (lane == 0) { wsum[warp] = term; wspan[warp] = sp; }
    __syncthreads();
    if (tid == 0) {
        a.partial[b] = ((wsum[0] + wsum[1]) + wsum[2]) + wsum[3];
        if (a.span) a.span[b] = wspan[0] + wspan[1] + wspan[2] + wspan[3];
    }
}

int launch_tree_rows_rnn(const TreeRowsRnn& a, int64_t max_chunks, cudaStream_t st)
{
    if (max_chunks == 0) return 0;
    k_tree_rows_rnn<<<(unsigned)max_chunks, kTreeRows, 0, st>>>(a);
    return 1;
}

int launch_rnn_amp(const RnnAmpArgs& a, cudaStream_t st)
{
    if (a.rows.max_chunks == 0) return 0;
    const int w = rnn_warps(a.an);
    const size_t smem = (size_t)w * ((a.an.K + 4) * a.an.D + a.an.tk_zy) * sizeof(double);
    allow_max_smem(k_rnn_amp);
    k_rnn_amp<<<(unsigned)a.rows.max_chunks, 32 * w, smem, st>>>(a);
    return 1;
}

// ---------------------------------------------------------------------------
// Full evaluation of arbitrary determinants (nqs_amplitude), one warp each
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(256) k_rnn_full(AnsatzView an, const uint64_t* dets, int64_t n,
                                                  double* log_abs, int8_t* sign)
{
    extern __shared__ double sm[];
    const int K = an.K, D = an.D;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int64_t id = (int64_t)blockIdx.x * nw + warp;
    if (id >= n) return;
    double* wc = sm + (size_t)warp * ((K + 4) * D + an.tk_zy);
    double* cand = wc + (size_t)K * D;
    double* tkz = cand + 4 * D;
    const uint64_t na = dets[2 * id], nb = dets[2 * id + 1];
    int nad = 0, nbd = 0, odd = 0;
    bool ok = true;
    double lp_sum = 0.0;
    for (int i = 0; i < K; ++i) {
        double P[4];
        rnn_vertex_warp(an, i, [&](int jj) { return (const double*)(wc + (size_t)jj * D); }, cand, P, lane, tkz);
        const int sg = sigma_at(na, nb, i);
        int neg;
        const double lp = rnn_pick(an, i, nad, nbd, sg, cand, P, lane, &neg);
        if (lp == -INFINITY) ok = false;
        else { lp_sum += lp; odd ^= neg; }
        for (int c = lane; c < D; c += 32) wc[(size_t)i * D + c] = cand[sg * D + c];
        __syncwarp();
        nad += sg & 1;
        nbd += sg >> 1;
    }
    // correlator log|f| and its sign
    double lf = 0.0;
    int oddf = 0;
    for (int k = lane; k < an.n_hidden; k += 32) {
        const double th = corr_theta(an, k, na, nb);
        lf += corr_log_factor(an.corr, th);
        if (an.corr != 0) oddf ^= cos(th) < 0.0;
    }
    for (int o = 16; o; o >>= 1) {
        lf += __shfl_xor_sync(kFull, lf, o);
        oddf ^= __shfl_xor_sync(kFull, oddf, o);
    }
    if (lane == 0) {
        if (!ok || lf == -INFINITY) { sign[id] = 0; log_abs[id] = -INFINITY; }
        else { sign[id] = (odd ^ oddf) ? -1 : 1; log_abs[id] = lp_sum + lf; }
    }
}

int launch_rnn_full(const AnsatzView& an, const uint64_t* dets, int64_t n, double* log_abs,
                    int8_t* sign, cudaStream_t st)
{
    if (n == 0) return 0;
    const int w = rnn_warps(an);
    const size_t smem = (size_t)w * ((an.K + 4) * an.D + an.tk_zy) * sizeof(double);
    allow_max_smem(k_rnn_full);
    int launches = 0;
    const int64_t per = (int64_t)w * 65535 * 1024;
    for (int64_t i0 = 0; i0 < n; i0 += per) {
        const int64_t m = (n - i0) < per ? (n - i0) : per;
        k_rnn_full<<<(unsigned)((m + w - 1) / w), 32 * w, smem, st>>>(an, dets + 2 * i0, m, log_abs + i0,
                                                                     sign + i0);
        ++launches;
    }
    return launches;
}

// ---------------------------------------------------------------------------
// Autoregressive sampling, one level per launch pair
// ---------------------------------------------------------------------------

// Per node of level i (one warp): the candidate cells of vertex i from the
// node's prefix, then every draw of the node picks a local state.
__global__ void __launch_bounds__(256) k_sample_level(SampleLevel a)
{
    const AnsatzView& an = a.an;
    const int D = an.D, i = a.level;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t q = (int64_t)blockIdx.x * 8 + warp;
    if (q >= a.n_nodes) return;
    double* cand = a.cand + (size_t)q * 4 * D;
    extern __shared__ double sm[];
    double* tkz = sm + (size_t)warp * an.tk_zy;         // tensor-term scratch of this warp
    // cell of vertex jj (< i) of this node: level jj + 1 through the parent links
    auto src = [&](int jj) {
        int64_t idx = q;
        for (int l = i; l > jj + 1; --l) idx = a.parents[l][idx];
        return (const double*)(a.cells[jj + 1] + (size_t)idx * D);
    };
    double P[4];
    rnn_vertex_warp(an, i, src, cand, P, lane, tkz);
    const int nad = __popcll(a.pa[q]), nbd = __popcll(a.pb[q]);
    bool ok[4];
    int last = -1;
    double Z = 0.0;
    for (int s = 0; s < 4; ++s) {
        ok[s] = rnn_allowed(an, i, nad, nbd, s);
        if (ok[s]) { Z += P[s]; last = s; }
    }
    int64_t hist[4] = {0, 0, 0, 0};
    const int64_t o = a.off[q], c = a.cnt[q];
    for (int64_t j0 = 0; j0 < c; j0 += 32) {
        int pick = -1;
        if (j0 + lane < c) {
            const uint64_t x = philox_first4((uint64_t)(o + j0 + lane), (uint64_t)i, 1ull, a.seed);
            const double u = (double)(x >> 11) * 0x1.0p-53;
            const double t = u * Z;
            double cum = 0.0;
            pick = last;
            for (int s = 0; s < 4; ++s) {
                if (!ok[s]) continue;
                cum += P[s];
                if (t < cum) { pick = s; break; }
            }
        }
        for (int s = 0; s < 4; ++s) hist[s] += __popc(__ballot_sync(kFull, pick == s));
    }
    if (lane < 4) {
        a.child_cnt[(size_t)q * 4 + lane] = hist[lane];
        a.child_flag[(size_t)q * 4 + lane] = hist[lane] > 0 ? 1 : 0;
    }
}

int launch_sample_level(const SampleLevel& a, cudaStream_t st)
{
    if (a.n_nodes == 0) return 0;
    k_sample_level<<<(unsigned)((a.n_nodes + 7) / 8), 256, (size_t)8 * a.an.tk_zy * sizeof(double), st>>>(a);
    return 1;
}

// The children of level i's nodes: one per (node, local state) with draws,
// at the position of the exclusive scan of the counts (prefix order).
__global__ void k_sample_children(SampleChildren a)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= a.n_nodes * 4) return;
    const int64_t c = a.child_cnt[g];
    if (c == 0) return;
    const int64_t q = g >> 2;
    const int s = (int)(g & 3);
    const int64_t pos = a.child_pos[g];
    int64_t before = 0;
    for (int t = 0; t < s; ++t) before += a.child_cnt[q * 4 + t];
    a.qa[pos] = a.pa[q] | ((uint64_t)(s & 1) << a.level);
    a.qb[pos] = a.pb[q] | ((uint64_t)(s >> 1) << a.level);
    a.qoff[pos] = a.off[q] + before;
    a.qcnt[pos] = c;
    a.qparent[pos] = (int32_t)q;
    for (int r = 0; r < a.D; ++r) a.qcell[(size_t)pos * a.D + r] = a.cand[((size_t)q * 4 + s) * a.D + r];
}

int launch_sample_children(const SampleChildren& a, cudaStream_t st)
{
    if (a.n_nodes == 0) return 0;
    const int64_t n = a.n_nodes * 4;
    k_sample_children<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a);
    return 1;
}

// ---------------------------------------------------------------------------
// The descent in one launch (up to 2^17 draws, no tensor term): one
// 512-thread block per SM, two grid barriers per level and no host in between.
// Launch by launch (cells + draws, scan, children, and a wait for the node count
// per level) the H50 sampler spent 2.2 of its 3.3 ms in 150 kernels bound by
// their latency, the first levels in one warp that picked every draw of the one
// node.
//   phase 1: a block numbers the children of its run of level i - 1's nodes (it
//     counts the children before them: at most 4 cap integers from L2), writes
//     their words, offsets and links and the node of every draw, then forms the
//     candidate cells of vertex i: the 4 D entries of all its nodes dealt out
//     one per thread, eight lanes per P. FP64 bounds this (2 lanes per clock and
//     SM), so full warps matter: a warp per node with 40 entries at D = 10 and
//     32-lane sums took 60 FP64 warp instructions per node instead of ~25;
//   phase 2: a thread per draw picks its node's local state and adds to the
//     node's counts (integers: any order).
// The decisions are those of k_sample_level up to the order of P's sum.
// ---------------------------------------------------------------------------

constexpr int kTreeThreads = 512;

// Grid barrier of a cooperative launch; `gen` counts the barriers passed. Gives
// up (stop flag 1) after ~2^24 polls, then every block leaves.
__device__ bool tree_barrier(int* status, int gen)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(status, 1);
        const int want = gen * (int)gridDim.x;
        int ok = 0;
        for (int it = 0; it < (1 << 24); ++it) {
            int v;
            asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(status) : "memory");
            if (v >= want) { ok = 1; break; }
        }
        if (!ok) atomicExch(status + 1, 1);
        int stop;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(stop) : "l"(status + 1) : "memory");
        s_ok = ok && stop != 1;
    }
    __syncthreads();
    return s_ok != 0;
}

__global__ void __launch_bounds__(kTreeThreads) k_sample_tree(SampleTree a)
{
    constexpr int NW = kTreeThreads / 32;
    __shared__ int s_part[NW];
    __shared__ int s_link[kTreeThreads], s_off[kTreeThreads];
    __shared__ uint64_t s_wa[kTreeThreads], s_wb[kTreeThreads];
    __shared__ int s_end;
    const AnsatzView& an = a.an;
    const int K = an.K, D = an.D;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const size_t cap = (size_t)a.cap;
    auto cand_of = [&](int l) { return a.cand + (size_t)(a.keep ? l : l & 1) * cap * 4 * D; };   // cells of vertex l
    auto link_of = [&](int l) { return a.link + (size_t)(a.keep ? l : l & 1) * cap; };
    int gen = 0;
    for (int i = 0; i <= K; ++i) {
        const int cur = i & 1, prv = cur ^ 1;
        uint64_t* pa = a.pa + cur * cap;
        uint64_t* pb = a.pb + cur * cap;
        int* off = a.off + cur * cap;
        int* cnt = a.cnt + cur * cap;
        int* child = a.child + cur * cap * 4;
        // level 0 is the child of a node that holds every draw
        const int np = i == 0 ? 1 : *(volatile int*)(a.status + 4 + i - 1);
        const int* pc = a.child + prv * cap * 4;
        const int per = (np + (int)gridDim.x - 1) / (int)gridDim.x;
        const int q0 = min(np, (int)blockIdx.x * per), q1 = min(np, q0 + per);
        int base = 0;
        if (q0 < q1) {
            int before = 0;
            for (int g = tid; g < q0; g += kTreeThreads) {
                const int4 c = __ldcg((const int4*)pc + g);
                before += (c.x > 0) + (c.y > 0) + (c.z > 0) + (c.w > 0);
            }
            before = (int)__reduce_add_sync(kFull, (unsigned)before);
            if (lane == 0) s_part[warp] = before;
            __syncthreads();
            for (int w = 0; w < NW; ++w) base += s_part[w];
        }
        for (int g0 = q0; g0 < q1; g0 += kTreeThreads / 4) {       // block-uniform
            // (parent, local state) per thread; the block's scan of the existing children
            const int g = g0 + (tid >> 2), s = tid & 3;
            int c = 0;
            if (g < q1) c = i == 0 ? (s == 0 ? (int)a.n_samples : 0) : __ldcg(pc + 4 * (size_t)g + s);
            const unsigned bal = __ballot_sync(kFull, c > 0);
            int pre = c;                                             // draws of the quad up to s
            for (int o = 1; o < 4; o <<= 1) {
                const int u = __shfl_up_sync(kFull, pre, o, 4);
                if (s >= o) pre += u;
            }
            __syncthreads();                                         // s_part and the lists are free
            if (lane == 0) s_part[warp] = __popc(bal);
            __syncthreads();
            int at = __popc(bal & ((1u << lane) - 1u)), nch = 0;
            for (int w = 0; w < NW; ++w) { if (w < warp) at += s_part[w]; nch += s_part[w]; }
            if (c > 0) {
                uint64_t wa = 0, wb = 0;
                int o = 0;
                if (i > 0) {
                    wa = __ldcg(a.pa + prv * cap + g) | ((uint64_t)(s & 1) << (i - 1));
                    wb = __ldcg(a.pb + prv * cap + g) | ((uint64_t)(s >> 1) << (i - 1));
                    o = __ldcg(a.off + prv * cap + g) + pre - c;
                }
                const int q = base + at;
                pa[q] = wa;
                pb[q] = wb;
                off[q] = o;
                cnt[q] = c;
                link_of(i)[q] = g * 4 + s;
                *(int4*)(child + 4 * (size_t)q) = make_int4(0, 0, 0, 0);
                s_link[at] = g * 4 + s;
                s_wa[at] = wa;
                s_wb[at] = wb;
                s_off[at] = o;
                if (at == nch - 1) s_end = o + c;
            }
            __syncthreads();
            if (i < K && nch > 0) {
                // the node of every draw of these children (their draws are contiguous)
                for (int j = s_off[0] + tid; j < s_end; j += kTreeThreads) {
                    int lo = 0, hi = nch - 1;
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (s_off[mid] <= j) lo = mid; else hi = mid - 1;
                    }
                    a.node[j] = base + lo;
                }
                // candidate cells of vertex i (as in rnn_vertex_warp)
                const int e0 = an.chain ? i : an.pred_ptr[i], e1 = an.chain ? i + 1 : an.pred_ptr[i + 1];
                double* cand = cand_of(i) + (size_t)base * 4 * D;
                for (int q = tid; q < nch * 4 * D; q += kTreeThreads) {
                    const int x = q / (4 * D), sr = q - x * 4 * D, ss = sr / D, r = sr - ss * D;
                    double acc = __ldg(an.rv + ((size_t)i * 4 + ss) * D + r);
                    for (int e = e0; e < e1; ++e) {
                        const int j = an.chain ? e - 1 : an.pred_idx[e];
                        const double* AT = an.AT + ((size_t)e * 4 + ss) * D * D;
                        if (j < 0) {
                            acc += __ldg(AT + r);
                        } else {
                            int lk = s_link[x];                      // candidate of vertex i - 1
                            for (int l = i - 1; l > j; --l) lk = link_of(l)[lk >> 2];
                            acc += dot_col4(AT, cand_of(j) + (size_t)lk * D, D, r);
                        }
                    }
                    cand[q] = acc;
                }
                __syncthreads();
                // P and the thresholds, a warp per node, eight lanes per local state
                for (int x = warp; x < nch; x += NW) {
                    const double* h = cand + ((size_t)x * 4 + (lane >> 3)) * D;
                    double p = 0.0;
                    for (int r = lane & 7; r < D; r += 8) p = fma(__ldg(an.reta + (size_t)i * D + r) * h[r], h[r], p);
                    for (int o = 4; o; o >>= 1) p += __shfl_xor_sync(kFull, p, o);
                    const int nad = __popcll(s_wa[x]), nbd = __popcll(s_wb[x]);
                    int last = -1;
                    double Z = 0.0, thr = -1.0;
                    for (int t = 0; t < 4; ++t) {
                        const double pt = __shfl_sync(kFull, p, 8 * t);
                        if (!rnn_allowed(an, i, nad, nbd, t)) continue;
                        Z += pt;
                        if (lane == t) thr = Z;
                        last = t;
                    }
                    if (lane == 4) thr = Z;
                    if (lane == 5) thr = (double)last;
                    if (lane < 6) a.thr[6 * (size_t)(base + x) + lane] = thr;
                }
            }
            base += nch;
        }
        if (q0 < q1 && q1 == np && tid == 0) {               // the last node's block knows the total
            a.status[4 + i] = base;
            if (base == 0) atomicExch(a.status + 1, 1 + i);
        }
        if (!tree_barrier(a.status, ++gen)) return;
        if (*(volatile int*)(a.status + 4 + i) <= 0) return;
        if (i == K) break;
        const int64_t step = (int64_t)gridDim.x * kTreeThreads;
        for (int64_t j0 = (int64_t)blockIdx.x * kTreeThreads + warp * 32; j0 < a.n_samples; j0 += step) {
            const int64_t j = j0 + lane;                     // whole warps: the match below needs them
            int key = -1;
            if (j < a.n_samples) {
                const int q = __ldcg(a.node + j);
                const double* t = a.thr + 6 * (size_t)q;
                const double t0 = __ldcg(t), t1 = __ldcg(t + 1), t2 = __ldcg(t + 2), t3 = __ldcg(t + 3);
                const double Z = __ldcg(t + 4), last = __ldcg(t + 5);
                const uint64_t x = philox_first4((uint64_t)j, (uint64_t)i, 1ull, a.seed);
                const double tt = (double)(x >> 11) * 0x1.0p-53 * Z;
                // the first allowed state above tt
                const int pick = tt < t0 ? 0 : tt < t1 ? 1 : tt < t2 ? 2 : tt < t3 ? 3 : (int)last;
                if (pick >= 0) key = q * 4 + pick;
            }
            const unsigned same = __match_any_sync(kFull, key);
            if (key >= 0 && lane == __ffs(same) - 1) atomicAdd(child + key, __popc(same));
        }
        if (!tree_barrier(a.status, ++gen)) return;
    }
}

bool sample_tree_fits(const AnsatzView& an, int n_sm)
{
    int dev = 0, coop = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop || n_sm < 1 || an.tk_rank) return false;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_sample_tree, kTreeThreads, 0) == cudaSuccess && occ >= 1;
}

int launch_sample_tree(const SampleTree& a, int n_sm, cudaStream_t st)
{
    // blocks beyond one thread per draw would only wait
    const int64_t want = (a.n_samples + 31) / 32;
    const unsigned grid = (unsigned)(want < n_sm ? want : n_sm);
    SampleTree args = a;
    void* p[] = {&args};
    cudaLaunchCooperativeKernel(k_sample_tree, dim3(grid), dim3(kTreeThreads), p, 0, st);
    return 1;
}

__global__ void k_sample_tree_output(SampleTree a, int64_t n, uint64_t* dets, double* counts)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const size_t at = (size_t)(a.an.K & 1) * a.cap + q;
    dets[2 * q] = a.pa[at];
    dets[2 * q + 1] = a.pb[at];
    counts[q] = (double)a.cnt[at];
}

int launch_sample_tree_output(const SampleTree& a, int64_t n, uint64_t* dets, double* counts, cudaStream_t st)
{
    if (n == 0) return 0;
    k_sample_tree_output<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a, n, dets, counts);
    return 1;
}

// The last level's nodes as determinants [n][2] and counts (as doubles).
__global__ void k_sample_output(const uint64_t* pa, const uint64_t* pb, const int64_t* cnt, int64_t n,
                                uint64_t* dets, double* counts)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    dets[2 * q] = pa[q];
    dets[2 * q + 1] = pb[q];
    counts[q] = (double)cnt[q];
}

int launch_sample_output(const uint64_t* pa, const uint64_t* pb, const int64_t* cnt, int64_t n,
                         uint64_t* dets, double* counts, cudaStream_t st)
{
    if (n == 0) return 0;
    k_sample_output<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(pa, pb, cnt, n, dets, counts);
    return 1;
}

}  // namespace nqs
