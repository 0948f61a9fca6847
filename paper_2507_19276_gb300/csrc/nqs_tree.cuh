// nqs_tree.cuh -- prefix trees of connected determinants (see nqs_tree.cu).
#pragma once

#include "nqs_kernels.cuh"

namespace nqs {

constexpr int kTreeRows = 128;            // rows per chunk of the row kernels

// A row's changed sites ascending, each as x = 3 site + alternative (the
// alternatives of a site are the three local states n does not have there, in
// ascending order), one byte each, the last repeated up to four.
__host__ __device__ __forceinline__ int tree_alt_state(int own, int a) { return a + (a >= own ? 1 : 0); }

struct TreeArgs {
    HamView h;
    const uint64_t* samples;              // all samples of the call
    int64_t s0;                           // batch = samples [s0, s0 + nb)
    int nb;
    int K;
    int full;                             // 1: every row is re-run to vertex K - 1 (a row is a node
                                          // itself); 0: a row ends on the node before its last change
    // rows: each sample's deterministic rows, then its drawn rows
    const uint32_t* det_rank; const int64_t* det_off; const int64_t* det_cnt; const double* det_coef;
    const uint32_t* draw_rank; int64_t draw_stride; const int64_t* draw_cnt; const double* draw_coef;   // or NULL
    const int64_t* row_base;              // [Ns+1] prefix of the samples' row counts
    const int64_t* chunk_base;            // [Ns+1] prefix of their chunks of kTreeRows
    // per batch row
    uint32_t* word;                       // changes (see above)
    uint32_t* rnode;                      // the node the row ends on
    // per batch sample
    int* e1;                              // [nb][3K] last level of the one-change nodes (-1 unused); e2 right behind
    int* e2;                              // [nb][3K][3K] the same of two-change nodes, then their index
    int* n2; int* n3;                     // [nb] two- and three-change nodes
    uint32_t* bits;                       // [nb][n2max][W] third changes of each two-change node
    uint32_t* bits_base;                  // [nb][n2max][W] three-change nodes before each word
    int n2max, W;
    // nodes: ids are roots [nb], one-change [nb][3K], two-change [nb][n2max],
    // three-change [rows], four-change [rows] (full)
    uint32_t id1, id2, id3, id4;          // first id of each kind
    uint32_t* parent;
    int* end;                             // last level the node is needed at (-1: none)
    uint32_t* start;                      // first level | new local state << 8
    uint32_t* base;                       // row of the state pool at level `start`, within the
                                          // sample's rows (a root: within the pool)
    // levels
    int64_t* pool_tot;                    // [nb + 1] pool rows per sample, then their prefix
    int64_t* level_cnt;                   // [K][4][nb] nodes per (level, local state, sample)
    int64_t* level_off;                   // their exclusive prefix (one more entry)
    uint32_t* items;                      // by (level, local state), see TreeLevels
    uint32_t pool0;                       // first pool row after the roots' rows [nb][K]
};

// Items of the levels: level t holds n[t] of them from `at[t]` of the items,
// first[t] before it in level_off's numbering. With sources, an item is the
// pool row its state goes to (level K - 1: its node) and, in n[t]-long arrays
// behind, the pool row of every vertex source of t's in-edges; else its node.
struct TreeLevels {
    uint32_t at[kMaxOrb], first[kMaxOrb], n[kMaxOrb];
    int sources;
};

// words, marks and nodes of the batch; fills pool_tot and level_cnt
int launch_tree_nodes(const TreeArgs& a, int64_t max_chunks, cudaStream_t st);
// pool rows of the nodes (pool_tot scanned) and the items (level_off scanned)
int launch_tree_items(const TreeArgs& a, const TreeLevels& lv, const int* pred_ptr, const int* pred_idx, cudaStream_t st);

// ---- node evaluations -------------------------------------------------------

// FP64 states of a chain or graph ansatz (linear readout): vertex t of every
// node of level t.
struct TreeGraph64 {
    AnsatzView an;                        // with the edge lists (a chain's too)
    const uint32_t* items;
    double* pool;                         // [rows][D]
    int* pool_e;                          // [rows]
};
int launch_tree_graph64(const TreeGraph64& a, int t, const TreeLevels& lv, const int64_t* bounds, cudaStream_t st);

// Covectors that close a row at its last changed vertex: for each (q,
// alternative a) and each vertex j < q read at or after q, Q_j with
// psi(m) = c + sum_j Q_j . h_j(node).
struct TreeClose {
    AnsatzView an;
    const uint64_t* samples; int64_t s0; int nb;
    const double* Gst; const int* Gexp;   // adjoints of n: sample s's vertex i at row s * g_stride + i
    int g_stride;
    const int* live_ptr; const int* live_idx;   // [K+1], vertices read at or after q
    int n_live;                           // live_ptr[K]
    double* Q; int* Qe;                   // [nb][n_live][3][D], [nb][n_live][3]
    double* c; int* ce;                   // [nb][K][3] the e_0 sources' part
};
int launch_tree_close(const TreeClose& a, cudaStream_t st);

// 2cosh correlator on the rows: cosh(theta + d) / cosh theta = A e^d + B e^-d
// with A = 1 / (1 + e^(-2 theta)), B = 1 - A, and e^d a product over the changed
// sites: expd [K][4 own][3 alternatives][n_hidden] = {e^d, e^-d} of one site's
// change d of theta_k, ab [samples][n_hidden] = {A, B}.
int launch_corr_exp(const double* W, int K, int n_hidden, double2* expd, cudaStream_t st);
int launch_corr_ab(const double* theta, int64_t n, double2* ab, cudaStream_t st);

struct TreeRows64 {
    TreeArgs t;
    TreeClose q;
    int chain;                            // the span of a chain's row ends at its last change
    const double2* expd; const double2* ab;   // NULL: no 2cosh correlator (ab: batch samples)
    const double* pool; const int* pool_e;
    const double* theta; const double* lc;
    const double* psi_mant; const int* psi_exp;
    double* partial; int64_t* span; int64_t* mv;
};
int launch_tree_rows64(const TreeRows64& a, int64_t max_chunks, cudaStream_t st);

// Mixed form of a graph ansatz: split-FP16 states, one vertex per launch.
// out[i] = off[i * stride] for i < n, then *last: what the host reads of a tree batch
int launch_tree_head(const int64_t* off, int stride, int n, const int64_t* last, int64_t* out, cudaStream_t st);
// the roots' states and powers of two (nb samples, K rows of D each out of src_rows
// per sample) into the pool's first rows
int launch_tree_roots(const double* h, const int* x, int src_rows, int nb, int K, int D, double* pool, int* pool_e,
                      cudaStream_t st);

struct TreeGraphTc {
    AnsatzView an;
    const uint32_t* items;
    unsigned char* pool;                  // [rows][hi D | lo D] FP16
    int* pool_e;
    const unsigned char* bimg; const int* bexp; const float* col0;
    float* mant; int* mexp;               // [nodes] psi_TN of the nodes of level K - 1
    DevError* err;
};
int launch_tree_graph_tc(const TreeGraphTc& a, int t, int deg, const TreeLevels& lv, const int64_t* bounds, int n_sm,
                         cudaStream_t st);

struct TreeRowsTc {
    TreeArgs t;
    int draws;                            // 0: the deterministic rows, 1: the drawn rows
    const int64_t* chunk_base;            // [Ns+1] chunks of kTreeRows of those rows
    const uint32_t* perm;                 // per batch row: the sample's rows of that kind sorted by
                                          // their first change (launch_tree_perm)
    AnsatzView an;
    const float* mant; const int* mexp;
    const float* tts; const float* WT; int np;
    const double* psi_mant; const int* psi_exp;
    double* partial; double* partial_abs; int64_t* span; int64_t* mv;
};
// stable order of each sample's deterministic and drawn rows by their first changed vertex
int launch_tree_perm(const TreeArgs& a, uint32_t* perm, cudaStream_t st);
int launch_tree_rows_tc(const TreeRowsTc& a, int64_t max_chunks, int n_sm, cudaStream_t st);
// split images and exponents of the roots' states into the pool, tanh theta
int launch_tree_graph_prep(const double* Hst, const int* Hexp, const double* theta, int64_t s0, int nb, int K, int D,
                           int NH, int NP, int corr, unsigned char* pool, int* pool_e, float* tts, cudaStream_t st);

// Normalised readout on a chain (D <= kTreeRnnMaxD): the nodes' running cell,
// weight and sign, in two buffers by level parity.
constexpr int kTreeRnnMaxD = 32;
struct TreeRnn {
    AnsatzView an;
    TreeArgs t;
    uint32_t n_nodes;
    const double* cells;                  // n's cells [Ns][K][D]
    double* cell;                         // [2][n_nodes][D]
    double* prod;                         // [2][n_nodes] prod of P / Z since the first change, times
    int* pex;                             // 2^(500 pex) ([2][n_nodes])
    uint32_t* flag;                       // [2][n_nodes] N_alpha | N_beta << 8 | odd << 16 | dead << 17
};
int launch_tree_rnn(const TreeRnn& a, int t, const TreeLevels& lv, const int64_t* bounds, int n_sm, cudaStream_t st);

struct TreeRowsRnn {
    TreeRnn r;
    const double* lp; const int8_t* sg;
    const double* theta; const double* lc;
    double* partial; int64_t* span;
};
int launch_tree_rows_rnn(const TreeRowsRnn& a, int64_t max_chunks, cudaStream_t st);

// ---- shared device helpers ---------------------------------------------------

constexpr uint32_t kNoNode = 0xffffffffu;

// sample (call index) of chunk b of the batch, -1 past its end
__device__ __forceinline__ int64_t tree_sample(const TreeArgs& a, const int64_t* chunk_base, int64_t b)
{
    if (b >= chunk_base[a.s0 + a.nb]) return -1;
    int64_t lo = a.s0, hi = a.s0 + a.nb - 1;
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (chunk_base[mid] <= b) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int64_t tree_sample(const TreeArgs& a, int64_t b) { return tree_sample(a, a.chunk_base, b); }

struct TreeWord {
    int c;                    // changes
    int x[4];
};

__device__ __forceinline__ TreeWord tree_unpack(uint32_t w)
{
    TreeWord r;
    for (int k = 0; k < 4; ++k) r.x[k] = (int)((w >> (8 * k)) & 255u);
    r.c = r.x[1] == r.x[0] ? 1 : (r.x[2] == r.x[1] ? 2 : (r.x[3] == r.x[2] ? 3 : 4));
    return r;
}

// pool row of vertex j's state seen from a node of batch sample sl (the node or
// an ancestor of it that lived at level j)
__device__ __forceinline__ uint32_t tree_source(const TreeArgs& a, int sl, uint32_t node, int j)
{
    int p = (int)(__ldg(a.start + node) & 255u);
    while (p > j) {
        node = __ldg(a.parent + node);
        p = (int)(__ldg(a.start + node) & 255u);
    }
    return __ldg(a.base + node) + (uint32_t)(j - p) + (node < a.id1 ? 0u : a.pool0 + (uint32_t)a.pool_tot[sl]);
}

// x 2^e with the exponent field where the result stays normal
__device__ __forceinline__ double scale_pow2(double x, int e)
{
    const long long bits = __double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7FF), ne = ex + e;
    if (ex != 0 && ex != 0x7FF && ne > 0 && ne < 0x7FF) return __longlong_as_double(bits + ((long long)e << 52));
    return ldexp(x, e);
}

// determinant of a row from its word
__device__ __forceinline__ void tree_det(const TreeWord& w, uint64_t na, uint64_t nb, uint64_t& ma, uint64_t& mb)
{
    ma = na;
    mb = nb;
    for (int k = 0; k < w.c; ++k) {
        const int p = w.x[k] / 3, sg = tree_alt_state(sigma_at(na, nb, p), w.x[k] - 3 * p);
        ma = (ma & ~(1ull << p)) | ((uint64_t)(sg & 1) << p);
        mb = (mb & ~(1ull << p)) | ((uint64_t)(sg >> 1) << p);
    }
}

__device__ __forceinline__ double tree_coef(const TreeArgs& t, int64_t s, int64_t r)
{
    const int64_t nd = t.det_cnt[s];
    return r < nd ? t.det_coef[t.det_off[s] + r] : t.draw_coef[s * t.draw_stride + (r - nd)];
}

struct TreeGroups {
    uint32_t b[5];            // item bounds of the four local states within the level
    int tile[5];              // their tiles
};

inline TreeGroups tree_groups(int t, const int64_t* bounds, int rows)
{
    TreeGroups g;
    g.tile[0] = 0;
    for (int k = 0; k < 5; ++k) g.b[k] = (uint32_t)(bounds[4 * t + k] - bounds[4 * t]);
    for (int k = 0; k < 4; ++k) g.tile[k + 1] = g.tile[k] + (int)((g.b[k + 1] - g.b[k] + rows - 1) / rows);
    return g;
}

__device__ __forceinline__ bool rnn_allowed(const AnsatzView& an, int i, int nad, int nbd, int s)
{
    if (an.mask_na < 0) return true;
    const int ea = nad + (s & 1), eb = nbd + (s >> 1), left = an.K - 1 - i;
    return ea <= an.mask_na && eb <= an.mask_nb && an.mask_na - ea <= left && an.mask_nb - eb <= left;
}

// Node `it` of a tile of level t chooses its local state sg: the normaliser over
// the allowed states, the phase's sign, the running weight and electron counts
// (cand [node][4][DP] the candidate cells, Pv [node][4] their weights).
__device__ __forceinline__ void tree_rnn_pick(const TreeRnn& a, int t, int it, int sg, uint32_t f, double prod, int pex, size_t out,
                                              const double* cand, int DP, const double* Pv, const double* rw, double rc)
{
    const AnsatzView& an = a.an;
    const int nad = (int)(f & 255u), nbd = (int)((f >> 8) & 255u);
    double Z = 0.0;
    for (int q = 0; q < 4; ++q)
        if (rnn_allowed(an, t, nad, nbd, q)) Z += Pv[it * 4 + q];
    const double P = Pv[it * 4 + sg];
    const double* h = cand + (size_t)(it * 4 + sg) * DP;
    double ph = rc;
    for (int c = 0; c < an.D; ++c) ph = fma(rw[c], h[c], ph);
    if (!rnn_allowed(an, t, nad, nbd, sg) || !(P > 0.0) || !(Z > 0.0)) f |= 1u << 17;
    else {
        const double q = P / Z;
        if (__double2hiint(q) >= 0x20B00000) {        // 2^-500 and above: the product stays normal
            prod *= q;
        } else {
            int ep, ez;
            const double m = frexp(P, &ep) / frexp(Z, &ez);
            const int k = (ez - ep) / 500;
            prod *= ldexp(m, ep - ez + 500 * k);
            pex -= k;
        }
        if (prod < 0x1p-500) { prod *= 0x1p500; --pex; }
        f ^= ph < 0.0 ? 1u << 16 : 0u;
    }
    a.prod[out] = prod;
    a.pex[out] = pex;
    a.flag[out] = f + (uint32_t)(sg & 1) + ((uint32_t)(sg >> 1) << 8);
}

}  // namespace nqs
