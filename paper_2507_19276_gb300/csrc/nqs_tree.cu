// nqs_tree.cu -- prefix trees of the connected determinants of a sample.
//
// A connected m differs from n on two to four sites. Everything an ansatz
// computes vertex by vertex up to vertex t depends on m's local states at the
// vertices up to t, so rows that share their first changes share the work up to
// the next one. A node is a distinct prefix of changes (site, new local state)
// together with n's states in between; it lives on the levels (vertices) from
// its last change to the last level some row needs it at, and continues its
// parent (the prefix without the last change; n itself is the root). On H18 at
// eps = 0 a sample's 9 315 rows re-run 139 700 vertices from their first change
// to the end; their tree has 51 900 (node, level) pairs, and 15 200 when a row
// stops before its last change (a linear readout: the rest is one covector per
// (site, alternative), see k_tree_close). H50 at eps = 0.01: 908 000 against
// 444 000.
//
// Building a batch's trees: the rows mark one- and two-change prefixes in
// tables indexed by change pairs, the two-change ones are numbered, third
// changes become bits of a row of 3K per two-change node (their rank is a
// popcount), and four-change rows are nodes of their own. Node ids are fixed
// regions per sample, so no count is read back before the pool of states is
// sized. Per level the nodes' ids are grouped by local state (one matrix per
// in-edge and group).
#include "nqs_tree.cuh"

namespace nqs {

namespace {

// Words of the rows, and the levels their one- and two-change prefixes are
// needed to (a prefix that a later change follows: one level before it; a
// whole row, full form: K - 1).
__global__ void __launch_bounds__(kTreeRows) k_tree_mark(TreeArgs a)
{
    __shared__ OrbLists lists;
    __shared__ int64_t s_s;
    if (threadIdx.x == 0) s_s = tree_sample(a, a.chunk_base[a.s0] + blockIdx.x);
    __syncthreads();
    const int64_t s = s_s;
    if (s < 0) return;
    const int64_t b = a.chunk_base[a.s0] + blockIdx.x;
    const uint64_t na = a.samples[2 * s], nb = a.samples[2 * s + 1];
    if (threadIdx.x < 32) build_lists_warp(na, nb, a.h.K, lists, threadIdx.x);
    __syncthreads();
    const int64_t r = (b - a.chunk_base[s]) * kTreeRows + threadIdx.x;
    if (r >= a.row_base[s + 1] - a.row_base[s]) return;
    const int64_t nd = a.det_cnt[s];
    const uint32_t rank = r < nd ? a.det_rank[a.det_off[s] + r] : a.draw_rank[s * a.draw_stride + (r - nd)];
    const Exc e = decode_rank<false>(a.h, lists, rank);
    uint64_t ma = na, mb = nb;
    flip(ma, mb, e.i); flip(ma, mb, e.a);
    if (e.kind == 2) { flip(ma, mb, e.j); flip(ma, mb, e.b); }
    uint64_t ch = (na ^ ma) | (nb ^ mb);
    int x[4], c = 0;
    #pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (ch) {
            const int p = __ffsll((long long)ch) - 1;
            ch &= ch - 1;
            const int own = sigma_at(na, nb, p), nw = sigma_at(ma, mb, p);
            x[k] = 3 * p + nw - (nw > own ? 1 : 0);
            ++c;
        } else {
            x[k] = k ? x[k - 1] : 0;
        }
    }
    a.word[a.row_base[s] - a.row_base[a.s0] + r] =
        (uint32_t)x[0] | ((uint32_t)x[1] << 8) | ((uint32_t)x[2] << 16) | ((uint32_t)x[3] << 24);
    const int T = 3 * a.K, sl = (int)(s - a.s0);
    int* e1 = a.e1 + (size_t)sl * T + x[0];
    const int n1 = c >= 2 ? x[1] / 3 - 1 : (a.full ? a.K - 1 : -1);
    if (*(volatile int*)e1 < n1) atomicMax(e1, n1);
    const int n2 = c >= 3 ? x[2] / 3 - 1 : (c == 2 && a.full ? a.K - 1 : -1);
    if (n2 >= 0) {
        int* e2 = a.e2 + ((size_t)sl * T + x[0]) * T + x[1];
        if (*(volatile int*)e2 < n2) atomicMax(e2, n2);
    }
}

// block-wide exclusive scan (one value per thread), total in *tot
__device__ __forceinline__ int block_excl(int v, int* sh, int* tot)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int incl = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += u;
    }
    __syncthreads();
    if (lane == 31) sh[warp] = incl;
    __syncthreads();
    int before = 0, t = 0;
    for (int w = 0; w < nw; ++w) { if (w < warp) before += sh[w]; t += sh[w]; }
    *tot = t;
    return before + incl - v;
}

// One block per sample: roots, one-change nodes, and the two-change nodes in
// the order of their changes (their table entries become indices), and the third
// changes' bits cleared.
__global__ void __launch_bounds__(512) k_tree_two(TreeArgs a)
{
    __shared__ int sh[16];
    const int sl = blockIdx.x, T = 3 * a.K;
    const int64_t s = a.s0 + sl;
    const uint64_t na = a.samples[2 * s], nb = a.samples[2 * s + 1];
    if (threadIdx.x == 0) {
        a.parent[sl] = kNoNode;
        a.start[sl] = 0;
        a.end[sl] = -1;
        a.base[sl] = (uint32_t)(sl * a.K);
    }
    for (int x = threadIdx.x; x < T; x += blockDim.x) {
        const uint32_t id = a.id1 + (uint32_t)(sl * T + x);
        const int p = x / 3;
        a.parent[id] = (uint32_t)sl;
        a.start[id] = (uint32_t)p | ((uint32_t)tree_alt_state(sigma_at(na, nb, p), x - 3 * p) << 8);
        a.end[id] = a.e1[(size_t)sl * T + x];
    }
    int* e2 = a.e2 + (size_t)sl * T * T;
    const uint32_t first = a.id2 + (uint32_t)sl * (uint32_t)a.n2max;
    int carry = 0;
    for (int q0 = 0; q0 < T * T; q0 += 512 * 4) {
        int e[4], cnt = 0;
        #pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int q = q0 + 4 * (int)threadIdx.x + k;
            e[k] = q < T * T ? e2[q] : -1;
            cnt += e[k] >= 0;
        }
        int tot;
        int at = carry + block_excl(cnt, sh, &tot);
        carry += tot;
        #pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (e[k] < 0) continue;
            const int q = q0 + 4 * (int)threadIdx.x + k;
            const int x1 = q / T, x2 = q - x1 * T, p = x2 / 3;
            const uint32_t id = first + (uint32_t)at;
            a.parent[id] = a.id1 + (uint32_t)(sl * T + x1);
            a.start[id] = (uint32_t)p | ((uint32_t)tree_alt_state(sigma_at(na, nb, p), x2 - 3 * p) << 8);
            a.end[id] = e[k];
            e2[q] = at++;
        }
    }
    uint32_t* bits = a.bits + (size_t)sl * a.n2max * a.W;
    for (int q = threadIdx.x; q < carry * a.W; q += blockDim.x) bits[q] = 0;
    if (threadIdx.x == 0) a.n2[sl] = carry;
}

// rows -> (sample, row of the sample, batch row); false past the end
__device__ __forceinline__ bool tree_row(const TreeArgs& a, int64_t& s, int64_t& r, int64_t& g)
{
    __shared__ int64_t s_s;
    const int64_t b = a.chunk_base[a.s0] + blockIdx.x;
    if (threadIdx.x == 0) s_s = tree_sample(a, b);
    __syncthreads();
    s = s_s;
    if (s < 0) return false;
    r = (b - a.chunk_base[s]) * kTreeRows + threadIdx.x;
    g = a.row_base[s] - a.row_base[a.s0] + r;
    return r < a.row_base[s + 1] - a.row_base[s];
}

// third changes
__global__ void __launch_bounds__(kTreeRows) k_tree_bits(TreeArgs a)
{
    int64_t s, r, g;
    if (!tree_row(a, s, r, g)) return;
    const TreeWord w = tree_unpack(a.word[g]);
    if (w.c < (a.full ? 3 : 4)) return;
    const int T = 3 * a.K, sl = (int)(s - a.s0);
    const int i2 = a.e2[((size_t)sl * T + w.x[0]) * T + w.x[1]];
    uint32_t* bits = a.bits + ((size_t)sl * a.n2max + i2) * a.W + (w.x[2] >> 5);
    const uint32_t m = 1u << (w.x[2] & 31);
    if (!(*(volatile uint32_t*)bits & m)) atomicOr(bits, m);
}

// One block per sample: ranks of the third changes' bits, the three-change nodes.
__global__ void __launch_bounds__(512) k_tree_three(TreeArgs a)
{
    __shared__ int sh[16];
    const int sl = blockIdx.x;
    const int64_t s = a.s0 + sl;
    const uint64_t na = a.samples[2 * s], nb = a.samples[2 * s + 1];
    const int words = a.n2[sl] * a.W;
    const uint32_t* bits = a.bits + (size_t)sl * a.n2max * a.W;
    uint32_t* base = a.bits_base + (size_t)sl * a.n2max * a.W;
    const uint32_t first = a.id3 + (uint32_t)(a.row_base[s] - a.row_base[a.s0]);
    int carry = 0;
    for (int q0 = 0; q0 < words; q0 += 512) {
        const int q = q0 + threadIdx.x;
        uint32_t m = q < words ? bits[q] : 0u;
        int tot;
        int at = carry + block_excl(__popc(m), sh, &tot);
        carry += tot;
        if (q < words) base[q] = (uint32_t)at;
        const int i2 = q / a.W, x0 = (q - i2 * a.W) * 32;
        while (m) {
            const int x = x0 + __ffs((int)m) - 1, p = x / 3;
            m &= m - 1;
            const uint32_t id = first + (uint32_t)at++;
            a.parent[id] = a.id2 + (uint32_t)sl * (uint32_t)a.n2max + (uint32_t)i2;
            a.start[id] = (uint32_t)p | ((uint32_t)tree_alt_state(sigma_at(na, nb, p), x - 3 * p) << 8);
            a.end[id] = -1;
        }
    }
    if (threadIdx.x == 0) a.n3[sl] = carry;
}

// The node each row ends on, the levels three-change nodes are needed to, and
// (full form) the four-change rows' own nodes.
__global__ void __launch_bounds__(kTreeRows) k_tree_rows(TreeArgs a)
{
    int64_t s, r, g;
    if (!tree_row(a, s, r, g)) return;
    const TreeWord w = tree_unpack(a.word[g]);
    const int T = 3 * a.K, sl = (int)(s - a.s0);
    const int depth = a.full ? w.c : w.c - 1;             // changes of the node the row ends on
    uint32_t id1 = depth <= 0 ? (uint32_t)sl : a.id1 + (uint32_t)(sl * T + w.x[0]);
    uint32_t node = id1;
    if (depth >= 2) {
        const int i2 = a.e2[((size_t)sl * T + w.x[0]) * T + w.x[1]];
        node = a.id2 + (uint32_t)sl * (uint32_t)a.n2max + (uint32_t)i2;
        if (depth >= 3) {
            const size_t q = ((size_t)sl * a.n2max + i2) * a.W + (w.x[2] >> 5);
            const uint32_t below = a.bits[q] & ((1u << (w.x[2] & 31)) - 1u);
            node = a.id3 + (uint32_t)(a.row_base[s] - a.row_base[a.s0]) + a.bits_base[q] + (uint32_t)__popc(below);
            const int n3 = w.c == 4 ? w.x[3] / 3 - 1 : a.K - 1;
            int* e3 = a.end + node;
            if (*(volatile int*)e3 < n3) atomicMax(e3, n3);
        }
    }
    if (a.full) {
        const uint32_t id = a.id4 + (uint32_t)g;
        if (depth == 4) {
            const int p = w.x[3] / 3;
            const uint64_t na = a.samples[2 * s], nb = a.samples[2 * s + 1];
            a.parent[id] = node;
            a.start[id] = (uint32_t)p | ((uint32_t)tree_alt_state(sigma_at(na, nb, p), w.x[3] - 3 * p) << 8);
            a.end[id] = a.K - 1;
            node = id;
        } else {
            a.end[id] = -1;
        }
    }
    a.rnode[g] = node;
}

// the q-th node slot of a sample (one-, two-, three-, then four-change)
struct TreeSlots {
    int T, n2, n3, rows;
    uint32_t f1, f2, f3, f4;
    __device__ TreeSlots(const TreeArgs& a, int sl)
    {
        const int64_t s = a.s0 + sl;
        const uint32_t rb = (uint32_t)(a.row_base[s] - a.row_base[a.s0]);
        T = 3 * a.K;
        n2 = a.n2[sl];
        n3 = a.n3[sl];
        rows = a.full ? (int)(a.row_base[s + 1] - a.row_base[s]) : 0;
        f1 = a.id1 + (uint32_t)(sl * T);
        f2 = a.id2 + (uint32_t)sl * (uint32_t)a.n2max;
        f3 = a.id3 + rb;
        f4 = a.id4 + rb;
    }
    __device__ int total() const { return T + n2 + n3 + rows; }
    __device__ uint32_t id(int q) const
    {
        if (q < T) return f1 + (uint32_t)q;
        q -= T;
        if (q < n2) return f2 + (uint32_t)q;
        q -= n2;
        return q < n3 ? f3 + (uint32_t)q : f4 + (uint32_t)(q - n3);
    }
};

// One block per sample: pool rows (relative) of its nodes, their number, and
// the nodes per (level, local state): those that start there with their new
// state, the others with n's.
__global__ void __launch_bounds__(512) k_tree_count(TreeArgs a)
{
    __shared__ int sh[16];
    __shared__ int s_cnt[4 * kMaxOrb], s_diff[kMaxOrb + 1];
    const int sl = blockIdx.x, K = a.K;
    const int64_t s = a.s0 + sl;
    for (int q = threadIdx.x; q < 4 * K; q += blockDim.x) s_cnt[q] = 0;
    for (int q = threadIdx.x; q <= K; q += blockDim.x) s_diff[q] = 0;
    __syncthreads();
    const TreeSlots sl_(a, sl);
    const int n = sl_.total();
    int carry = 0;
    for (int q0 = 0; q0 < n; q0 += 512) {
        const int q = q0 + threadIdx.x;
        int len = 0;
        uint32_t id = 0;
        if (q < n) {
            id = sl_.id(q);
            const uint32_t st = a.start[id];
            const int p = (int)(st & 255u), e = a.end[id];
            if (e >= p) {
                len = e - p + 1;
                atomicAdd(&s_cnt[4 * p + (int)(st >> 8)], 1);
                if (e > p) { atomicAdd(&s_diff[p + 1], 1); atomicAdd(&s_diff[e + 1], -1); }
            }
        }
        int tot;
        const int at = carry + block_excl(len, sh, &tot);
        carry += tot;
        if (len) a.base[id] = (uint32_t)at;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a.pool_tot[sl] = carry;
        const uint64_t na = a.samples[2 * s], nb = a.samples[2 * s + 1];
        int alive = 0;
        for (int t = 0; t < K; ++t) {
            alive += s_diff[t];
            s_cnt[4 * t + sigma_at(na, nb, t)] += alive;
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < 4 * K; q += blockDim.x) a.level_cnt[(size_t)q * a.nb + sl] = s_cnt[q];
}

// One block per sample: the items of every level. A warp walks its nodes' levels
// together: one atomic per level and local state. The sources are resolved here,
// where a node's ancestors sit in registers: left to the level kernels, the walk
// (four to eight dependent loads per in-edge) was most of a tile's 13 us.
__global__ void __launch_bounds__(512) k_tree_items(TreeArgs a, TreeLevels lv, const int* __restrict__ pred_ptr,
                                                    const int* __restrict__ pred_idx)
{
    __shared__ uint32_t cur[4 * kMaxOrb];
    __shared__ int s_ptr[kMaxOrb + 1];
    __shared__ short s_idx[kMaxOrb * 8];
    const int sl = blockIdx.x, K = a.K;
    const int lane = threadIdx.x & 31;
    const int64_t s = a.s0 + sl;
    const uint64_t na = a.samples[2 * s], nb = a.samples[2 * s + 1];
    for (int q = threadIdx.x; q < 4 * K; q += blockDim.x) cur[q] = (uint32_t)a.level_off[(size_t)q * a.nb + sl] - lv.first[q >> 2];
    if (lv.sources) {
        for (int q = threadIdx.x; q <= K; q += blockDim.x) s_ptr[q] = pred_ptr[q];
        const int E = pred_ptr[K];
        for (int q = threadIdx.x; q < E; q += blockDim.x) s_idx[q] = (short)pred_idx[q];
    }
    __syncthreads();
    const TreeSlots slots(a, sl);
    const int n = slots.total();
    const uint32_t pool = a.pool0 + (uint32_t)a.pool_tot[sl];
    for (int q0 = (int)(threadIdx.x & ~31u); q0 < n; q0 += blockDim.x) {
        const int q = q0 + lane;
        uint32_t id = 0;
        int p = kMaxOrb, e = -1, nw = 0;
        // the node and its ancestors: state of vertex j (start <= j) at row
        // off + j; those past the root repeat it
        int st[4] = {0, 0, 0, 0};
        uint32_t off[5] = {0, 0, 0, 0, 0};
        if (q < n) {
            id = slots.id(q);
            const uint32_t w = a.start[id];
            const int en = a.end[id];
            if (en >= (int)(w & 255u)) {
                p = (int)(w & 255u);
                e = en;
                nw = (int)(w >> 8);
                uint32_t x = id;
                for (int k = 0; k < 4 && lv.sources; ++k) {
                    if (x < a.id1) break;                  // the root: off stays to be set below
                    st[k] = (int)(a.start[x] & 255u);
                    off[k] = pool + a.base[x] - (uint32_t)st[k];
                    x = a.parent[x];
                }
                #pragma unroll
                for (int k = 0; k < 5; ++k)
                    if (off[k] == 0) off[k] = (uint32_t)(sl * K);      // (a node's row is at least pool0 - start > 0)
            }
        }
        const int t0 = __reduce_min_sync(kFull, p), t1 = __reduce_max_sync(kFull, e);
        for (int t = t0; t <= t1; ++t) {
            const bool on = t >= p && t <= e;
            const int sg = t == p ? nw : sigma_at(na, nb, t);
            uint32_t pos = 0;
            #pragma unroll
            for (int g = 0; g < 4; ++g) {
                const unsigned bal = __ballot_sync(kFull, on && sg == g);
                if (!bal) continue;
                uint32_t at = 0;
                if (lane == __ffs((int)bal) - 1) at = atomicAdd(&cur[4 * t + g], (uint32_t)__popc(bal));
                at = __shfl_sync(kFull, at, __ffs((int)bal) - 1);
                if (sg == g) pos = at + (uint32_t)__popc(bal & ((1u << lane) - 1u));
            }
            if (!on) continue;
            uint32_t* out = a.items + lv.at[t] + pos;
            if (!lv.sources) {
                *out = id;
                continue;
            }
            *out = t == K - 1 ? id : off[0] + (uint32_t)t;
            for (int k = s_ptr[t]; k < s_ptr[t + 1]; ++k) {
                const int j = s_idx[k];
                if (j < 0) continue;
                out += lv.n[t];
                const uint32_t o = j >= st[0] ? off[0] : j >= st[1] ? off[1] : j >= st[2] ? off[2] : j >= st[3] ? off[3] : off[4];
                *out = o + (uint32_t)j;
            }
        }
    }
}

// Stable counting sort by the first changed vertex, one block per (sample, kind
// of row): the order in which the mixed form adds its terms.
__global__ void __launch_bounds__(256) k_tree_perm(TreeArgs a, uint32_t* perm)
{
    __shared__ int off[kMaxOrb];                  // next position of each vertex
    __shared__ int wc[8][kMaxOrb];                // per-warp counts of the current 256 rows
    const int64_t s = a.s0 + blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nd = (int)a.det_cnt[s], all = (int)(a.row_base[s + 1] - a.row_base[s]);
    const int r0 = blockIdx.y ? nd : 0, cnt = blockIdx.y ? all - nd : nd;
    const uint32_t* word = a.word + (a.row_base[s] - a.row_base[a.s0]) + r0;
    perm += (a.row_base[s] - a.row_base[a.s0]) + r0;
    for (int q = tid; q < 8 * kMaxOrb; q += 256) (&wc[0][0])[q] = 0;
    if (tid < kMaxOrb) off[tid] = 0;
    __syncthreads();
    for (int c0 = 0; c0 < cnt; c0 += 256) {
        const int p = c0 + tid < cnt ? (int)(word[c0 + tid] & 255u) / 3 : -1;
        const unsigned m = __match_any_sync(kFull, p);
        if (p >= 0 && lane == __ffs((int)m) - 1) atomicAdd(&off[p], __popc(m));
    }
    __syncthreads();
    if (tid == 0) {
        int acc = 0;
        for (int v = 0; v < a.K; ++v) { const int c = off[v]; off[v] = acc; acc += c; }
    }
    __syncthreads();
    const unsigned below = (1u << lane) - 1u;
    for (int c0 = 0; c0 < cnt; c0 += 256) {
        const int r = c0 + tid;
        const bool valid = r < cnt;
        const int p = valid ? (int)(word[r] & 255u) / 3 : -1;
        const unsigned m = __match_any_sync(kFull, p);
        if (valid && lane == __ffs((int)m) - 1) wc[warp][p] = __popc(m);
        __syncthreads();
        if (valid) {
            int pos = off[p] + __popc(m & below);
            for (int w = 0; w < warp; ++w) pos += wc[w][p];
            perm[pos] = (uint32_t)(r0 + r);
        }
        __syncthreads();
        if (tid < a.K) {
            int t = 0;
            for (int w = 0; w < 8; ++w) { t += wc[w][tid]; wc[w][tid] = 0; }
            off[tid] += t;
        }
        __syncthreads();
    }
}

// 2^d as a double, 0 below the normal range (d <= 0)
__device__ __forceinline__ double pow2_neg64(int d)
{
    return d >= -1022 ? __longlong_as_double((long long)(1023 + d) << 52) : 0.0;
}

}  // namespace

int launch_tree_nodes(const TreeArgs& a, int64_t max_chunks, cudaStream_t st)
{
    const size_t T = (size_t)3 * a.K;
    cudaMemsetAsync(a.e1, 0xff, (char*)(a.e2 + a.nb * T * T) - (char*)a.e1, st);
    if (max_chunks > 0) k_tree_mark<<<(unsigned)max_chunks, kTreeRows, 0, st>>>(a);
    k_tree_two<<<a.nb, 512, 0, st>>>(a);
    if (max_chunks > 0) k_tree_bits<<<(unsigned)max_chunks, kTreeRows, 0, st>>>(a);
    k_tree_three<<<a.nb, 512, 0, st>>>(a);
    if (max_chunks > 0) k_tree_rows<<<(unsigned)max_chunks, kTreeRows, 0, st>>>(a);
    k_tree_count<<<a.nb, 512, 0, st>>>(a);
    return max_chunks > 0 ? 6 : 3;
}

int launch_tree_perm(const TreeArgs& a, uint32_t* perm, cudaStream_t st)
{
    k_tree_perm<<<dim3(a.nb, a.draw_cnt ? 2 : 1), 256, 0, st>>>(a, perm);
    return 1;
}

int launch_tree_items(const TreeArgs& a, const TreeLevels& lv, const int* pred_ptr, const int* pred_idx, cudaStream_t st)
{
    k_tree_items<<<a.nb, 512, 0, st>>>(a, lv, pred_ptr, pred_idx);
    return 1;
}

// ---------------------------------------------------------------------------
// FP64 states of a graph ansatz, one vertex of the nodes of a group
// ---------------------------------------------------------------------------

namespace {

// x 2^e: a change of the exponent field while both are normal numbers
__device__ __forceinline__ double tree_scale(double x, int e)
{
    const int hi = __double2hiint(x), f = (hi >> 20) & 0x7FF, g = f + e;
    if (f > 0 && f < 0x7FF && g > 0 && g < 0x7FF) return __hiloint2double(hi + e * (1 << 20), __double2loint(x));
    return x == 0.0 ? x : ldexp(x, e);
}

// A tile of IT items: per in-edge the sources' vectors in shared memory, a
// column for four items per thread (the matrix entries come through L1, one
// load per four FMAs; FP64 at 2 lanes per clock and SM bounds this), the edges'
// sums aligned by powers of two, one warp per item renormalising in integers (at
// D = 8 most lanes of an FP64 operation carry nothing, and each takes the pipe for
// 16 clocks). Small levels are latency: the seven of K8 (250 samples) take 81 us,
// with FP64 maxima, ldexp and one matrix load in flight 184 us.
__global__ void __launch_bounds__(256) k_tree_graph64(TreeGraph64 a, int t, uint32_t at, uint32_t nl, TreeGroups gr, int IT)
{
    extern __shared__ double sm[];
    __shared__ uint32_t s_src[8][32];
    __shared__ int s_ex[8][32], s_er[32];
    __shared__ uint32_t s_out[32];
    const int D = a.an.D;
    double* xs = sm;                                  // [IT][D] sources, then the sums
    int g = 0;
    while (g < 3 && (int)blockIdx.x >= gr.tile[g + 1]) ++g;
    const uint32_t i0 = gr.b[g] + (uint32_t)((int)blockIdx.x - gr.tile[g]) * (uint32_t)IT;
    const int n = (int)min(gr.b[g + 1] - i0, (uint32_t)IT);
    const int e0 = a.an.pred_ptr[t], e1 = a.an.pred_ptr[t + 1];
    // one warp per in-edge: the items' sources and their powers of two
    {
        const int w = threadIdx.x >> 5, it = threadIdx.x & 31;
        if (w < e1 - e0 && it < n) {
            int x = 0, slot = 0;
            for (int e = e0; e < e0 + w; ++e) slot += a.an.pred_idx[e] >= 0;
            if (a.an.pred_idx[e0 + w] >= 0) {
                const uint32_t r = __ldg(a.items + at + (size_t)(slot + 1) * nl + i0 + it);
                s_src[w][it] = r;
                x = a.pool_e[r];
            }
            s_ex[w][it] = x;
        }
        if (w == 7 && it < n) s_out[it] = __ldg(a.items + at + i0 + it);
    }
    __syncthreads();
    if ((int)threadIdx.x < n) {
        int er = -1000000;
        for (int k = 0; k < e1 - e0; ++k) er = max(er, s_ex[k][threadIdx.x]);
        s_er[threadIdx.x] = er;
    }
    // (group of four items, column) tasks of this thread
    const int tasks = (IT / 4) * D;
    double y[2][4];
    #pragma unroll
    for (int u = 0; u < 2; ++u)
        #pragma unroll
        for (int v = 0; v < 4; ++v) y[u][v] = 0.0;
    for (int e = e0; e < e1; ++e) {
        const int j = a.an.pred_idx[e];
        const double* AT = a.an.AT + ((size_t)e * 4 + g) * D * D;
        __syncthreads();
        if (j >= 0) {
            for (int q = threadIdx.x; q < n * D; q += 256) {
                const int it = q / D, c = q - it * D;
                xs[q] = a.pool[(size_t)s_src[e - e0][it] * D + c];
            }
            __syncthreads();
        }
        #pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int q = threadIdx.x + 256 * u;
            if (q >= tasks) continue;
            const int it = 4 * (q / D), c = q - (it >> 2) * D;
            if (it >= n) continue;
            double acc[4] = {0.0, 0.0, 0.0, 0.0};
            if (j < 0) {
                const double m = __ldg(AT + c);
                for (int v = 0; v < 4; ++v) acc[v] = m;
            } else {
                // (the tile's rows past n hold older numbers: their sums are not stored)
                const double* x = xs + (size_t)it * D;
                #pragma unroll 8
                for (int k = 0; k < D; ++k) {
                    const double m = __ldg(AT + (size_t)k * D + c);
                    #pragma unroll
                    for (int v = 0; v < 4; ++v) acc[v] = fma(m, x[v * D + k], acc[v]);
                }
            }
            #pragma unroll
            for (int v = 0; v < 4; ++v)
                if (it + v < n) y[u][v] += acc[v] * pow2_neg64(s_ex[e - e0][it + v] - s_er[it + v]);
        }
    }
    __syncthreads();
    #pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int q = threadIdx.x + 256 * u;
        if (q >= tasks) continue;
        const int it = 4 * (q / D), c = q - (it >> 2) * D;
        #pragma unroll
        for (int v = 0; v < 4; ++v)
            if (it + v < n) xs[(size_t)(it + v) * D + c] = y[u][v];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int it = threadIdx.x >> 5; it < n; it += 8) {
        const double* v = xs + (size_t)it * D;
        // the largest exponent field gives frexp's exponent of the largest magnitude,
        // and the scaling is a change of that field, in integers; zero, denormal and
        // non-finite rows take the general functions
        int top = 0;
        for (int c = lane; c < D; c += 32) top = max(top, (__double2hiint(v[c]) >> 20) & 0x7FF);
        top = __reduce_max_sync(kFull, top);
        const uint32_t row = s_out[it];
        int ex = 0;
        if (top > 0 && top < 0x7FF) {
            ex = top - 1022;
            for (int c = lane; c < D; c += 32) a.pool[(size_t)row * D + c] = tree_scale(v[c], -ex);
        } else {
            double m = 0.0;
            for (int c = lane; c < D; c += 32) m = fmax(m, fabs(v[c]));
            m = warp_max_f64(m);
            if (m != 0.0) frexp(m, &ex);
            for (int c = lane; c < D; c += 32) a.pool[(size_t)row * D + c] = ldexp(v[c], -ex);
        }
        if (lane == 0) a.pool_e[row] = s_er[it] + ex;
    }
}

}  // namespace

int launch_tree_graph64(const TreeGraph64& a, int t, const TreeLevels& lv, const int64_t* bounds, cudaStream_t st)
{
    const int D = a.an.D;
    // at most two (four items, column) tasks per thread
    int IT = 2048 / D / 4 * 4;
    IT = IT < 4 ? 4 : (IT > 32 ? 32 : IT);
    const TreeGroups g = tree_groups(t, bounds, IT);
    if (g.tile[4] == 0) return 0;
    k_tree_graph64<<<(unsigned)g.tile[4], 256, (size_t)IT * D * 8, st>>>(a, t, lv.at[t], lv.n[t], g, IT);
    return 1;
}

// ---------------------------------------------------------------------------
// Closing covectors. With the linear readout psi is linear in the states of the
// vertices below q given the local states from q on: for m equal to n above q
// and local state s at q,
//   psi(m) = sum_{j < q} h_j . [ sum_{e: j->i, i > q} M_e^{s_i(n) T} g_i(n)
//                               + sum_{e: j->q} M_e^{s T} g_q(n) ] + e_0 sources,
// g_i(n) = d psi / d h_i at n's states above (the adjoints). One block per
// (sample, q).
// ---------------------------------------------------------------------------

namespace {

// z[c] += 2^? M^T g in shared memory with a running power of two (block-wide)
__device__ void close_add(double* z, int* zx, const double* M, const double* g, int gx, int D, bool first)
{
    const int e = first ? gx : (*zx > gx ? *zx : gx);
    const double fz = first ? 0.0 : pow2_neg64(*zx - e), fg = pow2_neg64(gx - e);
    for (int c = threadIdx.x; c < D; c += blockDim.x) {
        double acc = 0.0;
        for (int r = 0; r < D; ++r) acc = fma(g[r], __ldg(M + (size_t)r * D + c), acc);
        z[c] = (first ? 0.0 : z[c] * fz) + acc * fg;
    }
    __syncthreads();
    if (threadIdx.x == 0) *zx = e;
    __syncthreads();
}

__global__ void __launch_bounds__(64) k_tree_close(TreeClose a)
{
    extern __shared__ double sm[];
    __shared__ int zx, cx;
    __shared__ double cv;
    const AnsatzView& an = a.an;
    const int K = an.K, D = an.D;
    double* z = sm;                                   // n's part of the current j
    double* g = sm + D;                               // an adjoint
    const int sl = blockIdx.x / K, q = blockIdx.x - sl * K;
    const int64_t s = a.s0 + sl;
    const uint64_t na = a.samples[2 * s], nb = a.samples[2 * s + 1];
    const int own = sigma_at(na, nb, q);
    auto load_g = [&](int i) {
        __syncthreads();
        for (int c = threadIdx.x; c < D; c += blockDim.x) g[c] = a.Gst[((size_t)s * a.g_stride + i) * D + c];
        __syncthreads();
        return a.Gexp[(size_t)s * a.g_stride + i];
    };
    for (int lj = a.live_ptr[q]; lj < a.live_ptr[q + 1]; ++lj) {
        const int j = a.live_idx[lj];
        bool first = true;
        for (int i = q + 1; i < K; ++i)
            for (int e = an.pred_ptr[i]; e < an.pred_ptr[i + 1]; ++e) {
                if (an.pred_idx[e] != j) continue;
                const int gx = load_g(i);
                close_add(z, &zx, an.A + ((size_t)e * 4 + sigma_at(na, nb, i)) * D * D, g, gx, D, first);
                first = false;
            }
        for (int alt = 0; alt < 3; ++alt) {
            const int sg = tree_alt_state(own, alt);
            double* out = a.Q + (((size_t)sl * a.n_live + lj) * 3 + alt) * D;
            // the alternative's part on top of n's, aligned
            int ex = first ? -1000000 : zx;
            for (int e = an.pred_ptr[q]; e < an.pred_ptr[q + 1]; ++e)
                if (an.pred_idx[e] == j) { const int gx = a.Gexp[(size_t)s * a.g_stride + q]; ex = gx > ex ? gx : ex; }
            const int gx = load_g(q);
            for (int c = threadIdx.x; c < D; c += blockDim.x) {
                double v = first ? 0.0 : z[c] * pow2_neg64(zx - ex);
                for (int e = an.pred_ptr[q]; e < an.pred_ptr[q + 1]; ++e) {
                    if (an.pred_idx[e] != j) continue;
                    const double* M = an.A + ((size_t)e * 4 + sg) * D * D;
                    double acc = 0.0;
                    for (int r = 0; r < D; ++r) acc = fma(g[r], __ldg(M + (size_t)r * D + c), acc);
                    v += acc * pow2_neg64(gx - ex);
                }
                out[c] = v;
            }
            if (threadIdx.x == 0) a.Qe[((size_t)sl * a.n_live + lj) * 3 + alt] = ex;
        }
        __syncthreads();
    }
    // e_0 sources: of q with the alternative, of later vertices with n's states
    for (int alt = 0; alt < 3; ++alt) {
        __syncthreads();
        if (threadIdx.x == 0) { cv = 0.0; cx = -1000000; }
        for (int i = q; i < K; ++i)
            for (int e = an.pred_ptr[i]; e < an.pred_ptr[i + 1]; ++e) {
                if (an.pred_idx[e] >= 0) continue;
                const int gx = load_g(i);
                if (threadIdx.x < 32) {
                    const int sg = i == q ? tree_alt_state(own, alt) : sigma_at(na, nb, i);
                    const double* col = an.AT + ((size_t)e * 4 + sg) * D * D;      // row 0 of the transpose
                    double acc = 0.0;
                    for (int r = threadIdx.x; r < D; r += 32) acc = fma(g[r], __ldg(col + r), acc);
                    acc = warp_sum_f64(acc);
                    if (threadIdx.x == 0) {
                        const int x = gx > cx ? gx : cx;
                        cv = cv * pow2_neg64(cx - x) + acc * pow2_neg64(gx - x);
                        cx = x;
                    }
                }
                __syncthreads();
            }
        __syncthreads();
        if (threadIdx.x == 0) {
            a.c[((size_t)sl * K + q) * 3 + alt] = cv;
            a.ce[((size_t)sl * K + q) * 3 + alt] = cx;
        }
    }
}

constexpr int kRowLanes = 8;

// Rows of the FP64 form: eight lanes per row dot the live states of the row's
// node with the closing covectors and take the correlator ratio as a product
// (9 FP64 operations per hidden unit; log 2cosh of every unit and row was ~80
// and 40% of the H18 time). A row one of whose lanes leaves 2^-125 .. 2^125 on the
// way is redone as a sum of logarithms, as the cos forms are: the eight lanes' product
// then stays a normal number whatever the order, where one that passed through the
// denormal numbers would come back with few bits.
__global__ void __launch_bounds__(256) k_tree_rows64(TreeRows64 a)
{
    __shared__ int64_t s_s;
    __shared__ double s_term[kTreeRows];
    __shared__ int s_span[kTreeRows], s_mv[kTreeRows];
    __shared__ unsigned char s_log[kTreeRows];
    const TreeArgs& t = a.t;
    const AnsatzView& an = a.q.an;
    const int64_t b = t.chunk_base[t.s0] + blockIdx.x;
    if (threadIdx.x == 0) s_s = tree_sample(t, b);
    __syncthreads();
    const int64_t s = s_s;
    if (s < 0) return;
    const int K = an.K, D = an.D, NH = an.n_hidden, sl = (int)(s - t.s0);
    const uint64_t na = t.samples[2 * s], nb = t.samples[2 * s + 1];
    const int64_t r0 = (b - t.chunk_base[s]) * kTreeRows, g0 = t.row_base[s] - t.row_base[t.s0] + r0;
    const int64_t left = t.row_base[s + 1] - t.row_base[s] - r0;
    const int nr = (int)(left < kTreeRows ? left : kTreeRows);
    const int l8 = threadIdx.x & 7, lane = threadIdx.x & 31;
    const double mant = a.psi_mant[s];
    const int pex = a.psi_exp[s];
    for (int rr = threadIdx.x >> 3; rr < kTreeRows; rr += 32) {      // whole warps: the shuffles need them
        const bool on = rr < nr;
        double tn = 0.0, ratio = 1.0;
        uint32_t top = 0x3FF00000u, bottom = 0x3FF00000u;            // of the running products' high words
        int er = 0;
        TreeWord w{};
        if (on) {
            w = tree_unpack(t.word[g0 + rr]);
            const uint32_t node = t.rnode[g0 + rr];
            const int x = w.x[w.c - 1], q = x / 3, alt = x - 3 * q;
            const size_t ci = ((size_t)sl * K + q) * 3 + alt;
            const int v0 = a.q.live_ptr[q], v1 = a.q.live_ptr[q + 1];
            er = a.q.ce[ci];
            for (int v = v0; v < v1; ++v) {
                const uint32_t row = tree_source(t, sl, node, a.q.live_idx[v]);
                const int e = a.pool_e[row] + a.q.Qe[((size_t)sl * a.q.n_live + v) * 3 + alt];
                er = e > er ? e : er;
            }
            tn = l8 == 0 ? a.q.c[ci] * pow2_neg64(a.q.ce[ci] - er) : 0.0;
            for (int v = v0; v < v1; ++v) {
                const uint32_t row = tree_source(t, sl, node, a.q.live_idx[v]);
                const size_t qi = ((size_t)sl * a.q.n_live + v) * 3 + alt;
                const double* hj = a.pool + (size_t)row * D;
                const double* Qj = a.q.Q + qi * D;
                double d = 0.0;
                for (int c = l8; c < D; c += kRowLanes) d = fma(__ldg(Qj + c), hj[c], d);
                tn = fma(d, pow2_neg64(a.pool_e[row] + a.q.Qe[qi] - er), tn);
            }
            if (a.expd) {
                const double2* ex[4];
                for (int k = 0; k < 4; ++k) {
                    const int p = w.x[k] / 3;
                    ex[k] = a.expd + (size_t)((p * 4 + sigma_at(na, nb, p)) * 3 + w.x[k] - 3 * p) * NH;
                }
                const double2* ab = a.ab + (size_t)sl * NH;
                for (int k = l8; k < NH; k += kRowLanes) {
                    const double2 h = __ldg(ab + k);
                    double2 e = __ldg(ex[0] + k);
                    for (int c = 1; c < w.c; ++c) {
                        const double2 f = __ldg(ex[c] + k);
                        e.x *= f.x;
                        e.y *= f.y;
                    }
                    ratio *= fma(h.x, e.x, h.y * e.y);
                    const uint32_t hw = (uint32_t)__double2hiint(ratio);      // (not negative; or a NaN)
                    top = max(top, hw);
                    bottom = min(bottom, hw);
                }
            }
        }
        for (int o = 4; o; o >>= 1) {
            tn += __shfl_xor_sync(kFull, tn, o);
            ratio *= __shfl_xor_sync(kFull, ratio, o);
        }
        const bool wide = top >= (1023u + 125u) << 20 || bottom < (1023u - 125u) << 20;
        const unsigned wides = __ballot_sync(kFull, wide) >> (lane & 24) & 255u;
        if (on && l8 == 0) {
            const int p = w.x[0] / 3;
            const bool by_log = NH > 0 && (!a.expd || wides);
            const double coef = tree_coef(t, s, r0 + rr);
            s_term[rr] = coef * scale_pow2(tn / mant, er - pex) * (by_log ? 1.0 : ratio);
            s_span[rr] = a.chain ? w.x[w.c - 1] / 3 - p + 1 : K - p;
            s_mv[rr] = graph_matvecs(an, p);
            s_log[rr] = by_log;
        }
    }
    __syncthreads();
    for (int rr = threadIdx.x >> 5; rr < nr; rr += 8) {
        if (!s_log[rr]) continue;                                    // uniform over the warp
        const TreeWord w = tree_unpack(t.word[g0 + rr]);
        uint64_t ma, mb;
        tree_det(w, na, nb, ma, mb);
        int neg;
        const double lr = corr_log_ratio_warp(an, s, a.theta, a.lc, na, nb, ma, mb, lane, &neg);
        if (lane == 0) s_term[rr] *= (neg ? -1.0 : 1.0) * exp(lr);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        double term = 0.0;
        int sp = 0, mv = 0;
        for (int rr = lane; rr < nr; rr += 32) { term += s_term[rr]; sp += s_span[rr]; mv += s_mv[rr]; }
        term = warp_sum_f64(term);
        sp = (int)__reduce_add_sync(kFull, (unsigned)sp);
        mv = (int)__reduce_add_sync(kFull, (unsigned)mv);
        if (lane == 0) {
            a.partial[b] = term;
            if (a.span) a.span[b] = sp;
            if (a.mv) a.mv[b] = mv;
        }
    }
}

__global__ void k_corr_exp(const double* __restrict__ W, int K, int NH, double2* expd)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= K * 12 * NH) return;
    const int k = idx % NH, row = idx / NH;
    const int p = row / 12, own = (row % 12) / 3, to = tree_alt_state(own, row % 3);
    const double wa = W[(size_t)k * 2 * K + 2 * p], wb = W[(size_t)k * 2 * K + 2 * p + 1];
    const double d = ((to & 1) - (own & 1)) * wa + ((to >> 1) - (own >> 1)) * wb;
    expd[idx] = make_double2(exp(d), exp(-d));
}

__global__ void k_corr_ab(const double* __restrict__ theta, int64_t n, double2* ab)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    // past 340, e^(-2 |theta|) nears the denormal numbers and the smaller factor loses its
    // bits: NaN sends the sample's rows to the logarithms
    const double x = fabs(theta[i]), e = x > 340.0 ? NAN : exp(-2.0 * x), big = 1.0 / (1.0 + e), small = e * big;
    ab[i] = theta[i] >= 0.0 ? make_double2(big, small) : make_double2(small, big);
}

}  // namespace

int launch_corr_exp(const double* W, int K, int n_hidden, double2* expd, cudaStream_t st)
{
    const int n = K * 12 * n_hidden;
    if (n == 0) return 0;
    k_corr_exp<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(W, K, n_hidden, expd);
    return 1;
}

int launch_corr_ab(const double* theta, int64_t n, double2* ab, cudaStream_t st)
{
    if (n == 0) return 0;
    k_corr_ab<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(theta, n, ab);
    return 1;
}

int launch_tree_close(const TreeClose& a, cudaStream_t st)
{
    k_tree_close<<<(unsigned)(a.nb * a.an.K), 64, (size_t)2 * a.an.D * 8, st>>>(a);
    return 1;
}

int launch_tree_rows64(const TreeRows64& a, int64_t max_chunks, cudaStream_t st)
{
    if (max_chunks == 0) return 0;
    k_tree_rows64<<<(unsigned)max_chunks, 256, 0, st>>>(a);
    return 1;
}

// Strided reads of a few words and the roots' rows: kernels in place of
// two-dimensional copies, whose calls cost 17 us of host time each against 4 us.
__global__ void k_tree_head(const int64_t* __restrict__ off, int stride, int n, const int64_t* __restrict__ last,
                            int64_t* __restrict__ out)
{
    for (int i = threadIdx.x; i <= n; i += blockDim.x) out[i] = i < n ? off[(int64_t)i * stride] : *last;
}

__global__ void __launch_bounds__(256) k_tree_roots(const double* __restrict__ h, const int* __restrict__ x, int src_rows,
                                                    int64_t n, int K, int D, double* __restrict__ pool,
                                                    int* __restrict__ pool_e)
{
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = q / D, s = row / K;
        const int c = (int)(q - row * D);
        const int64_t from = s * src_rows + (row - s * K);
        pool[q] = h[from * D + c];
        if (c == 0) pool_e[row] = x[from];
    }
}

int launch_tree_head(const int64_t* off, int stride, int n, const int64_t* last, int64_t* out, cudaStream_t st)
{
    k_tree_head<<<1, 128, 0, st>>>(off, stride, n, last, out);
    return 1;
}

int launch_tree_roots(const double* h, const int* x, int src_rows, int nb, int K, int D, double* pool, int* pool_e,
                      cudaStream_t st)
{
    const int64_t n = (int64_t)nb * K * D;
    k_tree_roots<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, st>>>(h, x, src_rows, n, K, D, pool, pool_e);
    return 1;
}

}  // namespace nqs
