// nqs_graph.cu -- the mixed (tensor-core) form of the graph-ordered ansatz.
//
// psi_TN(m) follows Eq. (bdg-rnn-update) with the linear readout and without
// the tensor term: h_i(m) = sum_{e in in(i)} M_e^{s_i(m)} h_{j(e)}(m), with
// h_{-1} = e_0 and psi_TN(m) = (h_{K-1}(m))_0. The rows of a sample share the
// nodes of their prefix tree (nqs_tree.cu, every row continued to vertex K-1);
// h_j(n) of the roots comes from the FP64 environment pass.
//
// One launch per vertex t advances every node of level t of a sample batch. The
// nodes are grouped by their local state there, so a 128-node tile multiplies
// one matrix per in-edge: per in-edge with a vertex source the nodes' source
// states (split into FP16 hi + lo, gathered from the pool of states, each node
// finding the ancestor that lived at the source vertex) times the split image
// of M_e^sigma (hi*hi + lo*hi + hi*lo, FP32 accumulation in tensor memory, one
// accumulator of D columns per edge). Thread r, which owns tensor-memory lane
// r, adds its node's accumulators, each scaled by the power of two of its
// source, renormalises the sum to a maximum in [0.5, 1) (the per-site log-scale
// of the mixed form) and writes it back split. Every node's arithmetic is its
// own, whatever tile it is in.
//
// A tile's chain (items, gather, MMA, read-back, store) is all latency, so one
// block per SM runs its parts in warps of their own: four warps copy source
// states into a ring of slots, an in-edge of a tile each; two warps make finished
// slots visible to the tensor cores; one thread issues the MMAs of each slot into
// one of four accumulators; four groups of four warps drain every fourth tile, a
// node per thread. H18 (D = 32, 16 384 samples): 97 ms. With the proxy fence in the
// copying warps (it drains their copies) and three groups 111 ms, with it in the
// MMA thread 123 ms. Three blocks per SM that each ran the chain in step took
// 170 ms (1.1 instructions per cycle, 2.2 TB/s); running 128 rows of one sample
// through all their vertices, states in shared memory, all four local states'
// products per edge and no sharing between rows, 417 ms. What is left is the drain
// groups' instructions and the gathers' latency: without any gather, power or
// store the kernel's chain alone takes about half of it.
//
// The ratio psi(m)/psi(n) = psi_TN(m)/psi_TN(n) f(m)/f(n) is formed in FP64
// from the FP32 result, with the correlator ratio of Eq. (RBM) (2cosh, or the
// cos form) as a product over hidden units of cosh(theta + d)/cosh(theta) =
// 1 + (cosh d - 1) + tanh(theta) sinh d (cos: 1 + (cos d - 1) - tan(theta)
// sin d) in FP32, carried as P - 1 (the even and the odd units' products apart).
// Per chunk of rows the terms H_nm psi(m)/psi(n) and their magnitudes are
// summed in a fixed order.
#include "nqs_tree.cuh"
#include "nqs_tc.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace nqs {

namespace {

constexpr int kGtRows = 128;
// groups of four warps that drain accumulators (a thread holds a row of D values)
constexpr int gt_groups(int D) { return D <= 32 ? 4 : 2; }
constexpr int kGtFence = 2;               // warps that pass the slots on to the MMAs
constexpr int gt_threads(int D) { return (4 + 4 * gt_groups(D) + 1 + kGtFence) * 32; }
// slots of the ring of source states; more take shared memory from the L1 that the
// item lists and shared ancestors hit (twelve: 102 ms where six take 97)
constexpr int kGtRing = 6;

// 2^d for d <= 0 in FP32 (0 below the normal range)
__device__ __forceinline__ float pow2_neg(int d)
{
    return d >= -126 ? __int_as_float((127 + d) << 23) : 0.f;
}

// cos d - 1 and sin d for |d| <= 1 from their Taylor series in z = d^2 (the
// first omitted terms are below 2^-28 of the sums)
__device__ __forceinline__ void cos_sin_small(float d, float& c1, float& sn)
{
    const float z = d * d;
    c1 = -z * fmaf(z, fmaf(z, fmaf(z, fmaf(z, 1.f / 3628800.f, -1.f / 40320.f), 1.f / 720.f), -1.f / 24.f), 0.5f);
    sn = fmaf(d * z, fmaf(z, fmaf(z, fmaf(z, fmaf(z, -1.f / 39916800.f, 1.f / 362880.f), -1.f / 5040.f),
                                 1.f / 120.f), -1.f / 6.f), d);
}

// Split images of the roots' states h_j(n) into the pool's first rows (FP64 ->
// FP32 -> FP16 hi + lo, [hi D | lo D]), their powers of two, and tanh theta_k(n)
// (cos form: tan theta_k(n)) in FP32, [np] per sample, zero-padded.
__global__ void k_tree_graph_prep(const double* __restrict__ Hst, const int* __restrict__ Hexp,
                                  const double* __restrict__ theta, int64_t s0, int64_t nb, int K, int D, int NH,
                                  int NP, int corr, unsigned char* __restrict__ pool, int* __restrict__ pool_e,
                                  float* __restrict__ tts)
{
    const int64_t n1 = nb * K * D, n2 = nb * NP;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n1 + n2;
         q += (int64_t)gridDim.x * blockDim.x) {
        if (q < n1) {
            const int64_t si = q / D;                  // (sample, vertex)
            const int c = (int)(q - si * D);
            const float v = (float)Hst[s0 * K * D + q];
            const __half hv = __float2half_rn(v);
            __half* row = (__half*)(pool + si * 4 * D);
            row[c] = hv;
            row[D + c] = __float2half_rn(v - __half2float(hv));
            if (c == 0) pool_e[si] = Hexp[s0 * K + si];
        } else {
            const int64_t t = q - n1, s = t / NP;
            const int k = (int)(t - s * NP);
            float x = 0.f;
            if (k < NH) {
                const double th = theta[(s0 + s) * NH + k];
                x = (float)(corr == 1 ? tan(th) : tanh(th));
            }
            tts[t] = x;
        }
    }
}

__device__ __forceinline__ void gt_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(tc::smem_addr(bar)) : "memory");
}

// wait with a limit; false once any role of the block has given up
__device__ __forceinline__ bool gt_wait(uint64_t* bar, uint32_t parity, volatile int* bad)
{
    for (int n = 0; n < 1024; ++n) {
        if (tc::mbar_wait(bar, parity, 1u << 14)) return true;
        if (*bad) return false;
    }
    *bad = 1;
    return false;
}

// 32 bytes to global memory (32-byte aligned)
__device__ __forceinline__ void st_32(void* p, const uint32_t* v)
{
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 :: "l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

// Vertex t of the nodes of level t (see the file header). Every wait gives up
// after a while; then all roles leave, what is in flight is waited for (bounded)
// and the tensor memory is freed.
template <int D>
__global__ void __launch_bounds__(gt_threads(D), 1) k_tree_graph_tc(TreeGraphTc a, int t, int deg, uint32_t at, uint32_t nl,
                                                                 TreeGroups gr, int n_slots)
{
    constexpr int NG = gt_groups(D);
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ uint32_t tmem_slot;
    // ring slot written / passed on / read by its MMAs; accumulator complete / read; images landed
    __shared__ __align__(8) uint64_t b_full[kGtRing], b_ready[kGtRing], b_used[kGtRing];
    __shared__ __align__(8) uint64_t b_acc[NG], b_free[NG], b_mat;
    __shared__ volatile int s_bad;
    constexpr int MD = 128 / D < kGtMaxDeg ? 128 / D : kGtMaxDeg;     // largest in-degree (see graph_tc_fits)
    __shared__ int t_e[MD];                       // edges with a vertex source, then the e_0 ones
    constexpr uint32_t kSlot = kGtRows * D * 4;   // hi then lo, 128 x D FP16 each
    constexpr uint32_t kLo = kGtRows * D * 2;
    constexpr uint32_t kMat = 2 * D * D;          // one half of one matrix image
    constexpr uint32_t kAcc = 128;                // columns of a tile's accumulators
    const int K = a.an.K;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kMmaWarp = 4 + 4 * NG;
    unsigned char* const Bs = smraw + (size_t)n_slots * kSlot;
    if (warp == kMmaWarp) { tc::tmem_alloc(&tmem_slot, 512); tc::tmem_relinquish(); }
    if (tid == 0) {
        for (int s = 0; s < kGtRing; ++s) { tc::mbar_init(&b_full[s], 128); tc::mbar_init(&b_ready[s], 1); tc::mbar_init(&b_used[s], 1); }
        for (int s = 0; s < NG; ++s) { tc::mbar_init(&b_acc[s], 1); tc::mbar_init(&b_free[s], 4); }
        tc::mbar_init(&b_mat, 1);
        s_bad = 0;
    }
    const int e0 = a.an.pred_ptr[t];
    int nv = 0;                                   // in-edges with a vertex source
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
    const int nt = gr.tile[4];
    const int tile0 = (int)((int64_t)nt * blockIdx.x / gridDim.x);
    const int tile1 = (int)((int64_t)nt * (blockIdx.x + 1) / gridDim.x);
    auto place = [&](int tile, int& sg, uint32_t& i0, int& n) {
        sg = 0;
        while (sg < 3 && tile >= gr.tile[sg + 1]) ++sg;
        const uint32_t b0 = sg == 0 ? gr.b[0] : sg == 1 ? gr.b[1] : sg == 2 ? gr.b[2] : gr.b[3];
        const uint32_t b1 = sg == 0 ? gr.b[1] : sg == 1 ? gr.b[2] : sg == 2 ? gr.b[3] : gr.b[4];
        const int f = sg == 0 ? 0 : sg == 1 ? gr.tile[1] : sg == 2 ? gr.tile[2] : gr.tile[3];
        i0 = b0 + (uint32_t)(tile - f) * kGtRows;
        n = (int)min(b1 - i0, (uint32_t)kGtRows);
    };
    // row r of a tile: its result row and the sources of its in-edges (rows past
    // the tile's repeat the first)
    auto fetch = [&](int tile, int r, uint32_t& out, uint32_t* src) {
        int sg, n;
        uint32_t i0;
        place(tile, sg, i0, n);
        const uint32_t* it = a.items + at + i0 + (r < n ? r : 0);
        out = __ldg(it);
        #pragma unroll
        for (int k = 0; k < MD; ++k)
            if (k < nv) src[k] = __ldg(it + (size_t)(k + 1) * nl);
    };

    if (warp < 4) {
        // the sources' states, an in-edge of a tile per slot: 16-byte pieces, eight
        // nodes x four pieces per warp so that shared memory is written in whole core
        // matrices and global memory read in 64-byte runs; the copies announce themselves
        uint32_t nxt[MD] = {}, out;
        uint32_t slot = 0, round = 0;
        bool ok = true;
        if (tile0 < tile1) fetch(tile0, 32 * warp + lane, out, nxt);
        for (int tile = tile0; ok && tile < tile1 && nv > 0; ++tile) {
            uint32_t cur[MD];
            #pragma unroll
            for (int k = 0; k < MD; ++k) cur[k] = nxt[k];
            if (tile + 1 < tile1) fetch(tile + 1, 32 * warp + lane, out, nxt);
            #pragma unroll
            for (int k = 0; k < MD; ++k) {
                if (k >= nv) break;
                if (round > 0) ok = __all_sync(kFull, ok && gt_wait(&b_used[slot], (round - 1) & 1, &s_bad));
                if (!ok) break;
                unsigned char* to = smraw + (size_t)slot * kSlot;
                #pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int rr = 8 * j + (lane & 7);
                    const unsigned char* row = a.pool + (size_t)__shfl_sync(kFull, cur[k], rr) * 4 * D;
                    #pragma unroll
                    for (int p = 0; p < D / 16; ++p) {
                        const int pc = 4 * p + (lane >> 3);
                        const bool lo = pc >= D / 8;
                        const int c8 = lo ? pc - D / 8 : pc;
                        tc::cp_async16(to + (lo ? kLo : 0) + tc::op_offset(32 * warp + rr, 8 * c8, D), row + 16 * pc);
                    }
                }
                tc::cp_async_arrive(&b_full[slot]);
                if (++slot == (uint32_t)n_slots) { slot = 0; ++round; }
            }
        }
        tc::cp_async_commit();
        tc::cp_async_wait<0>();
    } else if (warp < kMmaWarp) {
        // group gq drains every NG-th tile, a node per thread
        const int gq = (warp - 4) >> 2, r = 32 * (warp & 3) + lane;
        const uint32_t tlane = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + gq * kAcc;
        uint32_t src[MD] = {}, out = 0;           // of the group's next tile, and its sources' powers of two
        int es[MD] = {};
        auto powers = [&]() {
            #pragma unroll
            for (int k = 0; k < MD; ++k)
                if (k < nv) es[k] = a.pool_e[src[k]];
        };
        if (tile0 + gq < tile1) { fetch(tile0 + gq, r, out, src); powers(); }
        uint32_t use = 0;
        for (int tile = tile0 + gq; tile < tile1; tile += NG, ++use) {
            int sg, n;
            uint32_t i0;
            place(tile, sg, i0, n);
            const uint32_t dst = out;
            const bool more = tile + NG < tile1;
            int se[MD];
            int eref = nv < deg ? 0 : -(1 << 30);     // an e_0 source has power 0
            #pragma unroll
            for (int k = 0; k < MD; ++k)
                if (k < nv) { se[k] = es[k] + __ldg(a.bexp + t_e[k] * 4 + sg); eref = max(eref, se[k]); }
            if (more) fetch(tile + NG, r, out, src);
            if (nv > 0) {
                if (!__all_sync(kFull, gt_wait(&b_acc[gq], use & 1, &s_bad))) break;
                tc::fence_after_sync();
            }
            float y[D];
            #pragma unroll
            for (int c = 0; c < D; ++c) y[c] = 0.f;
            constexpr int CW = 16;                // columns read at a time
            #pragma unroll
            for (int k = 0; k < MD; ++k) {
                if (k < nv) {
                    const float f = pow2_neg(se[k] - eref);
                    #pragma unroll
                    for (int c0 = 0; c0 < D; c0 += CW) {
                        uint32_t v[CW];
                        #pragma unroll
                        for (int c1 = 0; c1 < CW; c1 += 16) tc::tmem_ld16(tlane + (uint32_t)(k * D + c0 + c1), v + c1);
                        tc::tmem_wait_ld();
                        #pragma unroll
                        for (int c = 0; c < CW; ++c) y[c0 + c] = fmaf(__uint_as_float(v[c]), f, y[c0 + c]);
                    }
                }
            }
            if (nv > 0) {
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) gt_arrive(&b_free[gq]);
            }
            if (more) powers();
            for (int k = nv; k < deg; ++k) {
                // M e_0: column 0 of the matrix
                const float f = pow2_neg(-eref);
                const float* col = a.col0 + ((size_t)t_e[k] * 4 + sg) * D;
                #pragma unroll
                for (int c = 0; c < D; ++c) y[c] = fmaf(__ldg(col + c), f, y[c]);
            }
            float mx = 0.f;
            #pragma unroll
            for (int c = 0; c < D; ++c) mx = fmaxf(mx, fabsf(y[c]));
            if (r < n) {
                int ge = 0;
                if (mx > 0.f) frexpf(mx, &ge);
                const int ex = eref + ge;
                // 2^-ge, in two factors where one would not be a normal number (the first
                // is exact, or the result is zero either way)
                const bool one = ge >= -126 && ge <= 126;
                const float f0 = __int_as_float((127 + (one ? -ge : -ge / 2)) << 23);
                #pragma unroll
                for (int c = 0; c < D; ++c) y[c] *= f0;
                if (!one) {
                    const float f1 = __int_as_float((127 - ge + ge / 2) << 23);
                    #pragma unroll
                    for (int c = 0; c < D; ++c) y[c] *= f1;
                }
                if (t == K - 1) {
                    a.mant[dst] = y[0];
                    a.mexp[dst] = ex;
                } else {
                    unsigned char* row = a.pool + (size_t)dst * 4 * D;
                    #pragma unroll
                    for (int c0 = 0; c0 < D; c0 += 16) {
                        __align__(16) __half2 hi[8], lo[8];
                        #pragma unroll
                        for (int q = 0; q < 8; ++q)
                            tc::split_half2(y[c0 + 2 * q], y[c0 + 2 * q + 1], hi[q], lo[q]);
                        st_32(row + 2 * c0, (const uint32_t*)hi);
                        st_32(row + 2 * D + 2 * c0, (const uint32_t*)lo);
                    }
                    a.pool_e[dst] = ex;
                }
            }
        }
    } else if (warp > kMmaWarp) {
        // the copies of every kGtFence-th slot, made visible to the MMAs: the proxy
        // fence takes a few hundred cycles, which neither the MMA thread nor the
        // copying warps (it drains all that they have in flight) should wait for
        const uint32_t total = nv > 0 && tile0 < tile1 ? (uint32_t)(tile1 - tile0) * nv : 0;
        uint32_t slot = warp - kMmaWarp - 1, round = 0;
        for (uint32_t i = slot; lane == 0 && i < total; i += kGtFence) {
            if (!gt_wait(&b_full[slot], round & 1, &s_bad)) break;
            tc::fence_proxy_async();
            gt_arrive(&b_ready[slot]);
            slot += kGtFence;
            if (slot >= (uint32_t)n_slots) { slot -= n_slots; ++round; }
        }
    } else if (lane == 0 && nv > 0) {
        const uint32_t idesc = tc::idesc_f16(kGtRows, D);
        const uint64_t d0 = tc::desc(0, 128, 16 * D);
        uint32_t slot = 0, round = 0, n_mat = 0, last = 0, last_p = 0;
        int held = -1;                            // local state whose images are in Bs
        bool ok = true, any = false;
        uint32_t it = 0;
        for (int tile = tile0; ok && tile < tile1; ++tile, ++it) {
            int sg, n;
            uint32_t i0;
            place(tile, sg, i0, n);
            if (sg != held) {
                if (any) ok = gt_wait(&b_used[last], last_p, &s_bad);     // the images' last readers
                if (!ok) break;
                tc::mbar_expect_tx(&b_mat, (uint32_t)nv * 2 * kMat);
                for (int k = 0; k < nv; ++k) {
                    const unsigned char* src = a.bimg + (size_t)t_e[k] * 8 * kMat + (size_t)sg * kMat;
                    tc::bulk_g2s(Bs + (size_t)k * 2 * kMat, src, kMat, &b_mat);
                    tc::bulk_g2s(Bs + (size_t)k * 2 * kMat + kMat, src + 4 * kMat, kMat, &b_mat);
                }
                ok = tc::mbar_wait(&b_mat, n_mat & 1, 1u << 24);          // not cut short: a copy in flight
                if (!ok) { s_bad = 1; break; }
                ++n_mat;
                held = sg;
            }
            const uint32_t buf = it % NG;
            if (it >= NG) ok = gt_wait(&b_free[buf], (it / NG - 1) & 1, &s_bad);
            for (int k = 0; ok && k < nv; ++k) {
                ok = gt_wait(&b_ready[slot], round & 1, &s_bad);
                if (!ok) break;
                tc::fence_after_sync();
                const uint64_t dA = d0 + (tc::smem_addr(smraw + (size_t)slot * kSlot) >> 4);
                const uint64_t dB = d0 + (tc::smem_addr(Bs + (size_t)k * 2 * kMat) >> 4);
                #pragma unroll
                for (int term = 0; term < 3; ++term)
                    #pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        const uint64_t ao = term == 1 ? (kLo >> 4) : 0;
                        const uint64_t bo = term == 2 ? (kMat >> 4) : 0;
                        tc::mma_f16(tmem + buf * kAcc + (uint32_t)(k * D), dA + ao + 16 * ks, dB + bo + 16 * ks, idesc,
                                    (term | ks) ? 1u : 0u);
                    }
                tc::mma_commit(&b_used[slot]);
                if (k == nv - 1) tc::mma_commit(&b_acc[buf]);
                any = true;
                last = slot;
                last_p = round & 1;
                if (++slot == (uint32_t)n_slots) { slot = 0; ++round; }
            }
        }
        if (any) tc::mbar_wait(&b_used[last], last_p, 1u << 24);          // nothing in flight at the end
    }
    __syncwarp();
    tc::fence_before_sync();
    __syncthreads();
    if (s_bad && tid == 0) report(a.err, 5, 6, (long long)blockIdx.x);
    if (warp == kMmaWarp) tc::tmem_dealloc(tmem, 512);
}

// Terms of the rows, one thread per row: psi_TN(m) from the row's node, the
// correlator product over the hidden units, the ratio in FP64.
__global__ void __launch_bounds__(kTreeRows) k_tree_rows_tc(TreeRowsTc a)
{
    extern __shared__ float WTs[];                // [NH][2K]
    __shared__ int64_t s_s;
    __shared__ double wsum[4], wabs[4];
    __shared__ int wspan[4], wmv[4];
    const TreeArgs& t = a.t;
    const int K = a.an.K, NH = a.an.n_hidden, NP = a.np;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // correlator weights as [unit][spin orbital]: the lanes of a warp read one
    // unit's weights of their rows' different flips
    for (int q = tid; q < 2 * K * NH; q += kTreeRows) {
        const int k = q / (2 * K), f = q - k * 2 * K;
        WTs[q] = a.WT[(size_t)f * NP + k];
    }
    const int64_t b0 = a.chunk_base[t.s0], b1 = a.chunk_base[t.s0 + t.nb];
    for (int64_t b = b0 + blockIdx.x; b < b1; b += gridDim.x) {
        __syncthreads();
        if (tid == 0) s_s = tree_sample(t, a.chunk_base, b);
        __syncthreads();
        const int64_t s = s_s;
        const uint64_t na = t.samples[2 * s], nb = t.samples[2 * s + 1];
        const int64_t r0 = (b - a.chunk_base[s]) * kTreeRows, rb = t.row_base[s] - t.row_base[t.s0];
        const int64_t first = a.draws ? t.det_cnt[s] : 0;
        const int64_t left = (a.draws ? t.draw_cnt[s] : t.det_cnt[s]) - r0;
        double term = 0.0, ab = 0.0;
        int sp = 0, mv = 0;
        if (tid < left) {
            const int64_t row = a.perm[rb + first + r0 + tid], g = rb + row;
            const TreeWord w = tree_unpack(t.word[g]);
            const uint32_t node = t.rnode[g];
            uint64_t ma, mb;
            tree_det(w, na, nb, ma, mb);
            // the flipped spin orbitals (at most four, +1 where m occupies them)
            int fi[4];
            float fs[4];
            uint64_t da = na ^ ma, db = nb ^ mb;
            #pragma unroll
            for (int q = 0; q < 4; ++q) {
                fi[q] = 0;
                fs[q] = 0.f;
                if (da) {
                    const int p = __ffsll((long long)da) - 1;
                    da &= da - 1;
                    fi[q] = 2 * p; fs[q] = ((ma >> p) & 1ull) ? 1.f : -1.f;
                } else if (db) {
                    const int p = __ffsll((long long)db) - 1;
                    db &= db - 1;
                    fi[q] = 2 * p + 1; fs[q] = ((mb >> p) & 1ull) ? 1.f : -1.f;
                }
            }
            const float* tts = a.tts + (size_t)(s - t.s0) * NP;
            const bool cos_kind = a.an.corr == 1;
            float X2[2] = {0.f, 0.f};             // prod (1 + x_k) - 1 of the even and the odd units
            auto unit = [&](int k, float X) {
                float d = 0.f;
                #pragma unroll
                for (int q = 0; q < 4; ++q) d = fmaf(fs[q], WTs[k * 2 * K + fi[q]], d);
                float x;
                if (!cos_kind) {
                    float ch1, sh;
                    if (fabsf(d) <= 1.f) {
                        cosh_sinh_small(d, ch1, sh);
                    } else {
                        const float em = expm1f(d), inv = 1.f / (1.f + em);
                        ch1 = 0.5f * em * em * inv;
                        sh = 0.5f * em * (1.f + inv);
                    }
                    x = fmaf(__ldg(tts + k), sh, ch1);
                } else {
                    float c1, sn;
                    if (fabsf(d) <= 1.f) {
                        cos_sin_small(d, c1, sn);
                    } else {
                        const float hs = sinf(0.5f * d);
                        c1 = -2.f * hs * hs;
                        sn = sinf(d);
                    }
                    x = fmaf(-__ldg(tts + k), sn, c1);
                }
                return fmaf(X, x, X + x);
            };
            for (int k = 0; k < NH; k += 2) {
                X2[0] = unit(k, X2[0]);
                if (k + 1 < NH) X2[1] = unit(k + 1, X2[1]);
            }
            const float X = fmaf(X2[0], X2[1], X2[0] + X2[1]);
            const double rpsi = 1.0 / a.psi_mant[s];
            const double tn = scale_pow2((double)a.mant[node] * rpsi, a.mexp[node] - a.psi_exp[s]);
            term = tree_coef(t, s, row) * tn * (1.0 + (double)X);
            ab = fabs(term);
            const int p = w.x[0] / 3;
            sp = K - p;
            mv = graph_matvecs(a.an, p);
        }
        for (int o = 16; o; o >>= 1) {
            term += __shfl_xor_sync(kFull, term, o);
            ab += __shfl_xor_sync(kFull, ab, o);
        }
        sp = (int)__reduce_add_sync(kFull, (unsigned)sp);
        mv = (int)__reduce_add_sync(kFull, (unsigned)mv);
        if (lane == 0) { wsum[warp] = term; wabs[warp] = ab; wspan[warp] = sp; wmv[warp] = mv; }
        __syncthreads();
        if (tid == 0) {
            a.partial[b] = ((wsum[0] + wsum[1]) + wsum[2]) + wsum[3];
            if (a.partial_abs) a.partial_abs[b] = ((wabs[0] + wabs[1]) + wabs[2]) + wabs[3];
            if (a.span) a.span[b] = wspan[0] + wspan[1] + wspan[2] + wspan[3];
            if (a.mv) a.mv[b] = wmv[0] + wmv[1] + wmv[2] + wmv[3];
        }
    }
}

}  // namespace

int launch_tree_graph_prep(const double* Hst, const int* Hexp, const double* theta, int64_t s0, int nb, int K, int D,
                           int NH, int NP, int corr, unsigned char* pool, int* pool_e, float* tts, cudaStream_t st)
{
    const int64_t n = (int64_t)nb * K * D + (int64_t)nb * NP;
    const int64_t grid = std::min<int64_t>((n + 255) / 256, 2048);
    k_tree_graph_prep<<<(unsigned)grid, 256, 0, st>>>(Hst, Hexp, theta, s0, nb, K, D, NH, NP, corr, pool, pool_e, tts);
    return 1;
}

int launch_tree_graph_tc(const TreeGraphTc& a, int t, int deg, const TreeLevels& lv, const int64_t* bounds, int n_sm,
                         cudaStream_t st)
{
    const int D = a.an.D;
    const TreeGroups g = tree_groups(t, bounds, kGtRows);
    if (g.tile[4] == 0) return 0;
    // one block per SM; its ring takes the shared memory that the images leave
    const size_t slot = (size_t)kGtRows * D * 4, images = (size_t)deg * 4 * D * D;
    const int n_slots = (int)std::min<size_t>(kGtRing, ((size_t)220 * 1024 - images) / slot);
    const size_t smem = n_slots * slot + images;
    const unsigned grid = (unsigned)std::min<int>(g.tile[4], n_sm);
    auto launch = [&](void (*kernel)(TreeGraphTc, int, int, uint32_t, uint32_t, TreeGroups, int)) {
        allow_max_smem(kernel);
        kernel<<<grid, gt_threads(D), smem, st>>>(a, t, deg, lv.at[t], lv.n[t], g, n_slots);
    };
    if (D == 16) launch(k_tree_graph_tc<16>);
    else if (D == 32) launch(k_tree_graph_tc<32>);
    else launch(k_tree_graph_tc<64>);
    return 1;
}

int launch_tree_rows_tc(const TreeRowsTc& a, int64_t max_chunks, int n_sm, cudaStream_t st)
{
    if (max_chunks == 0) return 0;
    allow_max_smem(k_tree_rows_tc);
    const unsigned grid = (unsigned)std::min<int64_t>(max_chunks, (int64_t)16 * n_sm);
    k_tree_rows_tc<<<grid, kTreeRows, (size_t)2 * a.an.K * a.an.n_hidden * 4, st>>>(a);
    return 1;
}

// Which graphs the mixed form takes is part of the interface. Two of its limits, 16
// live states and the bytes below (128 rows of every live state beside the matrix
// images), are those of tiles that kept the states in shared memory; the steps over the
// prefix trees keep none there and would need only the limit on D x in-degree.
static size_t graph_tiles_smem(int D, int K, int n_slots, int max_deg, int n_hidden, int nbuf)
{
    const size_t np = (size_t)((n_hidden + 3) & ~3);
    return (size_t)n_slots * kGtRows * D * 4 + (size_t)nbuf * max_deg * 16 * D * D + (size_t)K * 4 * D +
           (((size_t)2 * K * n_hidden + 3) & ~(size_t)3) * 4 + np * 4;
}

bool graph_tc_fits(const int* ptr, const int* idx, int K, int D, int n_hidden, const char** why)
{
    *why = nullptr;
    if (D != 16 && D != 32 && D != 64) { *why = "bond dimension must be 16, 32 or 64"; return false; }
    int max_deg = 0;
    for (int i = 0; i < K; ++i) max_deg = std::max(max_deg, ptr[i + 1] - ptr[i]);
    if (max_deg > kGtMaxDeg || max_deg * 4 * D > 512) {
        *why = "in-degree x 4 x bond dimension must fit 512 tensor-memory columns";
        return false;
    }
    // states alive at once, by greedy interval colouring
    std::vector<int> last(K, -1), busy;
    for (int i = 0; i < K; ++i)
        for (int e = ptr[i]; e < ptr[i + 1]; ++e)
            if (idx[e] >= 0) last[idx[e]] = std::max(last[idx[e]], i);
    for (int i = 0; i < K; ++i) {
        for (size_t s = 0; s < busy.size(); ++s)
            if (busy[s] >= 0 && last[busy[s]] <= i) busy[s] = -1;
        if (last[i] <= i) continue;
        size_t s = 0;
        while (s < busy.size() && busy[s] >= 0) ++s;
        if (s == busy.size()) busy.push_back(-1);
        busy[s] = i;
    }
    const int n_slots = std::max<int>(1, (int)busy.size());
    if (n_slots > kGtMaxSlots) { *why = "more than 16 vertex states live at once"; return false; }
    int dev = 0, mx = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&mx, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const size_t margin = 24576;
    if (mx > 0 && graph_tiles_smem(D, K, n_slots, max_deg, n_hidden, 1) + margin > (size_t)mx) {
        *why = "128 rows of the live vertex states and the matrix images exceed a block's shared memory";
        return false;
    }
    return true;
}

}  // namespace nqs
