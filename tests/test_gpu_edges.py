"""Kernels at the edges of their tiles and ranges, against plain float64
references. Tolerances are a multiple of 2^-53 times the sum of the magnitudes
added (the bound of a sum taken in any order)."""
import numpy as np
import pytest

from paper_2507_19276_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2507_19276_gb300 import nqs  # noqa: E402

U = 2.0 ** -53


@pytest.fixture(scope="module")
def ctx():
    c = nqs.Context(0)
    yield c
    c.close()


def _occ(s, K):
    b = (np.asarray(s, np.uint64)[:, None, :] >> np.arange(K, dtype=np.uint64)[None, :, None]) & np.uint64(1)
    return b.reshape(len(s), 2 * K).astype(np.float64)


@pytest.mark.parametrize("nh,ns", [(1, 1), (3, 31), (32, 33), (33, 4097 // 16), (36, 4900)])
def test_correlator_gradient_chunks(ctx, nh, ns):
    """Chunks of samples x 32 hidden units: remainders on both sides, a last
    chunked pass (grad_chunk) whose chunk count differs from the full passes'."""
    s = W.tiny_system(K=8, na=4, nb=4, D=3, n_hidden=nh, seed=nh + ns, n_samples=ns)
    u = np.random.default_rng(ns).normal(size=len(s.samples))
    n = _occ(s.samples, s.K)
    t = np.tanh(s.rbm_b + n @ s.rbm_W.T)
    ref_W, ref_b = (u[:, None] * t).T @ n, (u[:, None] * t).sum(0)
    size = np.abs(u)[:, None] * np.abs(t)
    ctx.set_system(s)
    for chunk in (0, max(1, ns // 2 + 1)):
        ctx.set_precision(nqs.NQS_PREC_FP64, grad_chunk=chunk)
        _, gW, gb = ctx.grad_log_psi_vjp(s.samples, u)
        tol = (len(u) + 64) * U
        assert np.all(np.abs(gb - ref_b) <= tol * size.sum(0) + 1e-300)
        assert np.all(np.abs(gW - ref_W) <= tol * size.sum(0)[:, None] + 1e-300)
    ctx.set_precision(nqs.NQS_PREC_FP64)


@pytest.mark.parametrize("graph,D", [(False, 1), (False, 16), (False, 33), (False, 80), (False, 192), (True, 16), (True, 33)])
def test_ansatz_forms_from_host_and_device(ctx, graph, D):
    """The device-made parameter forms (tiles of 32, one or several reduction
    chunks) serve every precision form; host and device parameters agree bitwise."""
    s = W.tiny_system(K=6, na=3, nb=3, D=D, n_hidden=5, seed=D, graph=graph, n_samples=40)
    ctx.set_system(s)
    got = {}
    for where in ("host", "device"):
        args = [s.tensors, s.rbm_W, s.rbm_b]
        if where == "device":
            args = [torch.from_numpy(x).cuda() for x in args]
        ctx.set_ansatz(args[0], s.pred_ptr, s.pred_idx, args[1], args[2])
        for prec in (nqs.NQS_PREC_FP64, nqs.NQS_PREC_MIXED):
            if graph and prec == nqs.NQS_PREC_MIXED and D != 16:
                continue
            ctx.set_precision(prec)
            got[where, prec] = ctx.local_energy(s.samples, s.counts, 0.0, 0, 1)[0]
    for prec in (nqs.NQS_PREC_FP64, nqs.NQS_PREC_MIXED):
        if ("host", prec) in got:
            assert np.array_equal(got["host", prec], got["device", prec])
            ref = got["host", nqs.NQS_PREC_FP64]
            assert np.all(np.abs(got["host", prec] - ref) <= 1e-5 * np.maximum(np.abs(ref), np.abs(ref).max()))
    ctx.set_precision(nqs.NQS_PREC_FP64)


@pytest.mark.parametrize("n", [1, 31, 33, 4097, 140000])
@pytest.mark.parametrize("graph", [False, True])
def test_sampler_sizes(ctx, n, graph):
    """One draw, part warps, several blocks, and the descent by levels (above
    2^17 draws): determinants and counts bit-equal to the oracle's."""
    from oracle import oracle as O
    s = W.with_readout(W.tiny_system(K=8, na=4, nb=3, D=5, n_hidden=3, seed=n % 97, graph=graph, n_samples=4), seed=2)
    if graph and n in (33, 4097):
        s = W.with_tensor_term(s, seed=1)        # the descent by levels at small sizes
    ctx.set_system(s)
    dets, counts = ctx.sample(n, 11 + n)
    ref, ref_c, _ = O.sample(O.Problem(s), n, 11 + n)
    assert counts.sum() == n
    assert np.array_equal(dets, ref) and np.array_equal(counts, ref_c)


def _dag(seed, K, D, n_hidden=4, n_samples=None, eps=0.0, n_draws=0):
    """A graph system whose edges skip vertices: e_0 sources in the middle, a
    vertex nothing reads, repeated sources."""
    import dataclasses
    rng = np.random.default_rng(seed)
    s = W.tiny_system(K=K, na=K // 2, nb=(K + 1) // 2, D=D, n_hidden=n_hidden, seed=seed, eps=eps, n_draws=n_draws,
                      n_samples=n_samples)
    ptr, idx = [0], []
    for i in range(K):
        src = [-1] if i == 0 else sorted(rng.integers(-1, i, size=rng.integers(1, 4)).tolist())
        if i == K - 1:
            src = sorted(set(src + [i - 1, max(0, i - 3)]))
        idx += src
        ptr.append(len(idx))
    T = rng.normal(size=(len(idx), 4, D, D)) / np.sqrt(D) + 0.3 * np.eye(D)
    return dataclasses.replace(s, pred_ptr=np.array(ptr, np.int32), pred_idx=np.array(idx, np.int32),
                               tensors=np.ascontiguousarray(T))


@pytest.mark.parametrize("seed,K,D,ns,eps,draws", [
    (1, 7, 5, None, 0.0, 0), (2, 7, 33, 40, 0.05, 50), (3, 5, 1, None, 0.0, 0), (4, 9, 8, 300, 1e3, 200),
    (5, 6, 130, 7, 0.0, 0), (6, 8, 16, 1, 0.02, 7), (7, 2, 4, None, 0.0, 0)])
def test_graph_prefix_tree_fp64(ctx, seed, K, D, ns, eps, draws):
    """FP64 form of graphs over the prefix trees: tiles and remainders of every
    kind, drawn rows alone (eps above every element), against the oracle within
    the FP64 bar of the other parity tests."""
    from oracle import oracle as O
    s = _dag(seed, K, D, n_samples=ns, eps=eps, n_draws=draws)
    ctx.set_system(s)
    ctx.set_precision(nqs.NQS_PREC_FP64)
    ref = O.local_energy(O.Problem(s), cond=True)
    ok = np.isfinite(ref["e_loc"])
    e, summ = ctx.local_energy(s.samples, s.counts, s.eps, s.n_draws, s.seed)
    scale = np.maximum(np.abs(ref["e_loc"]), ref["e_abs"]) + (2.0 ** -52 / 1e-12) * ref["e_cond"]
    assert np.all(np.abs(e - ref["e_loc"])[ok] <= 1e-12 * scale[ok])
    assert summ["n_det"] == int(ref["n_det"].sum())


@pytest.mark.parametrize("K,D,ns,eps,draws,nh", [(8, 1, 70, 0.0, 0, 0), (7, 16, 1, 0.02, 9, 5), (6, 17, None, 1e3, 300, 0),
                                                 (9, 32, 33, 0.05, 64, 4), (3, 33, None, 0.0, 0, 2), (1, 4, None, 0.0, 0, 0)])
def test_normalised_chain_prefix_tree(ctx, K, D, ns, eps, draws, nh):
    """Normalised readout of chains over the prefix trees (D up to 32) and row by
    row (33): 32- and 64-node tiles, drawn rows alone, one sample; FP64 bar."""
    from oracle import oracle as O
    s = W.with_readout(W.tiny_system(K=K, na=K // 2, nb=(K + 1) // 2, D=D, n_hidden=nh, seed=K + D, eps=eps,
                                     n_draws=draws, n_samples=ns), seed=D)
    ctx.set_system(s)
    ctx.set_precision(nqs.NQS_PREC_FP64)
    ref = O.local_energy(O.Problem(s))
    e, summ = ctx.local_energy(s.samples, s.counts, s.eps, s.n_draws, s.seed)
    assert np.all(np.abs(e - ref["e_loc"]) <= 1e-12 * np.maximum(np.abs(ref["e_loc"]), ref["e_abs"]) + 1e-300)
    assert summ["n_det"] == int(ref["n_det"].sum())


@pytest.mark.parametrize("seed,K,D,ns,eps,draws", [(11, 7, 16, None, 0.0, 0), (12, 6, 32, 5, 0.05, 40), (13, 8, 16, 1, 1e3, 200),
                                                   (14, 5, 64, None, 0.02, 16)])
def test_graph_prefix_tree_mixed(ctx, seed, K, D, ns, eps, draws):
    """Mixed form of graphs over the prefix trees: 128-node tiles of every local
    state, vertices without a vertex source, drawn rows alone; mixed bar."""
    import dataclasses
    from oracle import oracle as O
    s = _dag(seed, K, D, n_samples=ns, eps=eps, n_draws=draws)
    if D == 64:                                     # one in-edge: two matrices' images do not fit (refused)
        ptr, idx, keep = [0], [], []
        for i in range(K):
            e = list(range(s.pred_ptr[i], s.pred_ptr[i + 1]))[-1:]
            keep += e
            idx += [int(s.pred_idx[x]) for x in e]
            ptr.append(len(idx))
        s = dataclasses.replace(s, pred_ptr=np.array(ptr, np.int32), pred_idx=np.array(idx, np.int32),
                                tensors=np.ascontiguousarray(s.tensors[keep]))
    ctx.set_system(s)
    ctx.set_precision(nqs.NQS_PREC_MIXED)
    ref = O.local_energy(O.Problem(s))
    e, summ = ctx.local_energy(s.samples, s.counts, s.eps, s.n_draws, s.seed)
    ctx.set_precision(nqs.NQS_PREC_FP64)
    assert np.all(np.abs(e - ref["e_loc"]) <= 1e-6 * np.maximum(np.abs(ref["e_loc"]), ref["e_abs"]))
    assert summ["n_det"] == int(ref["n_det"].sum())


def _log_psi_ref(s, dets):
    """log|psi_TN|, sign and the sum's rounding scale in extended precision."""
    T = s.tensors.astype(np.longdouble)
    occ = _occ(dets, s.K).astype(int)
    sig = occ[:, 0::2] + 2 * occ[:, 1::2]
    la, sg, cond = [], [], []
    for n in sig:
        h = np.zeros(s.D, np.longdouble)
        h[0] = 1
        a, le = h.copy(), np.longdouble(0)
        for t in range(s.K):
            h, a = T[t, n[t]] @ h, np.abs(T[t, n[t]]) @ a
            m = np.abs(h).max()
            h, a, le = h / m, a / m, le + np.log(m)
        la.append(np.log(np.abs(h[0])) + le)
        sg.append(np.sign(h[0]))
        cond.append(a[0] / np.abs(h[0]))
    return np.array(la, float), np.array(sg, int), np.array(cond, float)


@pytest.mark.parametrize("D", [16, 32, 48, 64])
@pytest.mark.parametrize("n", [512, 777, 1201])
def test_fixed_point_steps(ctx, D, n):
    """Chains on the fixed-point tensor-core steps: every width, part tiles of
    every local state, entries over many powers of two. K (D + 1) 2^-53 of the
    running absolute product bounds an FP64 chain; the steps must keep to it."""
    import dataclasses
    s = W.tiny_system(K=8, na=4, nb=4, D=D, seed=D, n_samples=n)
    rng = np.random.default_rng(D)
    T = s.tensors * np.exp2(rng.integers(-20, 8, size=(s.K, 4, D, 1)))      # rows of unlike size
    T[2, 1, :, 3] = 0.0
    s = dataclasses.replace(s, tensors=T)
    ctx.set_system(s)
    la, sg = ctx.amplitude(s.samples)
    ref, rs, cond = _log_psi_ref(s, s.samples)
    tol = s.K * (D + 1) * U * cond + 8 * U * np.abs(ref)
    ok = tol < 1e-3
    assert ok.sum() > n // 2
    assert np.all(np.abs(la - ref)[ok] <= tol[ok]) and np.array_equal(sg[ok], rs[ok])
    # environments: the gradient of one call and of the row-by-row form in chunks
    u = np.random.default_rng(n).normal(size=n)
    ctx.set_precision(nqs.NQS_PREC_FP64)
    g1 = ctx.grad_log_psi_vjp(s.samples, u)[0]
    ctx.set_precision(nqs.NQS_PREC_FP64, grad_chunk=100)
    g2 = ctx.grad_log_psi_vjp(s.samples, u)[0]
    ctx.set_precision(nqs.NQS_PREC_FP64)
    assert np.all(np.abs(g1 - g2) <= 1e-10 * np.abs(g2).max())


def test_fixed_point_steps_not_finite(ctx):
    """A NaN in a site tensor reaches every amplitude whose local state reads it."""
    import dataclasses
    s = W.tiny_system(K=8, na=4, nb=4, D=16, seed=1, n_samples=600)
    T = s.tensors.copy()
    T[5, 3, 2, 7] = np.nan
    ctx.set_system(dataclasses.replace(s, tensors=T))
    la, _ = ctx.amplitude(s.samples)
    occ = _occ(s.samples, s.K)
    hit = (occ[:, 10] + occ[:, 11]) == 2
    assert np.all(np.isnan(la[hit])) and np.all(np.isfinite(la[~hit]))


@pytest.mark.parametrize("D,ns", [(16, 301), (32, 260), (48, 130), (64, 129)])
@pytest.mark.parametrize("chain", [False, True])
def test_prefix_tree_fixed_point(ctx, D, ns, chain):
    """Levels large enough for the fixed-point tiles, chains and graphs with up to
    four in-edges and e_0 sources, part tiles; the FP64 bar."""
    from oracle import oracle as O
    s = W.tiny_system(K=8, na=4, nb=4, D=D, n_hidden=3, seed=D, n_samples=ns, eps=0.01, n_draws=20) if chain \
        else _dag(D, 8, D, n_samples=ns, eps=0.01, n_draws=20)
    ctx.set_system(s)
    ctx.set_precision(nqs.NQS_PREC_FP64)
    ref = O.local_energy(O.Problem(s), cond=True)
    e, summ = ctx.local_energy(s.samples, s.counts, s.eps, s.n_draws, s.seed)
    scale = np.maximum(np.abs(ref["e_loc"]), ref["e_abs"]) + (2.0 ** -52 / 1e-12) * ref["e_cond"]
    assert np.all(np.abs(e - ref["e_loc"]) <= 1e-12 * scale)
    assert summ["n_det"] == int(ref["n_det"].sum())


@pytest.mark.parametrize("D,ns", [(4, 300), (10, 301), (16, 129), (17, 200), (24, 128)])
def test_normalised_chain_fixed_point(ctx, D, ns):
    """The same for the normalised readout's candidate cells: one to three blocks of
    32 entries, both reduction widths."""
    from oracle import oracle as O
    s = W.with_readout(W.tiny_system(K=8, na=4, nb=4, D=D, n_hidden=2, seed=D, eps=0.01, n_draws=20, n_samples=ns), seed=D)
    ctx.set_system(s)
    ctx.set_precision(nqs.NQS_PREC_FP64)
    ref = O.local_energy(O.Problem(s))
    e, _ = ctx.local_energy(s.samples, s.counts, s.eps, s.n_draws, s.seed)
    assert np.all(np.abs(e - ref["e_loc"]) <= 1e-12 * np.maximum(np.abs(ref["e_loc"]), ref["e_abs"]))


@pytest.mark.parametrize("K,na,nb", [(2, 1, 1), (3, 1, 2), (4, 0, 2), (5, 5, 1), (9, 4, 2), (13, 6, 7), (16, 2, 14), (24, 12, 11), (40, 3, 2)])
def test_count_pass_and_draws(ctx, K, na, nb):
    """Lists, weights and draws at block edges of the canonical order (empty and
    one-chunk blocks, short (j, b) runs, every weight width) against the oracle,
    bit by bit."""
    import dataclasses
    from oracle import oracle as O
    rng = np.random.default_rng(K)
    dec = W._decay_1d(K, 2.0)
    h, L = W._banded_h(rng, K, dec), W._sym_chol(rng, 2 * K, K, 0.3, dec)
    smp = W.random_dets(rng, K, na, nb, 3) if K > 5 else W.all_dets(K, na, nb)[:4]
    base = W.tiny_system(K=4, D=1)
    s = dataclasses.replace(base, K=K, n_alpha=na, n_beta=nb, h1e=h, chol=L, tensors=np.ones((K, 4, 1, 1)), samples=smp,
                            counts=np.ones(len(smp)))
    P = O.Problem(s)
    ctx.set_system(s)
    for eps in (0.0, 3e-3, 0.1, 1e3):
        off, rank, dets, H, sg = ctx.connected(s.samples, eps)
        ranks, w = ctx.draws(s.samples, eps, 300, 9)
        for i, d in enumerate(s.samples):
            od, oH, osg = O.connected(P, d)
            keep = np.abs(oH) >= eps
            assert np.array_equal(H[off[i]:off[i + 1]], oH[keep]) and np.array_equal(sg[off[i]:off[i + 1]], osg[keep])
            assert np.array_equal(rank[off[i]:off[i + 1]], np.flatnonzero(keep).astype(np.uint32))
            ref, rw, _ = O.draws(P, d, i, eps, 300, 9)
            assert int(w[i]) == int(rw) and np.array_equal(ranks[i], ref)


@pytest.mark.parametrize("D,ns", [(80, 131), (96, 5), (96, 300), (112, 131), (128, 300), (192, 130), (256, 1), (256, 130)])
def test_site_steps_of_wide_bonds(ctx, D, ns):
    """Site steps of 64 < D <= 256: one reduction chunk or several, tiles of one
    row to full ones, several matrices per block. Mixed bar, and 2^-20 of the
    rows' conditioning: both operands of a product carry 22 bits, lo x lo is left
    out, and the sums are FP32 (about 4 x 2^-22 a product)."""
    from oracle import oracle as O
    s = W.tiny_system(K=7, na=3, nb=4, D=D, n_hidden=5, seed=90 + D, eps=0.01, n_draws=20, n_samples=ns)
    ctx.set_system(s)
    ctx.set_precision(nqs.NQS_PREC_MIXED)
    try:
        e, summ = ctx.local_energy(s.samples, s.counts, s.eps, s.n_draws, s.seed)
    finally:
        ctx.set_precision(nqs.NQS_PREC_FP64)
    ref = O.local_energy(O.Problem(s), cond=True)
    bar = 1e-6 * np.maximum(np.abs(ref["e_loc"]), ref["e_abs"]) + 2.0 ** -20 * ref["e_cond"]
    assert np.all(np.abs(e - ref["e_loc"]) <= bar)
    assert summ["n_det"] == int(ref["n_det"].sum())


@pytest.mark.parametrize("D,nh", [(5, 0), (16, 3), (50, 0), (64, 3), (80, 3), (130, 0), (256, 3)])
def test_full_batches_equal_small_ones(ctx, D, nh):
    """Boundary vectors and psi(n) of batches that fill the GPU (several samples
    per block, the last block short) against the same samples in small calls
    (one per block): every row's arithmetic is the same, so are the results (without
    a tolerance: which samples are re-evaluated depends on the batch)."""
    s = W.tiny_system(K=8, na=4, nb=4, D=D, n_hidden=nh, seed=70 + D, eps=0.02, n_draws=10, n_samples=4900)
    n = 4133
    ctx.set_system(s)
    parts = (0, 2000, n - 500)
    try:
        ctx.set_precision(nqs.NQS_PREC_MIXED)
        e, _ = ctx.local_energy(s.samples[:n], s.counts[:n], s.eps, s.n_draws, s.seed)
        got = []
        for i in parts:
            ctx.set_precision(nqs.NQS_PREC_MIXED, sample_index_base=i)
            got.append(ctx.local_energy(s.samples[i:i + 500], s.counts[i:i + 500], s.eps, s.n_draws, s.seed)[0])
    finally:
        ctx.set_precision(nqs.NQS_PREC_FP64)
    for i, p in zip(parts, got):
        assert np.array_equal(p, e[i:i + 500])


@pytest.mark.parametrize("D", [16, 32, 64])
def test_graph_tiles_beyond_the_ring(ctx, D):
    """Vertex steps with many tiles per block (the ring of source states and the
    accumulators go round several times) against the same samples in small calls;
    a node's arithmetic is its own, so the results are equal."""
    import dataclasses
    s = _dag(40 + D, 8, D, n_samples=4800, eps=0.0, n_draws=0)
    if D == 64:                                    # one in-edge (two matrices' images are refused)
        ptr, idx, keep = [0], [], []
        for i in range(s.K):
            e = list(range(s.pred_ptr[i], s.pred_ptr[i + 1]))[-1:]
            keep += e
            idx += [int(s.pred_idx[x]) for x in e]
            ptr.append(len(idx))
        s = dataclasses.replace(s, pred_ptr=np.array(ptr, np.int32), pred_idx=np.array(idx, np.int32),
                                tensors=np.ascontiguousarray(s.tensors[keep]))
    ctx.set_system(s)
    ctx.set_precision(nqs.NQS_PREC_MIXED)
    try:
        e, _ = ctx.local_energy(s.samples, s.counts, 0.0, 0, 1)
        for i in (0, len(e) // 2, len(e) - 40):
            p, _ = ctx.local_energy(s.samples[i:i + 40], s.counts[i:i + 40], 0.0, 0, 1)
            assert np.array_equal(p, e[i:i + 40])
    finally:
        ctx.set_precision(nqs.NQS_PREC_FP64)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("kind", ["theta", "path"])
def test_correlator_ratio_of_large_weights(ctx, graph, kind):
    """2cosh ratios whose factors are far apart but whose product is not: an angle past
    the range of e^(-2 theta), and products that pass through the denormal numbers and
    come back (units 0, 8, 16, .. belong to one lane); the FP64 bar."""
    import dataclasses
    from oracle import oracle as O
    s = W.tiny_system(K=6, na=3, nb=3, D=4, seed=8, graph=graph, n_samples=120)
    nh = 2 if kind == "theta" else 41
    Wc, b = np.zeros((nh, 2 * s.K)), np.zeros(nh)
    # (occupied, empty) angles of orbital 0 alpha per unit: the factors' logarithms add to zero
    units = {0: (380.0, -20.0), 1: (20.0, 380.0)} if kind == "theta" else \
        {0: (330.0, -20.0), 8: (330.0, -20.0), 16: (120.0, -5.0),
         24: (20.0, 330.0), 32: (20.0, 330.0), 40: (5.0, 120.0)}
    for k, (occ, emp) in units.items():
        b[k], Wc[k, 0] = emp, occ - emp
    Wc += 0.1 * np.random.default_rng(1).normal(size=Wc.shape) * (np.arange(2 * s.K) > 1)
    s = dataclasses.replace(s, rbm_W=Wc, rbm_b=b)
    ctx.set_system(s)
    ctx.set_precision(nqs.NQS_PREC_FP64)
    ref = O.local_energy(O.Problem(s), cond=True)
    e, _ = ctx.local_energy(s.samples, s.counts, s.eps, s.n_draws, s.seed)
    scale = np.maximum(np.abs(ref["e_loc"]), ref["e_abs"]) + (2.0 ** -52 / 1e-12) * ref["e_cond"]
    assert np.all(np.abs(e - ref["e_loc"]) <= 1e-12 * scale)


@pytest.mark.parametrize("D", [4, 28])
def test_normalised_chain_tiny_conditionals(ctx, D):
    """Conditionals of 1e-240 at two vertices (every local state is allowed there) whose
    orbitals couple to no other, so that every m shares them with n: their product
    leaves the range of a double, the ratio does not."""
    import dataclasses
    from oracle import oracle as O
    s = W.with_readout(W.tiny_system(K=8, na=4, nb=4, D=D, seed=6), seed=4, v_std=1.0)
    T, (v, eta, w, c) = s.tensors.copy(), s.rnn
    v = v.copy()
    for q in (1, 3):
        T[q, 3] *= 1e-120
        v[q, 3] = 0.0
    h, L = s.h1e.copy(), s.chol.copy()
    alone = np.ones((s.K, s.K), bool)
    alone[[1, 3]], alone[:, [1, 3]] = False, False
    alone |= np.eye(s.K, dtype=bool)
    both = np.uint64((1 << 1) | (1 << 3))
    s = dataclasses.replace(s, tensors=T, rnn=(v, eta, w, c), h1e=h * alone, chol=L * alone, eps=1e-9)
    s = s.subset(np.flatnonzero(np.all((s.samples & both) == both, axis=1)))
    ctx.set_system(s)
    ctx.set_precision(nqs.NQS_PREC_FP64)
    ref = O.local_energy(O.Problem(s))
    first = (s.samples & np.uint64(1)).sum(1)          # one electron on orbital 0: m may change there
    assert np.all(ref["n_det"] > 0) and np.any(first == 1) and np.all(ref["e_abs"] < 1e6)
    e, _ = ctx.local_energy(s.samples, s.counts, s.eps, 0, 1)
    assert np.all(np.abs(e - ref["e_loc"]) <= 1e-12 * np.maximum(np.abs(ref["e_loc"]), ref["e_abs"]))


@pytest.mark.parametrize("kind", ["many weak units", "units that cancel"])
def test_shared_correlator_product(ctx, kind):
    """The product over hidden units in the shared FP64 form, alone: a chain of ones, one
    electron, one-body elements between pairs of orbitals, so E_loc = H f(m)/f(n) of one m.
    Weak units: each of the factors 1 + x_k and of the two outer products counts with four
    roundings of its x, the rest with four (the two products, the sum, the outer ones).
    Units that cancel: products of 2^-60 and 2^60 whose value is 1, 16 roundings per unit."""
    import dataclasses
    K, rng = 16, np.random.default_rng(5)
    nh = 512 if kind == "many weak units" else 60
    s = W.tiny_system(K=K, na=1, nb=0, D=1, n_hidden=nh, seed=3)
    if kind == "many weak units":
        Wc, b = 1e-3 * rng.normal(size=(nh, 2 * K)), 1e-3 * rng.normal(size=nh)
    else:
        Wc, b = 0.9 + 1e-3 * rng.normal(size=(nh, 2 * K)), -0.9 + 1e-3 * rng.normal(size=nh)
    h = np.zeros((K, K))
    h[np.arange(0, K, 2), np.arange(1, K, 2)] = h[np.arange(1, K, 2), np.arange(0, K, 2)] = rng.normal(size=K // 2)
    s = dataclasses.replace(s, tensors=np.ones_like(s.tensors), rbm_W=Wc, rbm_b=b, h1e=h, chol=np.zeros_like(s.chol))
    ctx.set_system(s)
    ctx.set_precision(nqs.NQS_PREC_FP64_SHARED)
    try:
        e, _ = ctx.local_energy(s.samples, s.counts, 1e-9, 0, 1)
    finally:
        ctx.set_precision(nqs.NQS_PREC_FP64)
    off, _, dets, H, _ = ctx.connected(s.samples, 1e-9)
    assert np.array_equal(np.diff(off), np.ones(K))

    def theta(d):
        bits = (d[:, None, :] >> np.arange(K, dtype=np.uint64)[None, :, None]) & np.uint64(1)
        return b.astype(np.longdouble) + bits.reshape(len(d), 2 * K).astype(np.longdouble) @ Wc.T.astype(np.longdouble)
    tn, tm = theta(s.samples), theta(dets)
    ref = H * np.exp(np.sum(np.log(np.cosh(tm)) - np.log(np.cosh(tn)), axis=1))
    x = np.maximum(np.abs(tn), np.abs(tm)) + 2 * np.abs(Wc).max()
    units = 4 * (1 + np.sum(x * x, axis=1).max()) if kind == "many weak units" else 16 * (1 + nh)
    assert kind != "many weak units" or units < 5
    assert np.all(np.abs(e - ref) <= float(units) * 2.0 ** -53 * np.abs(ref))


_FAKE_MALLOC = """
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
#include <stdlib.h>
int cudaMalloc(void** p, size_t n)
{
    static int (*real)(void**, size_t);
    if (n > strtoull(getenv("FAKE_MALLOC_LIMIT"), NULL, 10)) { *p = NULL; return 2; }
    if (!real) real = (int (*)(void**, size_t))dlsym(RTLD_NEXT, "cudaMalloc");
    return real(p, n);
}
"""

_FAKE_MALLOC_RUN = """
import sys
import numpy as np
from paper_2507_19276_gb300 import nqs, workloads as W
kind, out = sys.argv[1:]
s = W.tiny_system(K=8, na=4, nb=4, D=16, n_hidden=3, seed=4, graph=kind != "readout", n_samples=2500)
if kind == "readout":
    s = W.with_readout(s, seed=3)
c = nqs.Context(0)
c.set_system(s)
c.set_precision(nqs.NQS_PREC_MIXED if kind == "mixed" else nqs.NQS_PREC_FP64)
np.save(out, c.local_energy(s.samples, s.counts, 0.0, 0, 1)[0])
"""


@pytest.mark.parametrize("kind", ["plain", "mixed", "readout"])
def test_tree_batches_shrink_to_the_memory(tmp_path, kind):
    """An allocation refused by the runtime (a fake cudaMalloc in a child process: nothing
    past 64 MiB) cuts the batch of the prefix trees, and the energies keep their bits."""
    import os
    import subprocess
    import sys
    src, so, root = tmp_path / "fake.c", tmp_path / "fake.so", os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    src.write_text(_FAKE_MALLOC)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src), "-ldl"], check=True)
    got = []
    for limit in (1 << 60, 64 << 20):
        out = tmp_path / f"{limit}.npy"
        env = dict(os.environ, LD_PRELOAD=str(so), FAKE_MALLOC_LIMIT=str(limit))
        r = subprocess.run([sys.executable, "-c", _FAKE_MALLOC_RUN, kind, str(out)], cwd=root, env=env, capture_output=True,
                           text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        got.append(np.load(out))
    assert np.array_equal(got[0].view(np.uint64), got[1].view(np.uint64))
