"""The fixed-point tensor-core steps (nqs_fx.cu) where one power of two per row
is not enough by itself: matrices with empty columns, states and matrices whose
entries spread over many powers of two, infinities and NaN. Sizes follow the
thresholds of the dispatch, read from the sources, so that the steps are reached
wherever the thresholds lie."""
import dataclasses
import os
import re

import numpy as np
import pytest

from paper_2507_19276_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import oracle as O  # noqa: E402
from paper_2507_19276_gb300 import nqs  # noqa: E402
from paper_2507_19276_gb300.build import CSRC  # noqa: E402
from .test_gpu_edges import _dag, _log_psi_ref  # noqa: E402

U = 2.0 ** -53


def _const(name):
    """Value of `constexpr ... name = value` in the CUDA sources."""
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as h:
            m = re.search(r"constexpr\s+\w+\s+(?:\w+\s*=\s*\d+\s*,\s*)*" + name + r"\s*=\s*(\d+)\s*[,;]", h.read())
        if m:
            return int(m.group(1))
    raise KeyError(name)


def _rows(D):
    """Determinants from which a chain's sweeps take the steps."""
    return _const("kFxMinRows" if D >= 48 else "kFxMinRowsNarrow")


@pytest.fixture(scope="module")
def ctx():
    c = nqs.Context(0)
    yield c
    c.close()


def _energy(ctx, s, prec=nqs.NQS_PREC_FP64):
    ctx.set_system(s)
    ctx.set_precision(prec)
    try:
        return ctx.local_energy(s.samples, s.counts, s.eps, s.n_draws, s.seed)[0]
    finally:
        ctx.set_precision(nqs.NQS_PREC_FP64)


def _assert_energy(e, ref):
    """The FP64 bar of the other parity tests."""
    scale = np.maximum(np.abs(ref["e_loc"]), ref["e_abs"]) + (2.0 ** -52 / 1e-12) * np.nan_to_num(ref["e_cond"])
    assert np.all(np.isfinite(ref["e_loc"]))
    assert np.all(np.abs(e - ref["e_loc"]) <= 1e-12 * scale)


def _assert_log_psi(ctx, s, dets, run=None):
    """K (D + 1) 2^-53 of the running absolute product: the bound of an FP64 chain.
    ``run``: the system handed to the library, where it is not the reference's."""
    ctx.set_system(s if run is None else run)
    la, sg = ctx.amplitude(dets)
    ref, rs, cond = _log_psi_ref(s, dets)
    tol = s.K * (s.D + 1) * U * cond + 8 * U * np.abs(ref)
    ok = tol < 1e-3
    assert ok.sum() > len(dets) // 2
    assert np.all(np.abs(la - ref)[ok] <= tol[ok]) and np.array_equal(sg[ok], rs[ok])


@pytest.mark.parametrize("D", [16, 32, 48, 64])
@pytest.mark.parametrize("over", [-1, 0, 1, 701])
def test_log_psi_at_the_line(ctx, D, over):
    """Dense rows of unlike size on both sides of the size from which the steps run, one
    launch per site: every width, part tiles of every local state."""
    n, rng = _rows(D) + over, np.random.default_rng(D)
    s = W.tiny_system(K=8, na=4, nb=4, D=D, seed=D, n_samples=n)
    s = dataclasses.replace(s, tensors=s.tensors * np.exp2(rng.integers(-20, 8, size=(s.K, 4, D, 1))))
    ctx.set_system(s)
    ctx.stage_times()
    la, sg = ctx.amplitude(s.samples)
    launches = sum(k for _, k in ctx.stage_times().values())
    assert len(la) == n and (launches >= s.K) == (over >= 0)
    pick = rng.choice(n, 500, replace=False)
    ref, rs, cond = _log_psi_ref(s, s.samples[pick])
    tol = s.K * (D + 1) * U * cond + 8 * U * np.abs(ref)
    ok = tol < 1e-3
    assert ok.sum() > 250
    assert np.all(np.abs(la[pick] - ref)[ok] <= tol[ok]) and np.array_equal(sg[pick][ok], rs[ok])


def _isometric(rng, K, D):
    """Site tensors with sum_s M^s^T M^s = 1."""
    q = [np.linalg.qr(rng.normal(size=(4 * D, D)))[0].reshape(4, D, D) for _ in range(K)]
    return np.ascontiguousarray(np.stack(q))


@pytest.mark.parametrize("D", [10, 16, 20])
def test_normalised_chain_without_v(ctx, D):
    """The matrix-product limit of the normalised readout: v = 0, isometric tensors,
    the cells shrink with the probability of the prefix over 50 sites."""
    rng = np.random.default_rng(D)
    s = W.h50_chain(n_samples=3, D=D, n_hidden=0, eps=1e-2, n_draws=100)
    rnn = (np.zeros((s.K, 4, D)), np.ones((s.K, D)), rng.normal(size=(s.K, D)), np.zeros(s.K))
    s = dataclasses.replace(s, tensors=_isometric(rng, s.K, D), rnn=rnn)
    e = _energy(ctx, s)
    ref = O.local_energy(O.Problem(s))
    assert np.all(np.abs(e - ref["e_loc"]) <= 1e-12 * np.maximum(np.abs(ref["e_loc"]), ref["e_abs"]))


@pytest.mark.parametrize("D", [16, 32, 48, 64])
@pytest.mark.parametrize("graph", [False, True])
def test_empty_columns(ctx, D, graph):
    """Columns and rows without entries in small site tensors (2^-40), the states'
    entries there of order one: they meet only zeros and must not set the scale."""
    n = _rows(D) + 101
    if graph:
        s = _dag(D, 8, D, n_samples=150, eps=0.01, n_draws=20)
    else:
        s = W.tiny_system(K=8, na=4, nb=4, D=D, n_hidden=3, seed=D, n_samples=n, eps=0.01, n_draws=20)
    T = s.tensors * 2.0 ** -40
    T[:, :, :, 3] = 0.0                       # column 3 empty, row 3 not
    T[:, :, 5, :] = 0.0                       # the same for the transposed products
    s = dataclasses.replace(s, tensors=np.ascontiguousarray(T))
    if not graph:
        _assert_log_psi(ctx, dataclasses.replace(s, rbm_W=None, rbm_b=None), s.samples)
        s = s.subset(np.arange(200))
    ref = O.local_energy(O.Problem(s), cond=True)
    _assert_energy(_energy(ctx, s), ref)
    if not graph:
        _assert_energy(_energy(ctx, s, nqs.NQS_PREC_FP64_SHARED), ref)


def _graded(rng, s, kind):
    """Tensors whose states spread over many powers of two in a way that no scaling of
    columns and rows takes out: the first cell falls by 2^-4 per component ("steps")
    or the second half of the components by 2^-6 per site ("blocks"), the matrices in
    between keep the components apart, and the last one weighs them all alike."""
    E, D, K = s.n_edges, s.D, s.K
    idx = s.pred_idx if s.pred_idx is not None else np.arange(-1, K - 1)
    ptr = s.pred_ptr if s.pred_ptr is not None else np.arange(K + 1)
    r = lambda *n: rng.uniform(0.5, 1.5, size=n) * rng.choice([-1.0, 1.0], size=n)  # noqa: E731
    T = np.zeros((E, 4, D, D))
    k = np.arange(D)
    for e in range(E):
        if kind == "steps":
            T[e][:, k, k] = r(4, D)
            if idx[e] < 0:
                T[e][:, :, 0] = r(4, D) * np.exp2(-4.0 * k)
        else:
            h = D // 2
            T[e][:, :h, :h] = rng.normal(size=(4, h, h)) / np.sqrt(h)
            T[e][:, h:, h:] = rng.normal(size=(4, D - h, D - h)) / np.sqrt(D - h) * 2.0 ** -6
            if idx[e] < 0:
                T[e][:, :, 0] = r(4, D)
    for e in range(ptr[K - 1], ptr[K]):          # every source's components count alike in psi
        T[e][:, 0, :] = r(4, D) * (np.exp2(4.0 * k) if kind == "steps" else np.where(k < D // 2, 1.0, 2.0 ** (6 * K)))
    return dataclasses.replace(s, tensors=np.ascontiguousarray(T))


@pytest.mark.parametrize("D", [16, 32, 48, 64])
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("kind", ["steps", "blocks"])
def test_graded_states(ctx, D, graph, kind):
    """Components far below their row's largest that a later site brings up again."""
    rng = np.random.default_rng(D)
    if graph:
        s = _dag(D, 8, D, n_samples=150, eps=0.01, n_draws=20)
    else:
        s = W.tiny_system(K=8, na=4, nb=4, D=D, n_hidden=3, seed=D, n_samples=_rows(D) + 101, eps=0.01, n_draws=20)
    s = _graded(rng, s, kind)
    if not graph:
        _assert_log_psi(ctx, dataclasses.replace(s, rbm_W=None, rbm_b=None), s.samples)
        s = s.subset(np.arange(200))
    ref = O.local_energy(O.Problem(s), cond=True)
    _assert_energy(_energy(ctx, s), ref)
    if not graph:
        _assert_energy(_energy(ctx, s, nqs.NQS_PREC_FP64_SHARED), ref)


@pytest.mark.parametrize("D", [5, 10, 16, 20, 24])
@pytest.mark.parametrize("v", [0.0, 1e-3, 1.0])
def test_graded_cells(ctx, D, v):
    """The same for the normalised readout: cells that fall by 2^-4 per component, whose
    weights and phases count every component alike; v of one local state alone."""
    rng = np.random.default_rng(100 + D)
    s = W.tiny_system(K=8, na=4, nb=4, D=D, n_hidden=2, seed=D, eps=0.01, n_draws=20, n_samples=200)
    r = lambda *n: rng.uniform(0.5, 1.5, size=n) * rng.choice([-1.0, 1.0], size=n)  # noqa: E731
    k = np.arange(D)
    T = np.zeros((s.K, 4, D, D))
    T[:, :, k, k] = r(s.K, 4, D)
    T[0, :, :, 0] = r(4, D) * np.exp2(-4.0 * k)
    vv = np.zeros((s.K, 4, D))
    vv[:, 2] = v * r(s.K, D)
    rnn = (vv, np.abs(r(s.K, D)) * np.exp2(8.0 * k), r(s.K, D) * np.exp2(4.0 * k), np.zeros(s.K))
    s = dataclasses.replace(s, tensors=T, rnn=rnn)
    ref = O.local_energy(O.Problem(s))
    e = _energy(ctx, s)
    assert np.all(np.abs(e - ref["e_loc"]) <= 1e-12 * np.maximum(np.abs(ref["e_loc"]), ref["e_abs"]))


@pytest.mark.parametrize("D", [16, 64])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite_steps(ctx, D, bad):
    """A NaN or an infinity in a site tensor reaches every amplitude whose local state
    reads it, and none whose does not; the last site's unread rows reach none."""
    s = W.tiny_system(K=8, na=4, nb=4, D=D, seed=1, n_samples=_rows(D) + 101)
    occ = ((s.samples[:, None, :] >> np.arange(s.K, dtype=np.uint64)[None, :, None]) & np.uint64(1)).astype(int)
    T = s.tensors.copy()
    T[5, 3, 2, 7] = bad
    ctx.set_system(dataclasses.replace(s, tensors=T))
    la, _ = ctx.amplitude(s.samples)
    hit = occ[:, 5].sum(1) == 2
    assert not np.any(np.isfinite(la[hit])) and np.all(np.isfinite(la[~hit]))
    T = s.tensors.copy()
    T[-1, :, 1:, :] = bad
    _assert_log_psi(ctx, s, s.samples, dataclasses.replace(s, tensors=T))


@pytest.mark.parametrize("graph", [False, True])
def test_not_finite_levels(ctx, graph):
    """The same for the levels of the prefix trees: an energy is NaN where the oracle's
    is. Samples without the bad local state themselves; vertex 4, which the last one
    reads in the graph too."""
    s = W.tiny_system(K=8, na=4, nb=4, D=16, seed=2, n_samples=3000) if not graph else _dag(3, 8, 16, n_samples=3000)
    occ = ((s.samples[:, None, :] >> np.arange(s.K, dtype=np.uint64)[None, :, None]) & np.uint64(1)).astype(int)
    s = s.subset(np.flatnonzero(occ[:, 4].sum(1) < 2)[:300])
    e = s.pred_ptr[4] if graph else 4
    T = s.tensors.copy()
    T[e, 3, 2, 0] = np.nan                         # (column 0: read from e_0 too)
    s = dataclasses.replace(s, tensors=T, eps=0.3)
    ref = O.local_energy(O.Problem(s))["e_loc"]
    got = _energy(ctx, s)
    assert np.isnan(ref).any() and np.array_equal(np.isnan(got), np.isnan(ref))
    ok = ~np.isnan(ref)
    assert np.all(np.abs(got - ref)[ok] <= 1e-9 * np.abs(ref[ok]).max(initial=1.0))


GRAD = _const("kFxGradMin")           # samples from which the gradient takes the fixed-point products
CHUNK = _const("kGradChunk")          # samples per block, in products of kGradRed
RED = _const("kGradRed")


def _grad_ref(s, u):
    """sum_n u_n d log|psi_TN(n)| / d M_e^s in float64 over any graph, and 2 K (D + 1)
    2^-53 times the same sum of magnitudes (of the products of absolute values, times
    the conditioning of psi(n)): the rounding of FP64 recursions, both ways."""
    E, K, D = s.n_edges, s.K, s.D
    idx = s.pred_idx if s.pred_idx is not None else np.arange(-1, K - 1)
    ptr = s.pred_ptr if s.pred_ptr is not None else np.arange(K + 1)
    occ = ((s.samples[:, None, :] >> np.arange(K, dtype=np.uint64)[None, :, None]) & np.uint64(1)).astype(int)
    sig = occ[:, :, 0] + 2 * occ[:, :, 1]
    n = len(sig)
    e0 = np.eye(1, D)[0][None, :].repeat(n, 0)
    vert = np.repeat(np.arange(K), np.diff(ptr))
    out = []
    for T in (s.tensors, np.abs(s.tensors)):
        M = [T[e][sig[:, vert[e]]] for e in range(E)]
        h = {-1: e0}
        for i in range(K):
            h[i] = sum(np.einsum("nab,nb->na", M[e], h[idx[e]]) for e in range(ptr[i], ptr[i + 1]))
        g = {i: np.zeros((n, D)) for i in range(-1, K)}
        g[K - 1] = e0
        for i in range(K - 1, -1, -1):
            for e in range(ptr[i], ptr[i + 1]):
                g[idx[e]] = g[idx[e]] + np.einsum("nab,na->nb", M[e], g[i])
        out.append((h, g, h[K - 1][:, 0]))
    (h, g, psi), (ha, ga, psia) = out
    ref, mag = np.zeros(s.tensors.shape), np.zeros(s.tensors.shape)
    w = u / psi
    wa = np.abs(w) * (1.0 + psia / np.abs(psi))
    for e in range(E):
        for q in range(4):
            k = sig[:, vert[e]] == q
            ref[e, q] = (w[k, None] * g[vert[e]][k]).T @ h[idx[e]][k]
            mag[e, q] = (wa[k, None] * ga[vert[e]][k]).T @ ha[idx[e]][k]
    return ref, 2 * K * (D + 1) * U * mag


@pytest.mark.parametrize("D", [16, 32, 48, 64])
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("n", [GRAD - 1, GRAD, GRAD + 1, CHUNK - 1, CHUNK + 1, 4 * RED + 1, 4 * CHUNK + 3])
def test_outer_products(ctx, D, graph, n):
    """Groups around a product's samples and a block's, weights over 2^40."""
    s = W.tiny_system(K=7, na=3, nb=4, D=D, seed=n, n_samples=n) if not graph else _dag(n, 7, D, n_hidden=0, n_samples=n)
    rng = np.random.default_rng(D + n)
    n = len(s.samples)
    u = rng.normal(size=n) * np.exp2(rng.uniform(-20, 20, size=n))
    ctx.set_system(s)
    got = ctx.grad_log_psi_vjp(s.samples, u)[0]
    ref, tol = _grad_ref(s, u)
    assert np.all(np.abs(got - ref) <= tol)


@pytest.mark.parametrize("D", [16, 64])
def test_outer_products_of_sectors(ctx, D):
    """States of two sectors of components, the samples of one with weights 2^45 times
    the other's: the entries that only the light samples reach keep their digits."""
    s = W.tiny_system(K=7, na=3, nb=4, D=D, seed=5, n_samples=600)
    rng = np.random.default_rng(D)
    h = D // 2
    T = np.zeros_like(s.tensors)
    T[:, :, :h, :h] = rng.normal(size=(s.K, 4, h, h)) / np.sqrt(h)
    T[:, :, h:, h:] = rng.normal(size=(s.K, 4, D - h, D - h)) / np.sqrt(D - h)
    T[0] = 0.0
    T[0, 0::2, :h, 0] = rng.normal(size=(2, h))          # local states 0, 2: the first sector
    T[0, 1::2, h:, 0] = rng.normal(size=(2, D - h))
    T[-1, :, 0, :] = rng.normal(size=(4, D))
    s = dataclasses.replace(s, tensors=T)
    light = (s.samples[:, 0] & np.uint64(1)) == 1
    u = rng.normal(size=len(light)) * np.where(light, 1.0, 2.0 ** 45)
    ctx.set_system(s)
    got = ctx.grad_log_psi_vjp(s.samples, u)[0]
    ref, tol = _grad_ref(s, u)
    assert np.all(np.abs(got - ref) <= tol)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_outer_products_not_finite(ctx, bad):
    """A weight that is not finite reaches the gradients of its sample's local states."""
    s = W.tiny_system(K=7, na=3, nb=4, D=16, seed=5, n_samples=600)
    u = np.random.default_rng(1).normal(size=600)
    u[77] = bad
    ctx.set_system(s)
    got = ctx.grad_log_psi_vjp(s.samples, u)[0]
    occ = ((s.samples[77] >> np.arange(s.K, dtype=np.uint64)[:, None]) & np.uint64(1)).astype(int)
    hit = np.zeros((s.K, 4), bool)
    hit[np.arange(s.K), occ[:, 0] + 2 * occ[:, 1]] = True
    finite = np.isfinite(got)
    assert np.all(finite[~hit]) and not np.any(finite[1:-1][hit[1:-1]])


@pytest.mark.parametrize("kind,D", [("chain", 16), ("chain", 64), ("graph", 32), ("readout", 10), ("readout", 20)])
def test_energies_do_not_depend_on_the_split(ctx, kind, D):
    """A sample's plain-form energy has the same bits in a large batch, in small calls and
    under a table cap that cuts the batch (the levels' node counts differ a hundredfold)."""
    n = 1201
    if kind == "graph":
        s = _dag(D, 8, D, n_samples=n, eps=0.02, n_draws=10)
    else:
        s = W.tiny_system(K=8, na=4, nb=4, D=D, n_hidden=3, seed=D, n_samples=n, eps=0.02, n_draws=10)
    if kind == "readout":
        s = W.with_readout(s, seed=3)
    ctx.set_system(s)

    def run(lo, hi, **options):
        ctx.set_precision(nqs.NQS_PREC_FP64, sample_index_base=lo, **options)
        return ctx.local_energy(s.samples[lo:hi], s.counts[lo:hi], s.eps, s.n_draws, s.seed)[0].view(np.uint64)
    try:
        e = run(0, n)
        for lo, hi in [(0, 1), (3, 40), (500, 900), (n - 130, n)]:
            assert np.array_equal(run(lo, hi), e[lo:hi])
        assert np.array_equal(run(0, n, table_mb=1), e)
    finally:
        ctx.set_precision(nqs.NQS_PREC_FP64)
