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
    """Value of `constexpr ... name = value;` in the CUDA sources."""
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as h:
            m = re.search(r"constexpr\s+\w+\s+" + name + r"\s*=\s*(\d+)\s*;", h.read())
        if m:
            return int(m.group(1))
    raise KeyError(name)


ROWS = _const("kFxMinRows")          # determinants from which a chain's sweeps take the steps


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


def _assert_log_psi(ctx, s, dets):
    """K (D + 1) 2^-53 of the running absolute product: the bound of an FP64 chain."""
    ctx.set_system(s)
    la, sg = ctx.amplitude(dets)
    ref, rs, cond = _log_psi_ref(s, dets)
    tol = s.K * (s.D + 1) * U * cond + 8 * U * np.abs(ref)
    ok = tol < 1e-3
    assert ok.sum() > len(dets) // 2
    assert np.all(np.abs(la - ref)[ok] <= tol[ok]) and np.array_equal(sg[ok], rs[ok])


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
    n = ROWS + 101
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
