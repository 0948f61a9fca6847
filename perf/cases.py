"""The workloads that the library's speed is measured on.

A variational Monte Carlo program over this library samples determinants, takes
their local energies in one of the precision forms, and differentiates; the
cases are those calls, through the Python entry points, at the sizes of the
configurations in ``workloads.py`` and of the tests, from a 256-sample K = 8
batch to whole H50, Fe2S2 and H18 batches:

  energy    Context.local_energy on device-resident samples (every precision
            form; chain, grid-graph and dense systems; linear and normalised
            readout; with and without the stochastic part)
  gradient  Context.energy_gradient on host samples
  log_psi   forward and backward of the differentiable log|psi|, parameters
            uploaded each time as in a training loop
  sample    Context.sample, autoregressive sampling of the normalised readout
  batch     local_energy_batch over independent systems on their own streams

``exact`` evaluates the same formulas in plain float64 torch: every connected
determinant is enumerated by index arithmetic, every amplitude is a full
product over the sites.
"""
import math

import numpy as np
import torch

from paper_2507_19276_gb300 import nqs
from paper_2507_19276_gb300 import workloads as W

PREC = {"fp64": nqs.NQS_PREC_FP64, "mixed": nqs.NQS_PREC_MIXED, "fp64_shared": nqs.NQS_PREC_FP64_SHARED}


def _energy(name, system, K, D, hidden, samples, eps, draws, precision, tol=0.0, readout="linear"):
    c = dict(kind="energy", system=system, K=K, D=D, hidden=hidden, samples=samples, eps=eps,
             draws=draws, precision=precision, tol=tol, readout=readout)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call in use: the K = 8 configuration, default precision; launches and waits count
        _energy("k8 fp64", "chain", 8, 8, 0, 256, 0.0, 0, "fp64"),
        # the headline batch: H50 shape, mixed form held to 1e-6 Ha on the mean energy
        _energy("h50 mixed", "chain", 50, 64, 100, 4096, 1e-3, 1024, "mixed", 1e-6),
        # an ordinary optimisation step at the published eps = 0.01, N_eps = 100, ragged batch
        _energy("h50 mixed ragged", "chain", 50, 64, 100, 777, 1e-2, 100, "mixed"),
        # dense active space, largest bond dimension, everything deterministic
        _energy("fe2s2 mixed", "dense", 20, 256, 40, 8192, 0.0, 0, "mixed", 1e-6),
        # graph-ordered ansatz on the 3 x 3 x 2 cluster, whole batch
        _energy("h18 mixed", "grid", 18, 32, 36, 16384, 0.0, 0, "mixed", 1e-6),
        # the same ansatz in the default precision: a check batch
        _energy("h18 fp64", "grid", 18, 32, 36, 200, 0.0, 0, "fp64"),
        # FP64 shared-prefix form: the check of a mixed H50 batch
        _energy("h50 fp64 shared", "chain", 50, 64, 100, 200, 1e-3, 1024, "fp64_shared"),
        # normalised readout at chi = 10 (the published H50 setting)
        _energy("h50 rnn", "chain", 50, 10, 0, 300, 1e-2, 100, "fp64", 0.0, "rnn"),
        # the sampler that feeds it
        dict(name="h50 sample", kind="sample", system="chain", K=50, D=10, hidden=0, samples=4096, readout="rnn"),
        # one pass of a training loop over log|psi|: upload, forward, backward
        dict(name="h50 log_psi", kind="log_psi", system="chain", K=50, D=64, hidden=100, samples=4096),
        # the energy gradient of a small graph batch from host arrays
        dict(name="h18 gradient", kind="gradient", system="grid", K=18, D=32, hidden=36, samples=1000,
             eps=0.0, draws=0, precision="mixed", tol=0.0),
        # independent chains of uneven size in one call
        dict(name="uneven batch", kind="batch", systems=16, draws=1024, eps=1e-3, tol=1e-6, precision="mixed"),
    ]


# ---- sizes ------------------------------------------------------------------

def _electrons(case):
    return (15, 15) if case["system"] == "dense" else (case["K"] // 2, case["K"] // 2)


def _n_conn(K, na, nb):
    sa, sb = na * (K - na), nb * (K - nb)
    c2 = lambda n: n * (n - 1) // 2  # noqa: E731
    return sa + sb + c2(na) * c2(K - na) + c2(nb) * c2(K - nb) + sa * sb


def _rows(K, na, nb, eps, draws):
    """About how many amplitudes a sample needs: measured lists of the decaying integrals hold ~26 K^2
    entries above 1e-3 and ~10 K^2 above 1e-2; nearly every draw is distinct."""
    n = _n_conn(K, na, nb)
    if eps == 0:
        return n
    return min(n, (26 if eps < 5e-3 else 10) * K * K) + draws


def _edges(case):
    return case["K"] if case["system"] != "grid" else int(len(W.grid_graph()[2]))


def _energy_flops(case):
    """Per sample: |H| of every connected determinant, and per amplitude at least one D-long product, the
    correlator, and (graph and normalised readouts, which have no right environment) the last quarter of the sites."""
    K, D = case["K"], case["D"]
    na, nb = _electrons(case)
    rows = _rows(K, na, nb, case["eps"], case["draws"])
    per = 2 * D + 2 * case["hidden"]
    if case.get("readout") == "rnn":
        per = K // 4 * 8 * D * D
    elif case["system"] == "grid":
        per = _edges(case) // 4 * 2 * D * D + 2 * case["hidden"]
    return 2.0 * _n_conn(K, na, nb) + float(rows) * per


def work(case):
    if case["kind"] == "batch":
        by = fl = 0.0
        for c in _batch_sizes(case):
            w = work(c)
            by, fl = by + w["bytes"], fl + w["flops"]
        return {"bytes": by, "flops": fl}
    K, D, n = case["K"], case["D"], case["samples"]
    tens = 8.0 * _edges(case) * 4 * D * D + 16.0 * case["hidden"] * K
    sweep = 2.0 * _edges(case) * D * D          # one forward pass of one determinant
    if case["kind"] == "sample":
        return {"bytes": tens + 24.0 * n, "flops": 4 * sweep * n / 2}
    if case["kind"] == "log_psi":
        return {"bytes": 2 * tens + 33.0 * n, "flops": 3 * sweep * n}
    by = tens + 8.0 * K ** 4 + 32.0 * n
    fl = _energy_flops(case) * n
    if case["kind"] == "gradient":
        by, fl = by + tens, fl + 3 * sweep * n
    return {"bytes": by, "flops": fl}


def _odd(rng, lo, hi):
    """Log-uniform whole number in lo..hi."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges. The sample counts are bounded so that a pass stays within the largest listed one's."""
    kind = rng.choice(["mixed", "mixed", "shared", "plain", "grid", "grid fp64", "dense", "rnn", "sample", "log_psi",
                       "gradient", "batch"])
    if kind == "batch":
        return dict(kind="batch", systems=rng.randint(3, 16), draws=rng.choice([0, 100, 1024]), eps=1e-3,
                    tol=rng.choice([0.0, 1e-6]), precision="mixed")
    if kind == "grid":
        return _energy("", "grid", 18, rng.choice([16, 32]), rng.choice([0, 36, 51]), _odd(rng, 40, 5000),
                       rng.choice([0.0, 1e-3, 2e-2]), rng.choice([0, 100]), "mixed", rng.choice([0.0, 1e-6]))
    if kind == "grid fp64":
        return _energy("", "grid", 18, rng.choice([5, 16, 32, 37]), rng.choice([0, 36]), _odd(rng, 8, 200),
                       rng.choice([0.0, 1e-3, 2e-2]), rng.choice([0, 100]), "fp64")
    if kind == "dense":
        return _energy("", "dense", 20, rng.choice([96, 128, 192, 256]), rng.choice([0, 40]), _odd(rng, 100, 6000), 0.0, 0,
                       "mixed", rng.choice([0.0, 1e-6]))
    if kind == "gradient":
        return dict(kind="gradient", system="grid", K=18, D=rng.choice([16, 32]), hidden=rng.choice([0, 36]),
                    samples=_odd(rng, 40, 2000), eps=rng.choice([0.0, 1e-3]), draws=rng.choice([0, 100]),
                    precision="mixed", tol=rng.choice([0.0, 1e-6]))
    K = 2 * rng.randint(6, 25)
    if kind == "sample":
        return dict(kind="sample", system="chain", K=K, D=rng.randint(4, 32), hidden=0,
                    samples=_odd(rng, 100, 20000), readout="rnn")
    if kind == "log_psi":
        return dict(kind="log_psi", system="chain", K=K, D=rng.randint(4, 96), hidden=rng.choice([0, 36, 100]),
                    samples=_odd(rng, 30, 4096))
    if kind == "rnn":
        return _energy("", "chain", K, rng.randint(4, 12), 0, _odd(rng, 10, 300), 1e-2, rng.choice([0, 100]), "fp64", 0.0, "rnn")
    if kind == "plain":
        return _energy("", "chain", rng.choice([6, 8, 10]), rng.randint(4, 16), rng.choice([0, 12]), _odd(rng, 10, 250),
                       rng.choice([0.0, 1e-2]), rng.choice([0, 100]), "fp64")
    if kind == "shared":
        return _energy("", "chain", K, rng.choice([12, 16, 32, 50, 64]), rng.choice([0, 100]), _odd(rng, 10, 256),
                       rng.choice([1e-3, 1e-2]), rng.choice([0, 100, 1024]), "fp64_shared")
    return _energy("", "chain", K, rng.choice([16, 32, 40, 64, 128]), rng.choice([0, 36, 100]), _odd(rng, 16, 2500),
                   rng.choice([1e-3, 1e-2]), rng.choice([0, 100, 1024]), "mixed", rng.choice([0.0, 1e-6]))


# ---- inputs -----------------------------------------------------------------

def _dets(rng, K, na, nb, n):
    """n distinct determinants, uniform over fixed N_alpha, N_beta."""
    space = math.comb(K, na) * math.comb(K, nb)
    if space <= 4 * n:
        s = W.all_dets(K, na, nb)
        return s[rng.permutation(len(s))[: min(n, len(s))]]
    got = np.zeros((0, 2), np.uint64)
    while len(got) < n:
        w = []
        for ne in (na, nb):
            p = np.argsort(rng.random((n + 64, K)), axis=1)[:, :ne].astype(np.uint64)
            w.append(np.left_shift(np.uint64(1), p).sum(axis=1, dtype=np.uint64))
        got = np.unique(np.concatenate([got, np.stack(w, 1)]), axis=0)
    return np.ascontiguousarray(got[rng.permutation(len(got))[:n]])


def _system(case, seed):
    """A workloads.System of the case's shape, by the recipes of workloads.py."""
    rng = np.random.default_rng([int(seed), 7])
    K, D, nh = case["K"], case["D"], case["hidden"]
    na, nb = _electrons(case)
    ptr = idx = mask = None
    if case["system"] == "dense":
        g = rng.normal(0.0, 0.5, size=(K, K))
        h, L, ne = 0.5 * (g + g.T), W._sym_chol(rng, 4 * K, K, 0.2, np.ones((K, K))), K
    else:
        if case["system"] == "grid":
            pos, ptr, idx, mask = W.grid_graph()
            dec = np.exp(-np.sqrt(((pos[:, None, :] - pos[None, :, :]) ** 2).sum(-1)) / 1.5)
        else:
            dec = W._decay_1d(K, 2.0)
        h, L = W._banded_h(rng, K, dec), W._sym_chol(rng, 2 * K, K, 0.3, dec)
        ne = K if ptr is None else len(idx)
    T = W._mps_tensors(rng, ne, D, identity_mask=mask)
    Wm = rng.normal(0.0, 0.01, size=(nh, 2 * K)) if nh else None
    b = rng.normal(0.0, 0.1, size=nh) if nh else None
    n = case["samples"] if case["kind"] != "sample" else 1
    s = _dets(rng, K, na, nb, n)
    rnn = W.rnn_params(rng, K, D) if case.get("readout") == "rnn" else None
    return W.System("case", K, na, nb, np.ascontiguousarray(h), L, 0.0, D, T, ptr, idx, Wm, b, s,
                    rng.zipf(1.2, size=len(s)).astype(np.float64), case.get("eps", 0.0), case.get("draws", 0),
                    int(rng.integers(1 << 40)), rnn=rnn)


def _batch_sizes(case):
    """The systems' shapes: fixed by the case, as a user's list of molecules is."""
    rng = np.random.default_rng(2507 + 100 * case["systems"] + case["draws"])
    return [dict(kind="energy", system="chain", K=int(rng.choice(np.arange(12, 41, 2))), D=int(rng.choice([16, 32, 64])),
                 hidden=0, samples=int(rng.integers(512, 4097)), eps=case["eps"], draws=case["draws"])
            for _ in range(case["systems"])]


def _gpu(x):
    x = np.ascontiguousarray(x)
    return torch.from_numpy(x.view(np.int64) if x.dtype == np.uint64 else x).cuda()


def prepare(case, seed):
    if case["kind"] == "batch":
        parts = []
        for i, c in enumerate(_batch_sizes(case)):
            s = _system(c, seed * 64 + i)
            st = torch.cuda.Stream()
            ctx = nqs.Context(0, stream=st.cuda_stream)
            ctx.set_system(s)
            ctx.set_precision(PREC[case["precision"]], energy_tolerance=case["tol"])
            parts.append((ctx, st, dict(samples=_gpu(s.samples), counts=_gpu(s.counts), eps=s.eps, n_draws=s.n_draws,
                                        seed=s.seed, out=torch.empty(len(s.samples), dtype=torch.float64, device="cuda"))))
        torch.cuda.synchronize()
        return dict(kind="batch", contexts=[p[0] for p in parts], streams=[p[1] for p in parts], args=[p[2] for p in parts])
    s = _system(case, seed)
    ctx = nqs.Context(0)
    ctx.set_system(s)
    state = dict(kind=case["kind"], ctx=ctx, n=case["samples"], eps=s.eps, draws=s.n_draws, seed=s.seed)
    if case["kind"] in ("energy", "gradient"):
        ctx.set_precision(PREC[case["precision"]], energy_tolerance=case["tol"])
    if case["kind"] == "energy":
        state |= dict(samples=_gpu(s.samples), counts=_gpu(s.counts),
                      out=torch.empty(len(s.samples), dtype=torch.float64, device="cuda"))
    elif case["kind"] == "gradient":
        state |= dict(samples=s.samples, counts=s.counts)
    elif case["kind"] == "log_psi":
        u = np.random.default_rng([int(seed), 8]).normal(size=len(s.samples))
        p = [_gpu(x).requires_grad_(True) for x in (s.tensors, s.rbm_W, s.rbm_b) if x is not None]
        state |= dict(samples=_gpu(s.samples), u=_gpu(u), params=p)
    return state


def run(state):
    k = state["kind"]
    if k == "batch":
        return [dict(e_loc=e, e_mean=m["e_mean"], n_amplitudes=m["n_amplitudes"])
                for e, m in nqs.local_energy_batch(state["contexts"], state["args"])]
    ctx = state["ctx"]
    if k == "energy":
        e, m = ctx.local_energy(state["samples"], state["counts"], state["eps"], state["draws"], state["seed"],
                                out=state["out"])
        return dict(e_loc=e, e_mean=m["e_mean"], n_amplitudes=m["n_amplitudes"])
    if k == "gradient":
        gT, gW, gb, _, e, m = ctx.energy_gradient(state["samples"], state["counts"], state["eps"], state["draws"], state["seed"])
        return dict(sites=gT, W=gW, b=gb, e_loc=e, e_mean=m["e_mean"])
    if k == "sample":
        dets, counts = ctx.sample(state["n"], state["seed"])
        return dict(dets=dets.view(np.int64), counts=counts.astype(np.int64))
    la, sg = nqs.log_psi(ctx, state["samples"], *state["params"])
    return dict(log_abs=la.detach(), sign=sg, grads=list(torch.autograd.grad(la, state["params"], state["u"])))


# ---- the same in plain float64 ----------------------------------------------

def _t(x, dev):
    return torch.as_tensor(np.ascontiguousarray(x), device=dev)


def _bits(s, K):
    """Occupations [n][2K] over the interleaved spin orbitals."""
    s = np.asarray(s, np.uint64)
    b = (s[:, None, :] >> np.arange(K, dtype=np.uint64)[None, :, None]) & np.uint64(1)
    return b.reshape(len(s), 2 * K).astype(np.int64)


def _scaled(h):
    """h divided by its rows' largest entries, and their logs."""
    m = h.detach().abs().amax(1, keepdim=True).clamp_min(1e-300)
    return h / m, m.log().squeeze(1)


def _log_psi(sys_, occ, T, Wm, b):
    """log|psi| and sign of occupations [n][2K]: one full product over the sites each."""
    dev, n, K, D = occ.device, len(occ), sys_.K, sys_.D
    sig = occ[:, 0::2] + 2 * occ[:, 1::2]
    e0 = torch.zeros(n, D, dtype=torch.float64, device=dev)
    e0[:, 0] = 1.0
    hs, ls = [], []
    log = torch.zeros(n, dtype=torch.float64, device=dev)
    sign = torch.ones_like(log)
    if sys_.rnn is not None:
        v, eta, w, c = (_t(x, dev) for x in sys_.rnn)
        na = torch.zeros(n, dtype=torch.int64, device=dev)
        nb = torch.zeros_like(na)
    for i in range(K):
        pre = [(i, i - 1)] if sys_.pred_ptr is None else [(e, int(sys_.pred_idx[e]))
                                                          for e in range(sys_.pred_ptr[i], sys_.pred_ptr[i + 1])]
        top = torch.stack([ls[j] if j >= 0 else torch.zeros_like(log) for _, j in pre]).amax(0)
        if sys_.rnn is not None:
            cand = v[i][None].expand(n, 4, D).clone()
            for e, j in pre:
                cand += torch.einsum("sab,nb->nsa", T[e], hs[j] if j >= 0 else e0)
            P = (eta[i] * cand * cand).sum(-1)
            left = K - 1 - i
            ok = []
            for s in range(4):
                ea, eb = na + (s & 1), nb + (s >> 1)
                ok.append((ea <= sys_.n_alpha) & (eb <= sys_.n_beta) & (sys_.n_alpha - ea <= left) & (sys_.n_beta - eb <= left))
            Z = (P * torch.stack(ok, 1)).sum(1)
            at = sig[:, i]
            h = cand[torch.arange(n, device=dev), at]
            log = log + 0.5 * (P.gather(1, at[:, None]).squeeze(1).log() - Z.log())
            sign = sign * torch.where((h @ w[i]) + c[i] < 0, -1.0, 1.0)
            na, nb = na + (at & 1), nb + (at >> 1)
            hs.append(h)
            ls.append(torch.zeros_like(log))
            continue
        h = torch.zeros(n, D, dtype=torch.float64, device=dev)
        for s in range(4):
            at = (sig[:, i] == s).nonzero().squeeze(1)
            part = 0.0
            for e, j in pre:
                src = hs[j][at] if j >= 0 else e0[at]
                sc = ((ls[j][at] if j >= 0 else 0.0) - top[at]).exp()
                part = part + sc[:, None] * (src @ T[e, s].T)
            h = h.index_add(0, at, part)
        h, m = _scaled(h)
        hs.append(h)
        ls.append(top + m)
    if sys_.rnn is None:
        log, sign = ls[-1] + hs[-1][:, 0].abs().log(), torch.sign(hs[-1][:, 0])
    if Wm is not None:
        th = occ.double() @ Wm.T + b
        log = log + (th.abs() + torch.log1p(torch.exp(-2 * th.abs()))).sum(1)
    return log, sign


def _mulhi(a, b):
    m = np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    al, ah, bl, bh = a & m, a >> s, b & m, b >> s
    t = ah * bl + ((al * bl) >> s)
    u = al * bh + (t & m)
    return ah * bh + (t >> s) + (u >> s)


def _philox(c0, c1, key):
    """First word of Philox4x64-10 at counters (c0, c1, 0, 0), key (key, 0)."""
    M0, M1 = np.uint64(0xD2E7470EE14C6C93), np.uint64(0xCA5A826395121157)
    x = [c0.astype(np.uint64), np.full(c0.shape, c1, np.uint64), np.zeros(c0.shape, np.uint64), np.zeros(c0.shape, np.uint64)]
    k0, k1 = np.full(c0.shape, key, np.uint64), np.zeros(c0.shape, np.uint64)
    for _ in range(10):
        x = [_mulhi(M1, x[2]) ^ x[1] ^ k0, M1 * x[2], _mulhi(M0, x[0]) ^ x[3] ^ k1, M0 * x[0]]
        k0, k1 = k0 + np.uint64(0x9E3779B97F4A7C15), k1 + np.uint64(0xBB67AE8584CAA73B)
    return x[0]


class _Elements:
    """H_nm of every connected m of a sample, in the canonical order (singles by spin, same-spin doubles by spin,
    alpha-beta doubles; positions among the occupied / empty orbitals ascending, pairs lexicographic)."""

    def __init__(self, s, dev):
        self.K, self.dev = s.K, dev
        L = _t(s.chol, dev)
        self.h = _t(s.h1e, dev)
        self.g = torch.einsum("xpq,xrs->pqrs", L, L)
        r = torch.arange(s.K, device=dev)
        self.J = self.g[:, :, r, r]                      # (ai|pp)
        self.X = self.g[:, r, r, :].permute(0, 2, 1)     # (ap|pi) at [a][i][p]

    def of(self, occ):
        """occ [2K]: H_nn, then per connected m: emptied i, j and filled a, b (spin orbitals; -1 for a single's j, b), H."""
        dev, g = self.dev, self.g
        n = [occ[0::2].double(), occ[1::2].double()]
        o = [x.nonzero().squeeze(1) for x in n]
        v = [(x == 0).nonzero().squeeze(1) for x in n]
        tot = self.J @ (n[0] + n[1])
        F = [self.h + tot - self.X @ n[sp] for sp in (0, 1)]
        diag = sum(0.5 * (self.h.diagonal() + F[sp].diagonal()) @ n[sp] for sp in (0, 1))
        I, J, A, B, H = [], [], [], [], []

        def add(i, j, a, b, h):
            for to, x in ((I, i), (J, j), (A, a), (B, b), (H, h)):
                to.append(x.reshape(-1))

        for sp in (0, 1):
            i, a = torch.meshgrid(o[sp], v[sp], indexing="ij")
            none = torch.full_like(i, -1)
            add(2 * i + sp, none, 2 * a + sp, none, F[sp][a, i])
        for sp in (0, 1):
            po = torch.triu_indices(len(o[sp]), len(o[sp]), 1, device=dev)
            pv = torch.triu_indices(len(v[sp]), len(v[sp]), 1, device=dev)
            x, y = torch.meshgrid(torch.arange(po.shape[1], device=dev), torch.arange(pv.shape[1], device=dev), indexing="ij")
            i, j, a, b = o[sp][po[0][x]], o[sp][po[1][x]], v[sp][pv[0][y]], v[sp][pv[1][y]]
            add(2 * i + sp, 2 * j + sp, 2 * a + sp, 2 * b + sp, g[a, i, b, j] - g[a, j, b, i])
        i, a, j, b = torch.meshgrid(o[0], v[0], o[1], v[1], indexing="ij")
        add(2 * i, 2 * j + 1, 2 * a, 2 * b + 1, g[a, i, b, j])
        I, J, A, B, H = (torch.cat(x) for x in (I, J, A, B, H))
        below = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), occ.cumsum(0)])
        d = J >= 0
        odd = below[I] + below[A] - (I < A).long()
        odd = odd + torch.where(d, below[J] + below[B] - (I < J).long() - (I < B).long() - (J < B).long()
                                - (J < A).long() + (B < A).long(), torch.zeros_like(odd))
        return diag, I, J, A, B, torch.where(odd % 2 == 1, -H, H)


def _exact_energy(s):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    T, Wm, b = _t(s.tensors, dev), None, None
    if s.rbm_W is not None:
        Wm, b = _t(s.rbm_W, dev), _t(s.rbm_b, dev)
    el = _Elements(s, dev)
    occ = _t(_bits(s.samples, s.K), dev)
    ln, sn = _log_psi(s, occ, T, Wm, b)
    out = []
    for k in range(len(occ)):
        diag, I, J, A, B, H = el.of(occ[k])
        coef = torch.where(H.abs() >= s.eps, H, torch.zeros_like(H))
        use = H.abs() >= s.eps
        if s.n_draws:
            n_conn = len(H)
            shift = 62 - math.frexp(s.eps)[1] - n_conn.bit_length()
            w = np.where(use.cpu().numpy(), 0.0, np.ceil(np.ldexp(H.abs().cpu().numpy(), shift))).astype(np.uint64)
            pre = np.cumsum(w, dtype=np.uint64)
            if pre[-1]:
                x = _philox(np.arange(s.n_draws), k, s.seed)
                at = np.searchsorted(pre, _mulhi(x, np.full(x.shape, pre[-1])), side="right")
                u, mult = np.unique(at, return_counts=True)
                c = mult / s.n_draws * float(pre[-1]) / w[u].astype(np.float64)
                u = torch.as_tensor(u, device=dev)
                coef[u] = H[u] * torch.as_tensor(c, device=dev)
                use = use.clone()
                use[u] = True
        rows = use.nonzero().squeeze(1)
        m = occ[k][None].repeat(len(rows), 1)
        q = torch.arange(len(rows), device=dev)
        dbl = (J[rows] >= 0).nonzero().squeeze(1)
        m[q, I[rows]] = 0
        m[q, A[rows]] = 1
        m[q[dbl], J[rows][dbl]] = 0
        m[q[dbl], B[rows][dbl]] = 1
        lm, sm = _log_psi(s, m, T, Wm, b)
        out.append(diag + (coef[rows] * (lm - ln[k]).exp() * sm * sn[k]).sum())
    return torch.stack(out)


def _exact_vjp(s, u):
    """log|psi|, sign and sum_n u_n d log|psi(n)| / d (tensors, W, b)."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    p = [_t(x, dev).requires_grad_(True) for x in (s.tensors, s.rbm_W, s.rbm_b) if x is not None]
    la, sg = _log_psi(s, _t(_bits(s.samples, s.K), dev), *(p if len(p) == 3 else (p[0], None, None)))
    return la.detach(), sg.to(torch.int8), list(torch.autograd.grad(la, p, u.to(dev)))


def _exact_seconds(case):
    K, D = case["K"], case["D"]
    na, nb = _electrons(case)
    per = 2.0 * D * D * _edges(case) * (4 if case.get("readout") == "rnn" else 1)
    return case["samples"] * (_rows(K, na, nb, case["eps"], case["draws"]) * per / 4e11 + 1.5e-4 * K + 1e-3)


def exact(case, seed):
    if case["kind"] in ("sample", "batch") or (case["kind"] != "log_psi" and _exact_seconds(case) > 16):
        return None
    s = _system(case, seed)
    if case["kind"] == "log_psi":
        u = torch.from_numpy(np.random.default_rng([int(seed), 8]).normal(size=len(s.samples)))
        la, sg, g = _exact_vjp(s, u)
        return dict(log_abs=la, sign=None, grads=g)
    e = _exact_energy(s)
    c = _t(s.counts, e.device)
    mean = (c * e).sum() / c.sum()
    if case["kind"] == "energy":
        return dict(e_loc=e, e_mean=float(mean), n_amplitudes=None)
    _, _, g = _exact_vjp(s, 2 * c * (e - mean) / c.sum())
    g = [x.cpu().numpy() for x in g] + [None, None]
    return dict(sites=g[0], W=g[1], b=g[2], e_loc=e.cpu().numpy(), e_mean=float(mean))
