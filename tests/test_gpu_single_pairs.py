"""Single pairs through the forward: with every weight zero but one source's and one sink's, C is that
pair's determinant as the fixed-point or FP64 path forms it.  Against double-double determinants at the
per-pair tolerance of parity_util, 1e-12 of the value."""
import numpy as np
import pytest
import torch

import oracle
from paper_1411_3691_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_1411_3691_gb300 import build as B
    B.build()
    from paper_1411_3691_gb300 import mhc
    return mhc


SRC = [8, 5, 11, 7, 8, 9] * 16
SNK = [16] * 120 + [7, 1, 5, 2, 16, 31]


def make(n, seed, diag=2.0, **kw):
    L = [max(12 * ((x + 2) // 3) + 12, x + 16) for x in n]
    return wl.make_workload("pairs", n, L, SRC, SNK, seed=seed, diag=diag, **kw)


class Runner:
    """A plan and its propagators; C of chosen weights."""

    def __init__(self, M, w, **opts):
        o = M.default_opts()
        for k, v in opts.items():
            setattr(o, k, v)
        self.w, self.plan = w, M.Plan.from_workload(w, o)
        self.S = [torch.from_numpy(np.ascontiguousarray(s)).cuda() for s in w.S]

    def C(self, src, snk):
        """src, snk: {term: weight}, all others zero."""
        ws, wk = np.zeros(len(self.w.w_src)), np.zeros(len(self.w.w_snk))
        for x, pick in ((ws, src), (wk, snk)):
            for t, v in pick.items():
                x[t] = v
        out = self.plan.correlator(self.S, torch.from_numpy(ws).cuda(), torch.from_numpy(wk).cuda())
        return complex(*out.cpu().numpy())

    def all_dets(self, i):
        """|product of the flavours' determinants| of source i with every sink, from the oracle."""
        w, j = self.w, np.arange(len(self.w.w_snk))
        return np.abs(np.prod(oracle.pair_dets(w.S, w.n_f, w.labels_src, w.labels_snk, np.full(len(j), i), j, threads=8), axis=1))

    def exact(self, i, j):
        w, o, p = self.w, 0, 1.0
        for f, n in enumerate(w.n_f):
            hr, lr, hi, li = oracle.det_dd(w.S[f][np.ix_(w.labels_src[i, o:o + n], w.labels_snk[j, o:o + n])])
            p, o = p * complex(hr + lr, hi + li), o + n
        return p

    def tables(self):  # held, and used with these propagators
        self.C({}, {})
        return self.plan.forward_info()["tables_used"]


def families(run):
    """Work families as lists of source terms, the largest first."""
    fam = run.plan.families()
    terms = [list(fam["term"][a:b]) for a, b in zip(fam["offset"], fam["offset"][1:])]
    return sorted(terms, key=len, reverse=True)


@pytest.mark.parametrize("n", [[6, 5], [6], [12, 10]])
@pytest.mark.parametrize("binades", [0, 5, 8, 9, 12, 30])
def test_beside_a_heavy_member_that_vanishes(M, n, binades):
    """A member with a weight 2^binades above the others' of its family, whose changed row is zero in a
    sink's columns: the others' values keep their bits.  The smallest values of a family's pairs."""
    w = make(n, 40 + sum(n))
    first = Runner(M, w)
    picks = []
    for terms in families(first)[:4]:
        heavy, i = terms[1], terms[2]
        own = set(w.labels_src[heavy, :n[0]]) - set(w.labels_src[i, :n[0]])  # heavy's changed label
        assert len(own) == 1
        for j in np.argsort(first.all_dets(i))[:4]:
            picks.append((heavy, i, j, own.pop() if own else picks[-1][3]))
    first.plan.close()
    for heavy, i, j, label in picks:
        w.S[0][label, w.labels_snk[j, :n[0]]] = 0.0
    run = Runner(M, w)
    assert run.tables() == 1
    for heavy, i, j, _ in picks:
        ref = run.exact(i, j)
        if abs(ref) == 0.0:  # the family's shared rows hold another pick's label
            continue
        got = run.C({heavy: 2.0 ** binades, i: 1.0}, {j: 1.0})
        assert abs(got - ref) <= 1e-12 * abs(ref), (heavy, i, j, got, ref)
    run.plan.close()


@pytest.mark.parametrize("n", [[6, 5], [12, 10]])
def test_weights_over_many_decades(M, n):
    """Weights of 10^-12 to 10^12 and zeros within a family, complex ones too: the sum of the pairs."""
    w = make(n, 50 + sum(n))
    run = Runner(M, w)
    rng = np.random.default_rng(3)
    for terms in families(run)[:3]:
        j = int(rng.integers(len(w.w_snk)))
        dets = {t: run.exact(t, j) for t in terms}
        wt = {t: 0.0 if k % 4 == 3 else float(rng.normal() * 10.0 ** rng.uniform(-12, 12)) for k, t in enumerate(terms)}
        ref = sum(wt[t] * dets[t] for t in terms)
        scale = sum(abs(wt[t] * dets[t]) for t in terms)
        assert abs(run.C(wt, {j: 1.0}) - ref) <= 1e-12 * scale
        ws, wk = np.zeros(len(w.w_src), complex), np.zeros(len(w.w_snk), complex)
        for t in terms:
            ws[t] = wt[t] * (0.6 + 0.8j)
        wk[j] = 0.8 - 0.6j
        out = M.mhc_correlator_cw(run.plan.handle, run.S, torch.from_numpy(ws).cuda(), torch.from_numpy(wk).cuda())
        assert abs(complex(*out.cpu().numpy()) - ref * (0.6 + 0.8j) * (0.8 - 0.6j)) <= 1e-12 * scale
    run.plan.close()


def test_zero_weights_pass_the_guards(M):
    """Zero weights add nothing and leave the refactor counts as they are."""
    w = make([12, 10], 61, two_row_frac=0.3, forced_frac=0.05, twins=8)
    run = Runner(M, w)
    full = torch.from_numpy(w.w_src).cuda()
    run.plan.correlator(run.S, full)
    run.plan.status()
    before = run.plan.stats()
    assert before["refactor_child"] > 0 and run.tables() == 1
    run.plan.status()
    assert run.plan.correlator(run.S, torch.zeros_like(full)).abs().max().item() == 0.0
    run.plan.status()
    after = run.plan.stats()
    assert after["refactor_child"] == before["refactor_child"] and after["refactor_parent"] == before["refactor_parent"]
    run.plan.close()


@pytest.mark.parametrize("tau_child", [1e-3, 0.0])
@pytest.mark.parametrize("n", [[6, 5], [18], [12, 10]])
def test_smallest_values(M, n, tau_child):
    """The smallest of a source's determinants, also with no lemma guard behind the accuracy floor."""
    run = Runner(M, make(n, 70 + sum(n)), tau_child=tau_child)
    assert run.tables() == 1
    for terms in families(run)[::24]:
        for j in np.argsort(run.all_dets(terms[0]))[:4]:
            ref = run.exact(terms[0], j)
            assert abs(run.C({terms[0]: 1.0}, {j: 1.0}) - ref) <= 1e-12 * abs(ref)
    run.plan.close()


def scaled(w, pattern, spread, seed=4):
    """Propagators with rows, columns or both scaled by powers of two over 2^spread, or entries by
    2^-spread per step between 12-label sites."""
    rng = np.random.default_rng(seed)
    out = []
    for s in w.S:
        L = s.shape[0]
        r, c = (np.exp2(rng.integers(0, spread + 1, L)) for _ in range(2))
        site = np.arange(L) // 12
        f = {"rows": r[:, None], "cols": c[None, :], "both": r[:, None] * c[None, :],
             "decay": np.exp2(-float(spread) * np.abs(site[:, None] - site[None, :]))}[pattern]
        out.append(np.ascontiguousarray(s * f))
    w.S = out
    return w


@pytest.mark.parametrize("tau", [1e-4, 1e-9, 1e-12])
@pytest.mark.parametrize("pattern, spread", [("rows", 5), ("rows", 10), ("rows", 39), ("cols", 5), ("cols", 12), ("both", 8),
                                             ("decay", 2)])
@pytest.mark.parametrize("n", [[6, 5], [12, 10]])
def test_propagators_that_are_not_flat(M, n, pattern, spread, tau):
    """Rows, columns and entries of very different sizes, with pivot guards down to 1e-12: the call takes
    the FP64 path, though the plan has tables, and keeps its accuracy."""
    run = Runner(M, scaled(make(n, 80 + sum(n)), pattern, spread), tau_parent=tau)
    run.C({}, {})
    info = run.plan.forward_info()
    assert info["tables"] == 1 and info["tables_used"] == 0
    rng = np.random.default_rng(9)
    for _ in range(25):
        i, j = int(rng.integers(len(run.w.w_src))), int(rng.integers(len(run.w.w_snk)))
        ref = run.exact(i, j)
        assert abs(run.C({i: 1.0}, {j: 1.0}) - ref) <= 1e-12 * abs(ref)
    run.plan.close()


@pytest.mark.parametrize("n", [[6, 5], [12, 10]])
def test_labels_that_no_term_has(M, n):
    """Large entries, infinities and zeros in rows and columns that no term uses leave the call on the
    fixed-point path, as accurate as without them."""
    w = make(n, 90 + sum(n))
    rng = np.random.default_rng(10)
    for f, s in enumerate(w.S):
        L = s.shape[0]
        big = np.zeros((L + 9, L + 9), complex)
        big[:L, :L] = s
        big[:L, L:L + 3] = 2.0 ** 25 * rng.normal(size=(L, 3))
        big[L:L + 3, :L] = 2.0 ** -25 * rng.normal(size=(3, L))
        big[L + 3:L + 6, :], big[:, L + 3:L + 6] = np.inf, np.nan
        w.S[f] = big
    run = Runner(M, w)
    run.C({}, {})
    assert run.plan.forward_info()["tables_used"] == 1
    for i in rng.integers(len(w.w_src), size=3):
        for j in np.argsort(run.all_dets(i))[:4]:
            ref = run.exact(i, j)
            assert abs(run.C({i: 1.0}, {j: 1.0}) - ref) <= 1e-12 * abs(ref)
    run.plan.close()
