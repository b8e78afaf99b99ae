"""What the fixed-point forward (csrc/fx.cuh) does on the inputs it treats apart, in plans that hold
its tables (asserted): an empty first flavour, determinants that vanish exactly, repeated labels,
non-finite entries.  Against the oracle, |C_gpu - C_oracle| <= 1e-11 * sum_ij |w_i w_j prod det| as the
forward's tests, and against the FP64 path of the same terms (a one-sided plan): both are sums of
determinants good to a few n u of their own size, so 2e-14 of the same sum (n <= 12, u = 1.1e-16)."""
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
    return wl.make_workload("path", n, L, SRC, SNK, seed=seed, diag=diag, **kw)


def run(M, w, tables, one_sided=0, flat=True):
    """The plan's C; tables: whether it has to hold the fixed-point tables; flat: and to use them."""
    opts = M.default_opts()
    opts.one_sided = one_sided
    plan = M.Plan.from_workload(w, opts)
    S = [torch.from_numpy(np.ascontiguousarray(s)).cuda() for s in w.S]
    out = plan.correlator(S).cpu().numpy()
    info = plan.forward_info()
    assert info["tables"] == int(tables) and info["tables_used"] == int(tables and flat), info
    code = M.mhc_get_status_code(plan.handle)
    plan.close()
    return out, code


def check(M, w):
    out, code = run(M, w, True)
    fp64, _ = run(M, w, False, one_sided=1)
    ref, scale = oracle.correlator(w.S, w.n_f, w.labels_src, w.w_src, w.labels_snk, w.w_snk, threads=8)
    assert code == M.MHC_OK
    assert abs(complex(*out) - ref) <= 1e-11 * scale
    assert abs(complex(*out) - complex(*fp64)) <= 2e-14 * scale, (complex(*out), complex(*fp64), scale)


@pytest.mark.parametrize("n", [[3, 3], [0, 6], [6], [4, 5], [2, 7], [12, 10]])
def test_label_counts(M, n):
    check(M, make(n, 100 + sum(n)))


def test_exactly_vanishing_determinants(M):
    """A propagator row that repeats another: every pair whose term holds both labels is 0."""
    w = make([4, 5], 21)
    for s in w.S:
        s[3] = s[5]
        s[:, 7] = s[:, 2]
    check(M, w)


def test_repeated_labels_and_real_entries(M):
    w = make([5, 4], 22)
    w.S[1] = np.ascontiguousarray(w.S[1].real.astype(np.complex128))
    w.labels_src[5, 1] = w.labels_src[5, 0]
    w.labels_snk[9, 6] = w.labels_snk[9, 7]
    check(M, w)


def test_forward_info(M):
    w = make([4, 5], 23)
    plan = M.Plan.from_workload(w)
    with pytest.raises(M.MHCError):
        plan.forward_info()
    plan.correlator([torch.from_numpy(s).cuda() for s in w.S])
    info = plan.forward_info()
    assert info["tables"] == 1 and info["table_bytes"] > 2 * 16 * sum(s.size for s in w.S)
    # tables, block factors (n <= 6), the forward and, with 16 partials per thread and more, the sum
    items = len(plan.families()["rank"]) * ((len(w.w_snk) + 127) // 128)
    assert info["folded_sum"] == int(items <= 16 * 128) and info["launches"] == 4 - info["folded_sum"]
    plan.close()


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_nonfinite_entries_are_reported(M, value):
    w = make([4, 4], 24)
    w.S[0][int(w.labels_src[0, 0])] = value
    _, code = run(M, w, True, flat=False)
    assert code == M.MHC_ENONFINITE
