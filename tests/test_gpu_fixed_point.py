"""GPU parity of the forward's fixed-point path (csrc/fx.cuh): plans large enough to take it, at the
sizes and inputs where it can go wrong, against the oracle.  Tolerance as the forward's:
|C_gpu - C_oracle| <= 1e-11 * sum_ij |w_i w_j prod det|."""
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


def check(M, w, expect_refactors=None):
    plan = M.Plan.from_workload(w)
    S = [torch.from_numpy(np.ascontiguousarray(s)).cuda() for s in w.S]
    out = plan.correlator(S).cpu().numpy()
    again = plan.correlator(S).cpu().numpy()
    assert M.mhc_get_status_code(plan.handle) == M.MHC_OK
    assert out.tobytes() == again.tobytes()
    ref, scale = oracle.correlator(w.S, w.n_f, w.labels_src, w.w_src, w.labels_snk, w.w_snk, threads=8)
    assert abs(complex(*out) - ref) <= 1e-11 * scale, (complex(*out), ref, abs(complex(*out) - ref) / scale)
    plan.close()
    return w


def big(n, L, src, snk, seed, **kw):
    """About 60 source families against 63 warps of sinks, a ragged last one."""
    return wl.make_workload("fx", n, L, src, snk, seed=seed, **kw)


SINKS = [16] * 120 + [7, 1, 5, 2, 16, 31]


@pytest.mark.parametrize("n", [[1, 6], [2, 5], [3, 3], [5, 4], [6, 6], [7, 8], [9, 12], [18, 3], [17], [0, 6], [13, 18]])
def test_label_counts(M, n):
    L = [max(12 * ((x + 2) // 3) + 12, x + 16) for x in n]
    check(M, big(n, L, [1, 2, 3, 4, 5, 6, 9, 3] * 8, SINKS, seed=100 + sum(n), diag=3.0))


@pytest.mark.parametrize("two_row, forced", [(0.5, 0.0), (0.0, 0.05), (0.3, 0.05)])
def test_two_row_families_and_near_singular_members(M, two_row, forced):
    check(M, big([12, 10], [60, 48], [6, 3, 8, 5] * 16, SINKS, seed=7, two_row_frac=two_row, forced_frac=forced, twins=8))


def graded(w, rng, rows, cols):
    """Propagator rows and columns scaled by powers of two and ten over 10^+-rows, 10^+-cols."""
    w.S = [np.ascontiguousarray(s * 10.0 ** rng.uniform(-rows, rows, (s.shape[0], 1))
                                * 10.0 ** rng.uniform(-cols, cols, (1, s.shape[0]))) for s in w.S]
    return w


@pytest.mark.parametrize("rows, cols, diag", [(6, 0, 2.0), (0, 6, 2.0), (3, 3, 2.0), (0, 0, 1e6), (0, 0, 1e-3)])
def test_entries_of_very_different_sizes(M, rows, cols, diag):
    rng = np.random.default_rng(5)
    check(M, graded(big([6, 5], [48, 36], [4, 5, 6, 1] * 16, SINKS, seed=8, diag=diag), rng, rows, cols))


@pytest.mark.parametrize("spread", [1e3, 1e12])
def test_weights_of_very_different_sizes(M, spread):
    w = big([6, 6], [48, 48], [16, 3, 8, 5] * 16, SINKS, seed=9)
    rng = np.random.default_rng(6)
    w.w_src = w.w_src * spread ** rng.uniform(-1, 1, w.w_src.shape)
    w.w_src[::7] = 0.0
    check(M, w)


def test_complex_weights(M):
    """Complex weights in one pass: the four real-weight oracle sums of the bilinear form."""
    w = big([6, 4], [48, 36], [4, 5, 6, 1] * 16, SINKS, seed=12, forced_frac=0.05, twins=8)
    rng = np.random.default_rng(18)
    ws = w.w_src + 1j * rng.normal(size=w.w_src.shape)
    wk = w.w_snk + 1j * rng.normal(size=w.w_snk.shape)
    ws[3], ws[4], ws[5] = 1j, 2.0, 0.0
    plan = M.Plan.from_workload(w)
    S = [torch.from_numpy(s).cuda() for s in w.S]
    out = M.mhc_correlator_cw(plan.handle, S, torch.from_numpy(ws).cuda(), torch.from_numpy(wk).cuda())
    ref, scale = 0.0, 0.0
    for x, fx in ((ws.real, 1.0), (ws.imag, 1j)):
        for y, fy in ((wk.real, 1.0), (wk.imag, 1j)):
            c, s = oracle.correlator(w.S, w.n_f, w.labels_src, np.ascontiguousarray(x), w.labels_snk,
                                     np.ascontiguousarray(y), threads=8)
            ref, scale = ref + fx * fy * c, scale + s
    assert abs(complex(*out.cpu().numpy()) - ref) <= 1e-11 * scale
    assert M.mhc_get_status_code(plan.handle) == M.MHC_OK
    plan.close()


def test_structured_propagators(M):
    """Zeros, exactly repeated rows and labels, real entries: determinants that vanish exactly."""
    w = big([4, 3], [24, 24], [4, 5, 6, 1] * 16, SINKS, seed=10)
    w.S[0] = np.ascontiguousarray(np.diag(np.diag(w.S[0])))
    w.S[1][3] = w.S[1][5]
    w.S[1] = np.ascontiguousarray(w.S[1].real.astype(np.complex128))
    w.labels_src[5, 1] = w.labels_src[5, 0]
    check(M, w)


def test_nonfinite_input_is_reported(M):
    w = big([3, 3], [24, 24], [4, 5, 6, 1] * 16, SINKS, seed=11)
    w.S[0][int(w.labels_src[0, 0])] = np.inf
    plan = M.Plan.from_workload(w)
    plan.correlator([torch.from_numpy(s).cuda() for s in w.S])
    assert M.mhc_get_status_code(plan.handle) == M.MHC_ENONFINITE
    plan.close()
