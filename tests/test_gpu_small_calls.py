"""GPU parity of calls too small for tables of their own: the partials summed by the forward kernel's
last block or by a launch of their own, complex weights, and batches that give small plans tables.
Tolerance as the forward's: |C_gpu - C_oracle| <= 1e-11 * sum_ij |w_i w_j prod det|."""
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


def small(n, seed, src=60, snk=80, **kw):
    """src families of six against 8 snk + 3 sinks."""
    L = [max(12 * ((x + 2) // 3) + 12, x + 16) for x in n]
    return wl.make_workload("small", n, L, [6] * src, [8] * snk + [3], seed=seed, diag=3.0, **kw)


def reference(w, ws=None, wk=None):
    return oracle.correlator(w.S, w.n_f, w.labels_src, w.w_src if ws is None else np.ascontiguousarray(ws),
                             w.labels_snk, w.w_snk if wk is None else np.ascontiguousarray(wk), threads=8)


@pytest.mark.parametrize("tile, src, snk", [(32, 60, 80), (64, 60, 80), (128, 60, 80), (32, 1, 1), (128, 1, 1)])
def test_partial_sums(M, tile, src, snk):
    """60 families: 21 tiles of 32 sinks each are more than 16 per thread, 11 of 64 are not."""
    w = small([3, 3], 3, src, snk)
    opts = M.default_opts()
    opts.sink_tile = tile
    plan = M.Plan.from_workload(w, opts)
    S = [torch.from_numpy(s).cuda() for s in w.S]
    ref, scale = reference(w)
    outs = [plan.correlator(S).cpu().numpy() for _ in range(3)]
    assert abs(complex(*outs[0]) - ref) <= 1e-11 * scale
    assert all(o.tobytes() == outs[0].tobytes() for o in outs)
    assert M.mhc_get_status_code(plan.handle) == M.MHC_OK
    plan.close()


@pytest.mark.parametrize("n", [[3, 3], [12, 9], [20, 2]])
def test_complex_weights(M, n):
    w = small(n, 4, 12, 9, two_row_frac=0.3 if max(n) > 9 else 0.0)
    rng = np.random.default_rng(19)
    ws = w.w_src + 1j * rng.normal(size=w.w_src.shape)
    wk = w.w_snk + 1j * rng.normal(size=w.w_snk.shape)
    plan = M.Plan.from_workload(w)
    S = [torch.from_numpy(s).cuda() for s in w.S]
    out = M.mhc_correlator_cw(plan.handle, S, torch.from_numpy(ws).cuda(), torch.from_numpy(wk).cuda())
    ref, scale = 0.0, 0.0
    for x, fx in ((ws.real, 1.0), (ws.imag, 1j)):
        for y, fy in ((wk.real, 1.0), (wk.imag, 1j)):
            c, s = reference(w, x, y)
            ref, scale = ref + fx * fy * c, scale + s
    assert abs(complex(*out.cpu().numpy()) - ref) <= 1e-11 * scale
    plan.close()


def test_batch_of_small_plans(M):
    """One plan four times with propagators of its own and two others: 6 x 1260 warps of work."""
    ws = [small([5, 4], 5)] * 4 + [small([9, 10], 6, two_row_frac=0.3), small([2, 6], 7)]
    one = M.Plan.from_workload(ws[0])
    plans = [one] * 4 + [M.Plan.from_workload(w) for w in ws[4:]]
    host = [[np.ascontiguousarray(s * (1.0 + 0.25 * k)) for s in w.S] for k, w in enumerate(ws)]
    S = [[torch.from_numpy(s).cuda() for s in Sk] for Sk in host]
    outs = [torch.empty(2, dtype=torch.float64, device="cuda") for _ in ws]
    batch = M.mhc_batch_create([p.handle for p in plans])
    M.mhc_batch_correlator(batch, S, outs)
    torch.cuda.synchronize()
    for k, w in enumerate(ws):
        ref, scale = oracle.correlator(host[k], w.n_f, w.labels_src, w.w_src, w.labels_snk, w.w_snk, threads=8)
        assert abs(complex(*outs[k].cpu().numpy()) - ref) <= 1e-11 * scale, k
        plain = complex(*plans[k].correlator(S[k]).cpu().numpy())  # no tables in the plan itself
        assert abs(plain - ref) <= 1e-11 * scale, k
    M.mhc_batch_destroy(batch)
    for p in [one] + plans[4:]:
        p.close()
