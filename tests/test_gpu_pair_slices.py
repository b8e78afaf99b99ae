"""Per-pair determinants of more pairs than one launch takes (2^22): the last of a slice, the first of the
next, the very last and a bad index beyond, against the oracle at parity_util's tolerance."""
import numpy as np
import pytest
import torch

import oracle
from paper_1411_3691_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def test_slices():
    from paper_1411_3691_gb300 import build as B
    B.build()
    from paper_1411_3691_gb300 import mhc as M
    w = wl.make_workload("slices", [7, 3], [48, 24], [6, 5, 4], [8, 3, 7], seed=12, diag=3.0)
    plan = M.Plan.from_workload(w)
    S = [torch.from_numpy(s).cuda() for s in w.S]
    n = (1 << 23) + 37
    rng = np.random.default_rng(2)
    ii, jj = rng.integers(0, len(w.w_src), n), rng.integers(0, len(w.w_snk), n)
    path = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    got = plan.pair_dets(S, torch.from_numpy(ii).cuda(), torch.from_numpy(jj).cuda(), path)
    assert M.mhc_get_status_code(plan.handle) == M.MHC_OK
    at = np.unique(np.concatenate([rng.integers(0, n, 400)] + [np.clip(np.arange(-40, 40) + (k << 22), 0, n - 1) for k in range(3)] + [[n - 1]]))
    ref = oracle.pair_dets(w.S, w.n_f, w.labels_src, w.labels_snk, ii[at], jj[at], threads=8)
    assert (np.abs(got.cpu().numpy()[at] - ref) <= 1e-12 * np.abs(ref)).all()
    # the same pair has the same bits and path everywhere
    pair = torch.from_numpy(ii * len(w.w_snk) + jj).cuda()
    first = torch.full((len(w.w_src) * len(w.w_snk),), n, dtype=torch.int64, device="cuda")
    first.scatter_reduce_(0, pair, torch.arange(n, device="cuda"), "amin")
    assert torch.equal(got, got[first[pair]]) and torch.equal(path, path[first[pair]]) and int(path.min()) >= 0
    ii[-1] = len(w.w_src)
    plan.pair_dets(S, torch.from_numpy(ii).cuda(), torch.from_numpy(jj).cuda(), path)
    assert M.mhc_get_status_code(plan.handle) == M.MHC_EINVAL
    plan.close()
