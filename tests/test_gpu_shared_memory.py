"""Plans whose y cache fills most of a block's shared memory (232 448 bytes): a launch without
fixed-point tables needs the cache and the refactor scratch alone.  Oracle and tolerance of
test_gpu_forward.  Bytes of cache and scratch per block: 6 x n = 32 at tile 32 207 248, 3 x n = 14 at
tile 128 208 448, n = 22, 22 at tile 128 214 592, 8 x n = 12 at tile 64 219 936."""
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


@pytest.mark.parametrize("n, tile", [([32] * 6, 32), ([14] * 3, 128), ([22] * 2, 128), ([12] * 8, 64)])
def test_two_rows_in_every_flavour(M, n, tile):
    L = [max(12 * ((x + 2) // 3) + 12, x + 16) for x in n]
    w = wl.make_workload("smem", n, L, [3, 2], [5, 1, 4], seed=70 + len(n), diag=3.0, two_row_frac=1.0)
    opts = M.default_opts()
    opts.sink_tile = tile
    plan = M.Plan.from_workload(w, opts)
    assert (plan.families()["rank"] == 2).all(axis=1).any()  # the widest layout occurs
    out = plan.correlator([torch.from_numpy(s).cuda() for s in w.S]).cpu().numpy()
    assert M.mhc_get_status_code(plan.handle) == M.MHC_OK
    assert plan.forward_info()["tables"] == 0
    ref, scale = oracle.correlator(w.S, w.n_f, w.labels_src, w.w_src, w.labels_snk, w.w_snk, threads=8)
    assert abs(complex(*out) - ref) <= 1e-11 * scale
    plan.close()
