"""A plan given many times in one batch: its later entries' fixed-point tables stay within 4 GiB together,
and the entries beyond take the FP64 path.  Oracle and tolerance of test_gpu_batch."""
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


def test_repeated_plan_beyond_the_limit(M):
    count = 48
    w = wl.make_workload("rep", [6, 5], [1024, 1024], [8] * 512, [16] * 15 + [9], seed=31)
    plan = M.Plan.from_workload(w)
    S = [torch.from_numpy(s).cuda() for s in w.S]
    plan.correlator(S)
    info = plan.forward_info()
    assert info["tables"] == 1 and (count - 1) * info["table_bytes"] > 1.2 * 2 ** 32
    torch.cuda.synchronize()
    outs = [torch.empty(2, dtype=torch.float64, device="cuda") for _ in range(count)]
    free = torch.cuda.mem_get_info()[0]
    batch = M.mhc_batch_create([plan.handle] * count)
    M.mhc_batch_correlator(batch, [S] * count, outs)
    torch.cuda.synchronize()
    st = plan.stats()
    factors = st["families"] * st["sink_families"] * 16 * (25 + 5 + 2 + 16 + 4 + 2)  # each entry's block factors
    assert free - torch.cuda.mem_get_info()[0] <= 2 ** 32 + count * factors + 2 ** 29
    ref, scale = oracle.correlator(w.S, w.n_f, w.labels_src, w.w_src, w.labels_snk, w.w_snk, threads=8)
    for o in outs:
        assert abs(complex(*o.cpu().numpy()) - ref) <= 1e-11 * scale
    M.mhc_batch_destroy(batch)
    plan.close()
