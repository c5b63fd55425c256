"""Device blocks of finished jobs serve the next jobs: within the admission budget, with the
results of fresh memory, and given back when the loop is idle."""

import time

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

SHAPES = [(16, 16, 16, 32), (8, 8, 8, 8), (12, 12, 12, 24), (16, 16, 16, 32), (20, 4, 8, 8), (12, 12, 12, 24),
          (16, 16, 16, 32), (8, 8, 8, 8)]


@pytest.mark.parametrize("budget", [0, 60 << 20])
def test_blocks_are_reused_and_given_back(budget):
    import torch
    from paper_2203_09764_gb300 import vs
    ctx = vs.vs_create(0, hbm_budget_bytes=budget, max_slots=3)
    vs.vs_poll(ctx, vs.vs_submit(ctx, vs.make_job((4, 4, 4, 4), 0.05, 10, n_cool=1)))
    time.sleep(0.5)
    free = torch.cuda.mem_get_info()[0]
    jobs = []
    for turn in range(2):
        for k, dims in enumerate(SHAPES):
            out = np.empty((4, int(np.prod(dims)), 3, 3), dtype=np.complex128) if np.prod(dims) <= 8 ** 4 else None
            jobs.append(vs.make_job(dims, 0.06, 12, labels=synth.iid_labels(dims, 60 + k), links_out=out))
    tickets = [vs.vs_submit(ctx, j) for j in jobs]
    res = [vs.vs_poll(ctx, t) for t in tickets]
    assert all(r["status"] == vs.VS_OK and r["n_label_diff"] == 0 for r in res)
    # the same job in reused memory: the same bits
    for k in range(len(SHAPES)):
        a, b = res[k], res[k + len(SHAPES)]
        assert a["action"] == b["action"] and a["n_reject"] == b["n_reject"]
    if budget:
        assert vs.vs_serve_stats_get(ctx)["peak_bytes_in_use"] <= budget
    time.sleep(1.0)
    # what stays is graphs and streams, no field (a 16^3x32 field is 38 MB)
    assert torch.cuda.mem_get_info()[0] > free - (30 << 20)
    vs.vs_destroy(ctx)
