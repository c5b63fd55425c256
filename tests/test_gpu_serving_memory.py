"""Device memory that the serving loop holds, running jobs and kept blocks together, as the driver
counts it right after a job (kept blocks are freed 100 ms later): within a job's footprint after a job
that came with labels and took its links out, and within the cap, or without one within what jobs have
taken at a time and at least 1 GiB, when jobs of another shape follow."""

import time

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

MIB = 1 << 20
ROUNDING = 4 * MIB      # cudaMalloc hands out 2 MiB pieces; the scalars and the list of a field share one


def _free():
    import torch
    return torch.cuda.mem_get_info()[0]


def test_staging_is_within_the_footprint():
    from paper_2203_09764_gb300 import vs
    dims = (32, 32, 32, 64)          # labels 8 MiB, links out 1152 MiB
    lab = synth.iid_labels((8, 8, 8, 8), 3).reshape(4, 8, 8, 8, 8)
    lab = np.ascontiguousarray(np.tile(lab, (1, 8, 4, 4, 4))).reshape(4, -1)
    out = np.empty((4, int(np.prod(dims)), 3, 3), dtype=np.complex128)
    ctx = vs.vs_create(0)
    job = vs.make_job(dims, 0.06, 1, labels=lab, links_out=out)
    assert vs.vs_poll(ctx, vs.vs_submit(ctx, job))["status"] == vs.VS_OK
    footprint = vs.vs_serve_stats_get(ctx)["peak_bytes_in_use"]
    held = []
    for _ in range(3):
        time.sleep(0.6)
        before = _free()
        vs.vs_poll(ctx, vs.vs_submit(ctx, job))
        held.append(before - _free())
    vs.vs_destroy(ctx)
    assert max(held) > footprint - ROUNDING         # seen before the blocks were freed
    assert max(held) <= footprint + ROUNDING


@pytest.mark.parametrize("budget", [0, 900 * MIB])
def test_jobs_of_another_shape_replace_kept_blocks(budget):
    from paper_2203_09764_gb300 import vs
    ctx = vs.vs_create(0, hbm_budget_bytes=budget, max_slots=2)
    small = vs.make_job((32, 32, 32, 32), 0.06, 60, seed=1, n_cool=0)     # 300 MiB
    large = vs.make_job((32, 32, 32, 64), 0.06, 1, seed=2, n_cool=0)      # 600 MiB

    def both():
        tickets = [vs.vs_submit(ctx, small), vs.vs_submit(ctx, small)]
        assert all(vs.vs_poll(ctx, t)["status"] == vs.VS_OK for t in tickets)

    both()
    vs.vs_poll(ctx, vs.vs_submit(ctx, large))
    held = []
    for _ in range(3):
        time.sleep(0.6)
        before = _free()
        both()
        vs.vs_poll(ctx, vs.vs_submit(ctx, large))
        held.append(before - _free())
    peak = vs.vs_serve_stats_get(ctx)["peak_bytes_in_use"]
    vs.vs_destroy(ctx)
    assert max(held) > 600 * MIB                     # seen before the blocks were freed
    assert max(held) <= (budget or max(peak, 1 << 30)) + 2 * ROUNDING
