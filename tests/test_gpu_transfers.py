"""Copies of caller-side FP64 matrices in and out of a field (links, gauge, read-back): exact
conversions, from pointers aligned to one double only, on padded and ragged lattices."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    from paper_2203_09764_gb300 import vs
    ctx = vs.vs_create(0)
    yield vs, ctx
    vs.vs_destroy(ctx)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (20, 4, 12, 8), (12, 8, 4, 20)])
def test_links_in_and_out_of_device_buffers(env, dims, offset):
    import torch
    vs, ctx = env
    V = int(np.prod(dims))
    U = synth.haar_field(dims, 5)
    flat = torch.zeros(4 * V * 18 + 1, dtype=torch.float64, device="cuda")
    src = flat[offset:offset + 4 * V * 18]
    src.copy_(torch.from_numpy(np.ascontiguousarray(U).view(np.float64).reshape(-1)))
    for prec, storage in ((vs.VS_FP64, vs.VS_LINK18), (vs.VS_FP32, vs.VS_LINK18), (vs.VS_FP32, vs.VS_LINK12)):
        f = vs.vs_field_create(ctx, dims, prec, storage)
        torch.cuda.synchronize()
        vs.vs_load_field(f, links=src)
        back = torch.zeros(4 * V * 18 + 1, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        vs.vs_read_field(f, back[offset:offset + 4 * V * 18])
        vs.vs_synchronize(f)
        got = back[offset:offset + 4 * V * 18].cpu().numpy().reshape(4, V, 9, 2)
        assert back[0 if offset else -1].item() == 0.0      # the double beside the buffer
        want = U.view(np.float64).reshape(4, V, 9, 2)
        want = want if prec == vs.VS_FP64 else want.astype(np.float32).astype(np.float64)
        rows = 6 if storage == vs.VS_LINK12 else 9
        assert np.array_equal(got[:, :, :rows], want[:, :, :rows])
        # the reference labels are the sectors of the FP64 input's traces
        t = np.trace(U, axis1=2, axis2=3)
        lab = np.where(np.abs(np.angle(t)) < np.pi / 3, 0, np.sign(np.angle(t))).astype(np.int8)
        assert np.array_equal(vs.vs_read_labels(f), lab)
        vs.vs_field_destroy(f)
