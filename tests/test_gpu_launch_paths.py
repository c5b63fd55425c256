"""Launch paths that only certain sizes reach, against the oracle.

Over-improved Runge-Kutta stages above 786,432 sites (a launch per direction): one step of the
periodic 32^3x64 field, whose copies are equal bit for bit and match the oracle's step of one 8^4
period.  Simultaneous stout and APE sweeps and a Runge-Kutta step in one launch over every direction
on rows with unused positions (20, 24 and 28 sites), below and above the size at which three warps
share 32 links.  Tolerances as for the same comparisons elsewhere: 1e-6 for stout, 3e-6 for APE at
alpha = 0.02, 2e-6 for the flow."""

import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    from paper_2203_09764_gb300 import vs
    ctx = vs.vs_create(0)
    yield vs, ctx
    vs.vs_destroy(ctx)


@pytest.mark.parametrize("storage", [18, 12])
def test_over_improved_flow_of_a_large_field(env, storage):
    vs, ctx = env
    tile, reps = (8, 8, 8, 8), (4, 4, 4, 8)
    dims = tuple(t * r for t, r in zip(tile, reps))
    U0 = O.cool(tile, synth.haar_field(tile, 17), 1)
    big = np.tile(U0.reshape(4, *tile[::-1], 3, 3), (1, *reps[::-1], 1, 1)).reshape(4, -1, 3, 3)
    want = O.flow_rk3(tile, U0, 1, 0.02, eps=-0.25)
    f = vs.vs_field_create(ctx, dims, vs.VS_FP32, vs.VS_LINK12 if storage == 12 else vs.VS_LINK18)
    vs.vs_load_field(f, links=big)
    vs.vs_flow_rk3(f, 1, 0.02, -0.25, reunit_every=0)
    got = vs.vs_read_field(f).reshape(4, reps[3], 8, reps[2], 8, reps[1], 8, reps[0], 8, 3, 3)
    vs.vs_field_destroy(f)
    first = got[:, 0, :, 0, :, 0, :, 0]
    assert np.array_equal(got, np.broadcast_to(first[:, None, :, None, :, None, :, None], got.shape))
    assert np.abs(first.reshape(4, -1, 3, 3) - want).max() < 2e-6


@pytest.mark.parametrize("eps", [-0.25, 1.0])
@pytest.mark.parametrize("storage", [18, 12])
@pytest.mark.parametrize("dims", [(20, 4, 4, 8), (20, 12, 16, 16), (24, 8, 16, 16), (28, 12, 8, 16)])
def test_every_direction_at_once_on_padded_rows(env, dims, storage, eps):
    vs, ctx = env
    U0 = O.cool(dims, synth.haar_field(dims, 19), 1)
    f = vs.vs_field_create(ctx, dims, vs.VS_FP32, vs.VS_LINK12 if storage == 12 else vs.VS_LINK18)
    for gpu, cpu, tol in (
            (lambda: vs.vs_smooth(f, 1, 0.06, eps, vortex_preserve=False, reunit_every=0, kind=vs.VS_SIMULTANEOUS),
             lambda: O.smooth(dims, U0, None, 1, 0.06, eps=eps, vp=False, schedule=O.SIMULTANEOUS)[0], 1e-6),
            (lambda: vs.vs_smooth_ape(f, 1, 0.02, eps, schedule=vs.VS_SIMULTANEOUS, vortex_preserve=False,
                                      reunit_every=0),
             lambda: O.ape_ucp(dims, U0, None, 1, 0.02, eps=eps, schedule="simultaneous", vp=False)[0], 3e-6),
            (lambda: vs.vs_flow_rk3(f, 1, 0.02, eps, reunit_every=0),
             lambda: O.flow_rk3(dims, U0, 1, 0.02, eps=eps), 2e-6)):
        vs.vs_load_field(f, links=U0)
        gpu()
        assert np.abs(vs.vs_read_field(f) - cpu()).max() < tol
    vs.vs_field_destroy(f)


@pytest.mark.parametrize("dims", [(20, 12, 20, 32), (20, 16, 20, 40)])
def test_rows_of_20_in_order_and_in_whole_runs(env, dims):
    """38,400 links of a colour class, whose whole runs would add a layer of blocks over the SMs, and
    64,000, where they do not."""
    vs, ctx = env
    U0 = synth.haar_field(dims, 23)
    f = vs.vs_field_create(ctx, dims, vs.VS_FP32, vs.VS_LINK18)
    vs.vs_load_field(f, links=U0)
    vs.vs_smooth(f, 1, 0.06, -0.25, vortex_preserve=False, reunit_every=0)
    want, _ = O.smooth(dims, U0, None, 1, 0.06, eps=-0.25, vp=False)
    assert np.abs(vs.vs_read_field(f) - want).max() < 1e-6
    vs.vs_field_destroy(f)
