"""FP32 smoothers on both sides of the size at which a class launch changes from three warps per
32 links to a thread per link: one sweep of a general SU(3) field against the oracle.

Links per class launch (the flow: sites per stage launch, four times as many): 512, 12,288 (the
last plaquette-staple launch of three warps), 16,384, 28,672 (the last over-improved one),
32,768, 36,864, and 35,840 in rows of 20 (warps of six runs of five sites, the last one partial).  Tolerances are those of the same one-sweep comparisons on small lattices: 1e-6 for stout,
3e-6 for UCP and the flow (2e-6) and for AUS in 12-real storage, which rebuilds row 2 on each load."""

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


@pytest.mark.parametrize("eps", [-0.25, 1.0])
@pytest.mark.parametrize("storage", [18, 12])
@pytest.mark.parametrize("dims", [(8, 4, 8, 8), (16, 16, 16, 12), (16, 16, 16, 16), (16, 16, 16, 28), (16, 16, 16, 32),
                                  (16, 16, 16, 36), (20, 16, 16, 28)])
def test_one_sweep_on_both_sides_of_the_split(env, dims, storage, eps):
    vs, ctx = env
    U0 = O.cool(dims, synth.haar_field(dims, 3), 1)
    f = vs.vs_field_create(ctx, dims, vs.VS_FP32, vs.VS_LINK12 if storage == 12 else vs.VS_LINK18)
    runs = [
        (lambda: vs.vs_smooth(f, 1, 0.06, eps, vortex_preserve=False, reunit_every=0),
         lambda: O.smooth(dims, U0, None, 1, 0.06, eps=eps, vp=False)[0], 1e-6),
        (lambda: vs.vs_smooth_aus(f, 1, 0.02, eps, vortex_preserve=False, reunit_every=0),
         lambda: O.aus(dims, U0, None, 1, 0.02, eps=eps, vp=False)[0], 2e-6),
        (lambda: vs.vs_smooth_ape(f, 1, 0.02, eps, vortex_preserve=False, reunit_every=0),
         lambda: O.ape_ucp(dims, U0, None, 1, 0.02, eps=eps, vp=False)[0], 3e-6),
    ]
    if int(np.prod(dims)) <= 16 ** 4:
        runs.append((lambda: vs.vs_flow_rk3(f, 1, 0.02, eps, reunit_every=0),
                     lambda: O.flow_rk3(dims, U0, 1, 0.02, eps=eps), 2e-6))
    for gpu, cpu, tol in runs:
        vs.vs_load_field(f, links=U0)
        gpu()
        assert np.abs(vs.vs_read_field(f) - cpu()).max() < tol
    vs.vs_field_destroy(f)


@pytest.mark.parametrize("eps", [-0.25, 1.0])
@pytest.mark.parametrize("storage", [18, 12])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (4, 12, 20, 16), (8, 12, 16, 16)])
def test_every_direction_in_one_launch(env, dims, storage, eps):
    """Simultaneous stout and APE sweeps and a Runge-Kutta step where one launch takes every
    direction: 256 sites (three warps per 32 links), 15,360 (120 blocks per direction, a group of
    114 and one of 6) and 24,576 (114 and 78).  Tolerances as above; APE at alpha = 0.02 as UCP."""
    vs, ctx = env
    U0 = O.cool(dims, synth.haar_field(dims, 9), 1)
    lab = synth.iid_labels(dims, 4)
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
    # vortex preservation: a rejected link is written with its old value
    vs.vs_load_field(f, labels=lab)
    vs.vs_centrifuge(f, 0.02, 3)
    rho = 0.35 if eps != 1.0 else 0.75
    st = vs.vs_smooth(f, 1, rho, eps, reunit_every=0, kind=vs.VS_SIMULTANEOUS, stats=True)
    want, rej = O.smooth(dims, O.centrifuge(dims, lab, 0.02, 3), lab, 1, rho, eps=eps, vp=True,
                         schedule=O.SIMULTANEOUS)
    split = np.abs(vs.vs_read_field(f) - want).max(axis=(2, 3)) > 1e-4
    assert int(split.sum()) <= st[0]["n_undecidable"] and abs(st[0]["n_reject"] - int(rej[0])) <= st[0]["n_undecidable"]
    vs.vs_field_destroy(f)
