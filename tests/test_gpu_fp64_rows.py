"""FP64 stout class launches of every block kind (42 links per block, 21, 7, and whole layers with
a remainder), annealed and simultaneous, against the oracle on general SU(3) fields and with
vortex preservation.

Tolerance: a candidate is a sum of 24 products of up to 6 unitary matrices times rho, then two
products: ~100 roundings of 1.1e-16 on entries of size 1 per update, and one sweep passes an error
on at most a few times.  1e-12 leaves a factor of ten."""

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


# links per class launch: 64, 320, 2560 (21-link blocks), 3456, 10368 (one layer and a remainder), 32768
@pytest.mark.parametrize("eps", [-0.25, 1.0])
@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (4, 20, 4, 4), (8, 8, 8, 20), (12, 12, 8, 12), (12, 12, 12, 24),
                                  (16, 16, 16, 32)])
def test_one_sweep_matches_the_oracle(env, dims, eps):
    vs, ctx = env
    V = int(np.prod(dims))
    lab = synth.iid_labels(dims, 11)
    U0 = synth.haar_field(dims, 7)
    Uc = O.centrifuge(dims, lab, 0.02, 3)
    f = vs.vs_field_create(ctx, dims, vs.VS_FP64, vs.VS_LINK18)
    for kind, okind in ((vs.VS_ANNEALED, O.ANNEALED), (vs.VS_SIMULTANEOUS, O.SIMULTANEOUS)):
        vs.vs_load_field(f, links=U0)
        st = vs.vs_smooth(f, 1, 0.06, eps, kind=kind, vortex_preserve=False, stats=True)
        want, _ = O.smooth(dims, U0, lab, 1, 0.06, eps=eps, vp=False, schedule=okind)
        assert np.abs(vs.vs_read_field(f) - want).max() < 1e-12
        assert st[0]["n_accept"] == 4 * V
        vs.vs_load_field(f, labels=lab)
        vs.vs_centrifuge(f, 0.02, 3)
        st = vs.vs_smooth(f, 1, 0.06, eps, kind=kind, vortex_preserve=True, stats=True)
        want, rej = O.smooth(dims, Uc, lab, 1, 0.06, eps=eps, vp=True, schedule=okind)
        assert np.abs(vs.vs_read_field(f) - want).max() < 1e-12
        assert st[0]["n_reject"] == int(rej[0])
    vs.vs_field_destroy(f)
