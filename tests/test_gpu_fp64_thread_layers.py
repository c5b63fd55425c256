"""FP64 stout launches that take a thread per link: colour classes of 16,384 links (both staples) and
of 36,864 (the last layer of blocks nearly full), and a simultaneous sweep, against the oracle.
Tolerance as for the row kernels: ~100 roundings of 1.1e-16 per update, passed on at most a few times
within a sweep; 1e-12 leaves a factor of ten."""

import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [-0.25, 1.0])
@pytest.mark.parametrize("dims", [(16, 16, 16, 16), (12, 16, 24, 32)])
def test_one_sweep_matches_the_oracle(dims, eps):
    from paper_2203_09764_gb300 import vs
    ctx = vs.vs_create(0)
    f = vs.vs_field_create(ctx, dims, vs.VS_FP64, vs.VS_LINK18)
    lab = synth.iid_labels(dims, 12)
    U0 = synth.haar_field(dims, 8)
    Uc = O.centrifuge(dims, lab, 0.02, 3)
    for kind, okind in ((vs.VS_ANNEALED, O.ANNEALED), (vs.VS_SIMULTANEOUS, O.SIMULTANEOUS)):
        vs.vs_load_field(f, links=U0)
        vs.vs_smooth(f, 1, 0.06, eps, kind=kind, vortex_preserve=False)
        want, _ = O.smooth(dims, U0, lab, 1, 0.06, eps=eps, vp=False, schedule=okind)
        assert np.abs(vs.vs_read_field(f) - want).max() < 1e-12
        vs.vs_load_field(f, labels=lab)
        vs.vs_centrifuge(f, 0.02, 3)
        st = vs.vs_smooth(f, 1, 0.06, eps, kind=kind, vortex_preserve=True, stats=True)
        want, rej = O.smooth(dims, Uc, lab, 1, 0.06, eps=eps, vp=True, schedule=okind)
        assert np.abs(vs.vs_read_field(f) - want).max() < 1e-12
        assert st[0]["n_reject"] == int(rej[0])
    vs.vs_field_destroy(f)
    vs.vs_destroy(ctx)
