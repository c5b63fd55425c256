"""Rounding of the action and of the observables' action density.

FP64: links U_0 = diag(1 - d, 1, 1), d = 2^-25, the others 1.  The plaquettes (0, nu) have trace
(1 - d)^2 + 2, exact in FP64 in any order, and 3 less it, 2 d - d^2, is exact too; the other plaquettes
give 0.  So a site's sum 3 (2 d - d^2) has 28 bits and the action's sum over the sites is exact: what is
left are two roundings of the scale, 1e-15.  The observables scale each site before they add: 256
additions, 1e-13."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    from paper_2203_09764_gb300 import vs
    ctx = vs.vs_create(0)
    yield vs, ctx
    vs.vs_destroy(ctx)


def _links(dims, first):
    U = np.zeros((4, int(np.prod(dims)), 3, 3), dtype=np.complex128)
    U[:] = np.eye(3)
    U[0] = np.diag(first)
    return U


def test_a_small_fp64_action_keeps_its_digits(env):
    vs, ctx = env
    dims, d = (4, 4, 4, 4), 2.0 ** -25
    f = vs.vs_field_create(ctx, dims, vs.VS_FP64, vs.VS_LINK18)
    vs.vs_load_field(f, links=_links(dims, (1 - d, 1, 1)))
    want = 2.0 / 72.0 * 3 * (2 * d - d * d)
    assert abs(vs.vs_action(f) / want - 1) < 1e-15
    o = vs.vs_observables(f, per_site=True)
    assert abs(o["mean_S"] / want - 1) < 1e-13
    assert np.abs(o["S"] / want - 1).max() < 1e-15
    vs.vs_field_destroy(f)
