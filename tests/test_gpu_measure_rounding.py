"""Rounding of the action and of the observables' action density.

FP64: links U_0 = diag(1 - d, 1, 1), d = 2^-25, the others 1.  The plaquettes (0, nu) have trace
(1 - d)^2 + 2, exact in FP64 in any order, and 3 less it, 2 d - d^2, is exact too; the other plaquettes
give 0.  So a site's sum 3 (2 d - d^2) has 28 bits and the action's sum over the sites is exact: what is
left are two roundings of the scale, 1e-15.  The observables scale each site before they add: 256
additions, 1e-13.

FP32 adds the traces as an error-free pair: an infinite one stays infinite."""

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


@pytest.mark.parametrize("storage", [18, 12])
def test_an_infinite_fp32_trace_stays_infinite(env, storage):
    """diag(1e20, 1, 1e20) squared passes the largest float: the plaquettes (0, nu) have trace
    +inf, so the action is -inf, as a sum of 3 - Re Tr P in any precision gives it."""
    vs, ctx = env
    dims = (4, 4, 4, 8)
    f = vs.vs_field_create(ctx, dims, vs.VS_FP32, vs.VS_LINK12 if storage == 12 else vs.VS_LINK18)
    vs.vs_load_field(f, links=_links(dims, (1e20, 1, 1e20)))
    assert vs.vs_action(f) == -np.inf
    vs.vs_field_destroy(f)
