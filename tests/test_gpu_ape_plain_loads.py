"""Unit circle projection with plaquette staples on rows of an odd number of class sites, where a
colour class of FP32 links takes plain loads: 32,256 and 59,904 links in rows of 4 (one site per row
and class), 60,480 in rows of 12 and, with 18 reals, 64,512 in rows of 36.  One sweep of a periodic
field against the oracle's sweep of one period; tolerance as for the same sweep on small lattices,
3e-6."""

import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,tile,reps", [(18, (4, 8, 8, 4), (1, 3, 6, 13)), (12, (4, 8, 8, 4), (1, 3, 6, 13)),
                                               (18, (4, 8, 8, 4), (1, 3, 6, 7)), (12, (4, 8, 8, 4), (1, 3, 6, 7)),
                                               (18, (12, 4, 4, 12), (1, 5, 7, 3)), (12, (12, 4, 4, 12), (1, 5, 7, 3)),
                                               (18, (36, 4, 4, 4), (1, 4, 4, 7))])
def test_one_sweep_of_a_periodic_field(storage, tile, reps):
    from paper_2203_09764_gb300 import vs
    dims = tuple(t * r for t, r in zip(tile, reps))
    U0 = O.cool(tile, synth.haar_field(tile, 6), 1)
    big = U0.reshape(4, tile[3], tile[2], tile[1], tile[0], 3, 3)
    big = np.tile(big, (1, reps[3], reps[2], reps[1], reps[0], 1, 1)).reshape(4, -1, 3, 3)
    want, _ = O.ape_ucp(tile, U0, None, 1, 0.02, eps=1.0, vp=False)
    ctx = vs.vs_create(0)
    f = vs.vs_field_create(ctx, dims, vs.VS_FP32, vs.VS_LINK12 if storage == 12 else vs.VS_LINK18)
    vs.vs_load_field(f, links=big)
    vs.vs_smooth_ape(f, 1, 0.02, 1.0, vortex_preserve=False, reunit_every=0)
    got = vs.vs_read_field(f).reshape(4, reps[3], tile[3], reps[2], tile[2], reps[1], tile[1], reps[0], tile[0], 3, 3)
    first = got[:, 0, :, 0, :, 0, :, 0]
    assert np.array_equal(got, np.broadcast_to(first[:, None, :, None, :, None, :, None], got.shape))
    assert np.abs(first.reshape(4, -1, 3, 3) - want).max() < 3e-6
    vs.vs_field_destroy(f)
    vs.vs_destroy(ctx)
