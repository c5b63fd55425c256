"""FP64 vortex check on both sides of the field size up to which it takes a thread per link (65,536
sites), in the original gauge and in a random one, against numpy: label and charge differences of a
general field from given labels, links near a sector edge and the smallest margin."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _labels(tr):
    a = np.angle(tr)
    return np.where(np.abs(a) < np.pi / 3, 0, np.sign(a)).astype(np.int64)


def _charges(lab, dims):
    n = lab.reshape(4, *dims[::-1])
    out = []
    for mu in range(4):
        for nu in range(mu + 1, 4):
            ax = [3 - mu, 3 - nu]      # axes of [t][z][y][x]
            p = n[mu] + np.roll(n[nu], -1, ax[0]) - np.roll(n[mu], -1, ax[1]) - n[nu]
            out.append(p % 3)
    return np.array(out)


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (16, 16, 16, 16), (16, 16, 16, 20)])
@pytest.mark.parametrize("gauge", [False, True])
def test_check_matches_numpy(dims, gauge):
    from paper_2203_09764_gb300 import vs
    V = int(np.prod(dims))
    U = synth.haar_field(dims, 21)
    ref = synth.iid_labels(dims, 22)
    ctx = vs.vs_create(0)
    f = vs.vs_field_create(ctx, dims, vs.VS_FP64, vs.VS_LINK18)
    vs.vs_field_restore(f, U, ref, 0)
    if gauge:
        # a centre element per site leaves the traces to the transformed test to undo
        k = np.arange(V) % 3
        G = np.exp(2j * np.pi * k / 3)[:, None, None] * np.eye(3)
        vs.vs_gauge_transform(f, G)
    got = vs.vs_vortex_check(f)
    vs.vs_field_destroy(f)
    vs.vs_destroy(ctx)
    tr = np.trace(U.reshape(4, V, 3, 3), axis1=2, axis2=3)
    a = np.angle(tr)
    margin = np.minimum(np.minimum(np.abs(a - np.pi / 3), np.abs(a + np.pi / 3)), np.pi - np.abs(a))
    lab, old = _labels(tr), np.asarray(ref, dtype=np.int64).reshape(4, V)
    assert got["n_label_diff"] == int((lab != old).sum())
    assert got["n_charge_diff"] == int((_charges(lab, dims) != _charges(old, dims)).sum())
    assert got["n_near_boundary"] == int((margin < 1e-5).sum())
    # the trace's rounding (3e-15 here, a few more in a gauge) over its size, 1e-3 or more at the smallest margin
    assert abs(got["min_margin"] - margin.min()) < 1e-11
