"""Fields beyond the positions at which an element offset passes 2^31 (18 reals: 119,304,647; 12
reals: 178,956,970): links repeated along t from a field of eight time slices, whose updates take the
same kernels.  Every updated link of every copy is the small field's, bit for bit."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


class _Device:
    def __init__(self, ptr, n, typestr):
        self.__cuda_array_interface__ = {"data": (int(ptr), False), "shape": (n,), "typestr": typestr, "version": 2}


def _planes(torch, d, components, typestr):
    n = components * d["plane_stride"]
    return torch.as_tensor(_Device(d["links"], 4 * n, typestr), device="cuda").view(4, n)


# GB of the large field: 39, 39, 77
@pytest.mark.parametrize("precision,storage,space,copies", [("fp32", 18, (64, 128, 128), 16),
                                                            ("fp32", 12, (96, 128, 128), 16),
                                                            ("fp64", 18, (64, 128, 128), 16)])
def test_links_repeated_beyond_the_32_bit_offsets(precision, storage, space, copies):
    import torch
    from paper_2203_09764_gb300 import vs
    small, large = space + (8,), space + (8 * copies,)
    V = int(np.prod(large))
    assert storage * V > 2 ** 31
    if torch.cuda.mem_get_info()[0] < 4 * V * (storage * (8 if precision == "fp64" else 4) + 6) * 1.1:
        pytest.skip("not enough device memory")
    prec = vs.VS_FP64 if precision == "fp64" else vs.VS_FP32
    st = vs.VS_LINK12 if storage == 12 else vs.VS_LINK18
    typestr = "<f8" if precision == "fp64" else "<f4"
    ctx = vs.vs_create(0)
    fs = vs.vs_field_create(ctx, small, prec, st)
    fl = vs.vs_field_create(ctx, large, prec, st)
    lab = torch.from_numpy(synth.iid_labels((8, 8, 8, 8), 5)).cuda().view(4, 8, 8, 8, 8)
    lab = lab.repeat(1, 1, *(e // 8 for e in space[::-1])).contiguous()
    torch.cuda.synchronize()
    vs.vs_load_field(fs, labels=lab.view(-1))
    vs.vs_centrifuge(fs, 0.02, 3)
    vs.vs_load_field(fl, labels=lab.repeat(1, copies, 1, 1, 1).view(-1))
    vs.vs_synchronize(fs)
    vs.vs_synchronize(fl)
    ps = _planes(torch, vs.vs_field_describe(fs), storage, typestr)
    pl = _planes(torch, vs.vs_field_describe(fl), storage, typestr)
    pl.view(4, copies, -1).copy_(ps.view(4, 1, -1).expand(4, copies, -1))
    torch.cuda.synchronize()
    for f in (fs, fl):
        if precision == "fp32":
            vs.vs_smooth(f, 1, 0.06, -0.25)
            vs.vs_subsweep(f, 1, 3, 0.06, 1.0)
        else:
            vs.vs_subsweep(f, 0, 2, 0.06, -0.25)
            vs.vs_subsweep(f, 3, 1, 0.06, -0.25)
        vs.vs_synchronize(f)
    for mu in range(4):
        for c in range(copies):
            assert torch.equal(pl[mu].view(copies, -1)[c], ps[mu])
    a, b = vs.vs_vortex_check(fs), vs.vs_vortex_check(fl)
    assert a["n_label_diff"] == 0 and b["n_label_diff"] == 0 and a["min_margin"] == b["min_margin"]
    assert b["n_near_boundary"] == copies * a["n_near_boundary"]
    # sums of the same terms, up to 1e5 in a row: 1e5 half-ulps
    assert abs(vs.vs_action(fl) / vs.vs_action(fs) - 1) < 1.2e-11
    vs.vs_field_destroy(fl)
    vs.vs_field_destroy(fs)
    vs.vs_destroy(ctx)
