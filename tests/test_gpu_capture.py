"""Smoothing calls captured into a CUDA graph by the caller: class launches overlap through
programmatic stream serialisation, which a capture turns into graph edges.  Replays give the bits
of direct calls, on small launches (three warps per 32 links, FP64 rows), on larger ones and after
the memory operations that precede a single class update."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,dims", [("fp32", (8, 8, 8, 8)), ("fp32", (16, 16, 16, 32)), ("fp32", (20, 16, 16, 28)),
                                            ("fp64", (4, 4, 4, 8)), ("fp64", (12, 12, 8, 12))])
@pytest.mark.parametrize("eps", [-0.25, 1.0])
def test_captured_calls_replay_the_direct_result(precision, dims, eps):
    import torch
    from paper_2203_09764_gb300 import vs
    ctx = vs.vs_create(0)
    stream = torch.cuda.Stream()
    prec = vs.VS_FP64 if precision == "fp64" else vs.VS_FP32
    lab = torch.from_numpy(synth.iid_labels(dims, 8)).cuda()
    f = vs.vs_field_create(ctx, dims, prec, vs.VS_LINK18, stream)

    def start():
        vs.vs_load_field(f, labels=lab)
        vs.vs_centrifuge(f, 0.02, 3)

    def work():
        vs.vs_smooth(f, 2, 0.06, eps, reunit_every=0)
        vs.vs_subsweep(f, 1, 2, 0.05, eps)
        vs.vs_smooth_aus(f, 1, 0.02, eps, reunit_every=0)

    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        start()
        work()
        want = vs.vs_read_field(f)
        start()
        vs.vs_synchronize(f)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            work()
        for _ in range(2):
            start()
            graph.replay()
            assert np.array_equal(vs.vs_read_field(f), want)
    vs.vs_field_destroy(f)
    vs.vs_destroy(ctx)
