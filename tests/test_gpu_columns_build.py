"""The first column-form adjoint of a geometry, which builds the geometry's
column records: it waits for no stream, and other streams read the records
only once they are written.  No call disturbs another thread's graph capture."""
import threading

import numpy as np
import pytest

import synth
from synth.geometry import VolumeGeometry

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gjp():
    from paper_1609_00958_gb300 import build
    build.build()
    import paper_1609_00958_gb300 as m
    return m


def _case(gjp):
    """A grid, projections, their adjoint, and a new geometry whose per-view table is there."""
    vg = VolumeGeometry.centred((128, 128, 128))
    cg = synth.circular(12, 100, 130, 400.0, 800.0, 2.0, angles=0.1 + 0.51 * np.arange(12))
    y = torch.from_numpy(np.random.default_rng(2).standard_normal((12, 130, 100)).astype(np.float32)).cuda()
    ref = gjp.adjoint(y, gjp.Geometry.from_cone(cg), vg.n, vg.h)
    g = gjp.Geometry.from_cone(cg)
    gjp.forward(torch.zeros(vg.n, device="cuda"), g, vg.h)
    torch.cuda.synchronize()
    return vg, g, y, ref


def _same(a, b):
    return bool(((a - b).abs().max() <= 1e-5 * b.abs().max()).item())


def test_first_call_waits_for_no_stream(gjp):
    vg, g, y, ref = _case(gjp)
    outs = [torch.full(vg.n, 3.0, device="cuda") for _ in range(2)]
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(first):
        torch.cuda._sleep(1_500_000_000)                 # earlier work on the stream, most of a second
        gjp.adjoint(y, g, vg.n, vg.h, out=outs[0])
    assert not first.query()                             # the call returned before that work was done
    with torch.cuda.stream(second):
        gjp.adjoint(y, g, vg.n, vg.h, out=outs[1])       # its records are still to be written
    assert not first.query()
    torch.cuda.synchronize()
    gjp.stream_status()
    assert _same(outs[0], ref) and _same(outs[1], ref)


@pytest.mark.parametrize("warm", [False, True])
def test_call_during_another_threads_capture(gjp, warm):
    vg, g, y, ref = _case(gjp)
    if warm:
        gjp.adjoint(y, g, vg.n, vg.h)
    out = torch.full(vg.n, 3.0, device="cuda")
    captured = torch.zeros(1000, device="cuda")
    errors = []

    def work(stream):
        try:
            with torch.cuda.stream(stream):
                gjp.adjoint(y, g, vg.n, vg.h, out=out)
        except Exception as e:                           # reported by the test's thread
            errors.append(e)

    worker = threading.Thread(target=work, args=(torch.cuda.Stream(),))
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        captured += 1.0
        worker.start()
        worker.join()
        captured += 1.0
    graph.replay()
    torch.cuda.synchronize()
    assert not errors
    assert float(captured[0]) == 2.0
    assert _same(out, ref)
