"""Steps captured into a caller's own CUDA graph form the correction field of the
state they find when the graph is replayed, not of the one before the capture:
populations set in between are stepped as by a handle that was never captured."""
import numpy as np
import pytest

from paper_2107_01370_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2107_01370_gb300 import build, lbfsi
    build.build()
    lbfsi.load()
    return lbfsi


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_captured_steps_start_from_the_state_at_replay(L, precision):
    import torch
    prec = L.FP32 if precision == "fp32" else L.FP64
    case = inputs.cylinder_case(48, 64, r_far=8.0, re=10.0)
    M0 = inputs.initial_field(48, 64, case.flow, noise=0.05, seed=1)
    other = inputs.initial_field(48, 64, case.flow, noise=0.05, seed=2)
    stream = torch.cuda.Stream()

    def start(field):
        m = L.Mesh(case.r, case.e, case.bodies, precision=prec, stream=stream.cuda_stream)
        m.init_fields(case.flow, field[None])
        m.step(2)
        m.step(2)
        m.synchronize()
        return m

    a = start(other)
    state = (*a.get_populations(0), a.get_fields())
    a.set_populations(*state)
    a.step(2)
    want = a.get_fields()
    a.close()
    b = start(M0)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        b.step(2)
    b.set_populations(*state)
    graph.replay()
    torch.cuda.synchronize()
    got = b.get_fields()
    b.set_populations(*state)             # a plain call behind the capture
    b.step(2)
    again = b.get_fields()
    b.close()
    assert np.array_equal(got, want) and np.array_equal(again, want)
