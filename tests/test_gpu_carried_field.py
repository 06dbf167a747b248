"""The correction field that a call leaves for the next: formed only by a call
that itself followed another with the state unchanged (the launch count: two per
step, one more where a call forms the field of its first state), and the same
bits however a run is cut into calls."""
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


def _start(L, precision):
    body = inputs.BodySpec(dof=1, r_in=0.75, r_out=2.0, m_star=3.0, v_r=4.0)
    case = inputs.cylinder_case(32, 64, r_far=8.0, body=body)
    m = L.Mesh(case.r, case.e, case.bodies, precision=L.FP64 if precision == "fp64" else L.FP32)
    m.init_fields(case.flow, inputs.initial_field(32, 64, case.flow, noise=1e-2, seed=2)[None])
    return m


def _launches(m, n):
    before = m.launch_count()
    m.step(n)
    return m.launch_count() - before


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_field_is_left_only_where_calls_follow(L, precision):
    m = _start(L, precision)
    first = _launches(m, 3)
    assert first in (6, 7)                 # (7: the initial state put in place by a field launch)
    assert _launches(m, 3) == 7            # forms its first state's field, leaves the last's
    assert _launches(m, 3) == 6 and _launches(m, 1) == 2
    for _ in range(2):                     # the bodies set between calls: nothing left, nothing taken
        m.blend_mesh([(0.01, 0.0, 0.0, 0.0)], [(0.01, 0.0, 0.0, 0.0)])
        assert _launches(m, 2) == 5
    assert _launches(m, 2) == 5 and _launches(m, 2) == 4
    m.field_ptr(L.FIELD_MOMENTS)           # a field's address handed out: every call forms its own
    assert _launches(m, 2) == 5 and _launches(m, 2) == 5
    m.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_cuts_of_a_run_agree_to_the_bit(L, precision):
    got = []
    for cuts in ((12,), (1,) * 12, (5, 1, 6), (2, 4, 6)):
        m = _start(L, precision)
        for n in cuts:
            m.step(n)
            m.get_populations(1)
        got.append((m.get_fields(), *m.get_populations(0), m.body_forces()))
        m.close()
    for g in got[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(g, got[0]))
