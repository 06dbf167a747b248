"""The float64 path's reciprocals are rounded correctly: a node's velocity is its
momentum, summed in the stream's order, times the correctly rounded 1 / rho, to
the last bit (a reciprocal an ulp off would miss at every few nodes)."""
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


@pytest.mark.parametrize("kind", ["rings", "section"])
def test_fp64_velocity_is_momentum_times_the_rounded_reciprocal(L, kind):
    body = inputs.BodySpec(dof=1, r_in=0.75, r_out=2.0, m_star=3.0, v_r=4.0)
    if kind == "rings":
        case = inputs.cylinder_case(48, 64, r_far=8.0, body=body)
        m = L.Mesh(case.r, case.e, case.bodies, precision=L.FP64)
    else:
        case = inputs.xy_case(inputs.ellipse_wall(64, 0.6, 0.35), 48, r_far=8.0, length=1.2, body=body)
        m = L.Mesh.xy(case.X, case.bodies, precision=L.FP64)
    m.init_fields(case.flow, inputs.initial_field(48, 64, case.flow, noise=0.1, seed=9)[None])
    m.step(5)
    M = m.get_fields()[0].reshape(4, 48, 64)[:, :-1]          # off the far field
    f = m.get_populations(0)[0][0].reshape(9, 48, 64)[:, :-1]
    m.close()
    rho = (((f[0] + f[1]) + f[2]) + (f[3] + f[4])) + ((f[5] + f[6]) + (f[7] + f[8]))
    jx = (f[1] + -f[3]) + ((f[5] - f[6]) + (f[8] - f[7]))
    jy = (f[2] + -f[4]) + ((f[5] + f[6]) + -(f[7] + f[8]))
    assert np.array_equal(M[0], rho)
    assert np.array_equal(M[1], jx * (1.0 / rho))
    assert np.array_equal(M[2], jy * (1.0 / rho))
