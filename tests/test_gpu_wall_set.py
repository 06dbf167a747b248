"""Which populations a wall node misses is decided in float64 on the float path
too: a cylinder turning about its own centre has a wall velocity along the
wall, so its rest population is never missing.  Far from the origin float
coordinates round by 2^-24 of 10^4, and the wall's float velocity (turning at
0.1) is off by up to w = 0.1 x 6e-4 across the wall, which a sign test in float
takes for a wall node without its rest population: Grad's approximation in
place of the streamed one, a change of some 1e-2.

Tolerance of the float populations against the float64 handle's: w enters them
through the wall velocity of Grad's populations (df/du below 1) and the
departure points (dt w of a cell's spacing times the field's change over it):
2 w, and 1e-5 for the path's own rounding."""
import numpy as np
import pytest

from paper_2107_01370_gb300 import inputs

pytestmark = pytest.mark.gpu
FAR = 1.0e4


@pytest.fixture(scope="module")
def L():
    from paper_2107_01370_gb300 import build, lbfsi
    build.build()
    lbfsi.load()
    return lbfsi


@pytest.mark.parametrize("kind", ["rings", "coordinates"])
@pytest.mark.parametrize("at", [0.0, FAR])
def test_fp32_missing_set_is_the_float64_set(L, kind, at):
    turn = 0.1
    body = inputs.BodySpec(dof=2, xc=at, xp=at, r_in=0.75, r_out=2.0, m_star=80.0, v_r=0.2, x_alpha=0.0, r_alpha=0.5,
                           wh_wa=0.5)
    case = inputs.cylinder_case(32, 64, r_far=8.0, body=body)
    a = 0.5 * turn * case.flow.dt
    M0 = inputs.initial_field(32, 64, case.flow, noise=1e-2, seed=4)
    got = []
    for prec in (L.FP64, L.FP32):
        if kind == "rings":
            m = L.Mesh(case.r, case.e, case.bodies, precision=prec, centre=(at, 0.0))
        else:
            X = case.r[:, None, None] * case.e[None] + np.array([at, 0.0])
            m = L.Mesh.xy(X, case.bodies, precision=prec, centre=(at, 0.0))
        m.init_fields(case.flow, M0[None])
        m.blend_mesh([(0.0, a, 0.0, turn)], [(0.0, -a, 0.0, turn)])
        m.step(1)
        got.append(np.stack(m.get_populations(0)).reshape(2, 9, 32, 64)[:, :, 0])
        m.close()
    w = turn * 2.0 ** -24 * max(at, 1.0)
    assert np.abs(got[1] - got[0])[0].max() < 2.0 * w + 1e-5
