"""Layouts of the step that follow the sizes: the tile shape a float handle
or batch takes when no schedule is asked for, and the element list's blocks of
256 nodes and gradient rows in slices of 32.

Tolerance of the float paths against the float64 oracle: a population is a sum
of nine terms whose weights' magnitudes sum to at most 1.6, on deviations from
the free stream, so a step adds at most some ten roundings (6e-8 each) of the
field; 8 steps 5e-6, held to 1e-5.  Loads: the same relative error of a sum of
pressures of order p_inf over the wall, 1e-4 of p_inf D."""
import numpy as np
import pytest

import oracle.mesh as OM
import oracle.solver as OS
import oracle.unstructured as OU
from paper_2107_01370_gb300 import inputs

pytestmark = pytest.mark.gpu
STEPS = 8
P_SCALE = 1.0 / 3.0


@pytest.fixture(scope="module")
def L():
    from paper_2107_01370_gb300 import build, lbfsi
    build.build()
    lbfsi.load()
    return lbfsi


def _err(a, b):
    return max(np.abs(a[0] - b[0]).max() / np.abs(b[0]).max(),
               np.hypot(a[1] - b[1], a[2] - b[2]).max() / np.hypot(b[1], b[2]).max(),
               np.abs(a[3] - b[3]).max() / np.abs(b[3]).max())


# solves of 4 or 6 tiles of 16 x 32 nodes (the last with one row, ragged
# columns) on both sides of the default shape's lines at 152 and 608 tiles
@pytest.mark.parametrize("nr,nt,nb", [(17, 34, 37), (17, 34, 38), (33, 62, 101), (33, 62, 102)])
def test_float_default_shape_either_side_of_its_lines(L, nr, nt, nb):
    body = inputs.BodySpec(dof=1, r_in=0.75, r_out=2.0, m_star=3.0, v_r=5.0)
    case = inputs.cylinder_case(nr, nt, r_far=10.0, body=body)
    M0 = inputs.initial_field(nr, nt, case.flow, seed=nr)
    s = OS.Solver.from_case(OM.ogrid_mesh(case.r, case.e), case, M0)
    for _ in range(STEPS):
        r = s.step()
    out = []
    for schedule in (None, (0, 0), (1, 0), (4, 1)):
        m = L.Mesh(case.r, case.e, case.bodies * nb, precision=L.FP32)
        if schedule is not None:
            m.set_schedule(*schedule)
        m.init_fields(case.flow, np.ascontiguousarray(np.broadcast_to(M0, (nb,) + M0.shape)))
        m.step(STEPS)
        out.append((m.get_fields(), m.body_forces()))
        m.close()
    b = L.Batch(128 << 20, precision=L.FP32)
    ids = [b.add(case.r, case.e, case.bodies[0], case.flow, STEPS, M0) for _ in range(nb)]
    while b.step(1) > 0:
        pass
    got = [b.get(i) for i in ids]
    b.close()
    out.append((np.stack([g[0] for g in got]), np.stack([g[1] for g in got])))
    for f, F in out:
        assert np.array_equal(f, out[0][0]) and np.array_equal(F, out[0][1])
        assert all(np.array_equal(f[k], f[0]) for k in (1, nb - 1))
    assert _err(out[0][0][0], r.M) < 1e-5
    assert np.abs(out[0][1][0] - np.array(r.force)).max() < 1e-4 * P_SCALE


# node counts below, at and past whole blocks and slices; solves that fill a
# pair or not; and a thin ring whose blocks' elements reach 1288 nodes (its
# first step alone, the one without a correction field: second derivatives over
# spacings of 1e-3 multiply float roundings by 1e6, so the bound above does not
# hold for the steps that follow)
@pytest.mark.parametrize("nr,nt,nb,thin", [(7, 24, 1, False), (16, 16, 2, False), (17, 32, 3, False),
                                           (25, 48, 2, False), (257, 16, 3, True)])
def test_float_element_list_blocks(L, nr, nt, nb, thin):
    if thin:
        body = inputs.BodySpec(dof=1, r_in=0.6, r_out=0.75, m_star=2.0, v_r=4.0)
        case = inputs.cylinder_case(25, 48, r_far=8.0, re=1e4, body=body)
        case.flow.dt = 0.001 / 3.0
        X = inputs.ogrid_radii(nr, 0.5, 0.8, 0.001)[:, None, None] * inputs.ogrid_directions(nt)[None]
    else:
        body = inputs.BodySpec(dof=1, r_in=0.75, r_out=2.0, m_star=2.0, v_r=4.0)
        case = inputs.cylinder_case(nr + 1 - nr % 2, nt, r_far=8.0, body=body)
        X = case.r[:nr, None, None] * case.e[None]
    if nr % 2 == 0:
        X = X[:nr - 1]
    el = inputs.ogrid_element_list(X, seed=nr)
    M0 = inputs.initial_field(X.shape[0], nt, case.flow, seed=nr, noise=1e-2)
    h, hdot = 1e-3, 4e-3
    state = {"h": h, "alpha": 0.0, "hdot": hdot, "adot": 0.0}
    prev = dict(state, h=h - hdot * case.flow.dt)
    s = OU.UnstructuredSolver.from_case(OU.UnstructuredQ2Mesh(el.X, el.elements), el.wall, el.far, case, el.to_list(M0))
    s.S, s.S_prev = [dict(state)], [dict(prev)]
    steps = 1 if thin else STEPS
    for _ in range(steps):
        r = s.step()
    m = L.ElementMesh(el.X, el.elements, el.wall, el.far, case.bodies * nb, precision=L.FP32)
    m.init_fields(case.flow, np.ascontiguousarray(np.broadcast_to(el.to_list(M0), (nb, 4, el.X.shape[0]))))
    m.blend_mesh([(h, 0.0, hdot, 0.0)] * nb, [(prev["h"], 0.0, hdot, 0.0)] * nb)
    m.step(steps)
    f, F = m.get_fields(), m.body_forces()
    m.close()
    assert all(np.array_equal(f[k], f[0]) and np.array_equal(F[k], F[0]) for k in range(nb))
    assert _err(f[0], r.M) < 1e-5
    assert np.abs(F[0] - np.array(r.force)).max() < 1e-4 * P_SCALE
