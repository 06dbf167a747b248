"""Default tile shapes and CTA orders of float handles by their size: every solve
of a handle has the same inputs, so a handle of one solve (8-row tiles on general
meshes), of as many as fill 16-row tiles of 256 or 512 threads, and of as many as
take the solve-by-solve order give the same bits; and those are the oracle's
within the float path's bound of 1e-5 after eight steps."""
import numpy as np
import pytest

import oracle.mesh as OM
import oracle.solver as OS
from paper_2107_01370_gb300 import inputs

pytestmark = pytest.mark.gpu
STEPS = 8


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


# 16-row tiles of a solve: 6 (rings, section; 2112 nodes), 6 (section of 50
# columns, staged by per-thread copies), 9 (C-grid)
@pytest.mark.parametrize("dof", [0, 1])
@pytest.mark.parametrize("kind,counts", [("rings", (26, 102, 180)), ("section", (38, 39, 76, 77, 101, 102, 180)),
                                         ("section50", (38, 39, 102)), ("cgrid", (25, 26, 68)), ("box", (38, 39))])
def test_default_shapes_and_orders_agree_to_the_bit(L, kind, counts, dof):
    body = inputs.BodySpec(dof=dof, r_in=0.75, r_out=2.0, m_star=3.0, v_r=5.0, length=1.2)
    if kind == "rings":
        case = inputs.cylinder_case(33, 64, r_far=8.0, body=body)
        mesh = OM.ogrid_mesh(case.r, case.e)
        make = lambda nb: L.Mesh(case.r, case.e, case.bodies * nb, precision=L.FP32)
    elif kind == "box":
        if dof:
            pytest.skip("a box has no body")
        X, si, sj = inputs.box_mesh(34, 66, 34.0, 66.0, skew=0.2)
        case = inputs.cylinder_case(34, 66, r_far=10.0)
        case.flow.dt = 0.5
        mesh = OM.periodic_box_mesh(34, 66, 34.0, 66.0, skew=0.2)
        make = lambda nb: L.Mesh.box(X, si, sj, nbatch=nb, precision=L.FP32)
    elif kind == "cgrid":
        case = inputs.cgrid_case(49, 10, 33, 0.6, 0.35, r_far=6.0, wake=4.0, length=1.2, body=body)
        mesh = OM.CGridMesh(case.X, case.n_cut)
        make = lambda nb: L.Mesh.cgrid(case.X, case.n_cut, case.bodies * nb, precision=L.FP32)
    else:
        nt = 64 if kind == "section" else 50
        case = inputs.xy_case(inputs.ellipse_wall(nt, 0.6, 0.35), 33, r_far=8.0, length=1.2, body=body)
        mesh = OM.Q2Mesh(case.X)
        make = lambda nb: L.Mesh.xy(case.X, case.bodies * nb, precision=L.FP32)
    nr, nt = mesh.X.shape[:2]
    M0 = inputs.initial_field(nr, nt, case.flow, noise=1e-2, seed=nt)
    if kind == "box":
        fl = case.flow
        s = OS.Solver(mesh, gamma=fl.gamma, Pr=fl.pr, mu=fl.mu, dt=fl.dt, rho_inf=1.0, u_inf=(fl.u_inf, 0.0),
                      T_inf=fl.t_inf, bodies=[], M0=M0, walls=False)
    else:
        s = OS.Solver.from_case(mesh, case, M0)
    for _ in range(STEPS):
        r = s.step()
    first = None
    for nb in (1,) + counts:
        m = make(nb)
        m.init_fields(case.flow, np.ascontiguousarray(np.broadcast_to(M0, (nb,) + M0.shape)))
        m.step(STEPS)
        f = m.get_fields().reshape(nb, 4, nr, nt)
        m.close()
        if first is None:
            first = f[0]
            assert _err(first, r.M) < 1e-5
        assert all(np.array_equal(f[k], first) for k in (0, nb // 2, nb - 1)), nb
