"""The float correction field node by node: the post-collision populations of a
state against the oracle's collision of the same populations and moments, on
widths and heights on both sides of the field kernel's strips (28 columns x 6
rows on separable meshes, 26 x 4 on meshes by coordinates; a C-grid's outlet
columns alone in the last strip, in its halo, or with it full).

Tolerance: a population passes some sixteen roundings of 2^-24, 1e-6 of the
largest one.  Y = d[(mu/p) d dQ] is a sum of products of two index derivatives
(coefficients of one-sided stencils sum to 4) and two metrics: 16 terms of
size (mu/p) |dQ| J^2 near the node, each with some ten roundings; 256 x 2^-24
of that size times dt / 2."""
import numpy as np
import pytest

import oracle.ale as OA
import oracle.kinetics as K
import oracle.mesh as OM
import oracle.solver as OS
from paper_2107_01370_gb300 import inputs

pytestmark = pytest.mark.gpu
REST = {"h": 0.0, "alpha": 0.0, "hdot": 0.0, "adot": 0.0}


@pytest.fixture(scope="module")
def L():
    from paper_2107_01370_gb300 import build, lbfsi
    build.build()
    lbfsi.load()
    return lbfsi


def _near(a):
    """Largest value within two nodes (across the ends too, never smaller)."""
    for axis in (0, 1):
        a = np.max([np.roll(a, k, axis) for k in range(-2, 3)], axis=0)
    return a


def _check(m, s, state, far):
    """Collide the handle's state with the oracle s's mesh and flow, bodies in
    the given state; compare the nodes off the far field."""
    M = m.get_fields()[0]
    f, g = (a[0] for a in m.get_populations(0))
    post = m.get_populations(1)[0][0]
    m.close()
    shape = M.shape[1:]
    f, g, post = (a.reshape((9,) + shape) for a in (f, g, post))
    F = OA.deformation_gradient(s.mesh.X, s.bodies, [state] * len(s.bodies))
    dqx, dqy = K.delta_q(*M)
    mu_p = s.mu / (M[0] * M[3])
    Yx = s._physical_grad(F, mu_p * s._physical_grad(F, dqx)[0])[0]
    Yy = s._physical_grad(F, mu_p * s._physical_grad(F, dqy)[1])[1]
    with np.errstate(divide="ignore", invalid="ignore"):
        want = K.collide(f, g, Yx, Yy, s.mu, s.dt, s.Cv, s.Pr)[0]
    x_xi, y_xi, x_eta, y_eta = s.mesh.metrics()
    det = np.abs(x_xi * y_eta - y_xi * x_eta)
    J = np.maximum(np.abs(y_eta) + np.abs(y_xi), np.abs(x_eta) + np.abs(x_xi)) / det
    size = 0.5 * s.dt * _near(mu_p * np.maximum(np.abs(dqx), np.abs(dqy))) * _near(J) ** 2
    tol = 1e-6 * np.abs(f).max() + 256 * 2.0 ** -24 * size
    err = np.abs(post - want).max(axis=0)
    err[far] = 0.0
    worst = np.unravel_index(np.argmax(err / tol), shape)
    assert (err <= tol).all(), (worst, err[worst], tol[worst])


def _far_rows(shape):
    far = np.zeros(shape, bool)
    far[-1] = True
    return far


# (Y is largest where the field varies from node to node: noise, in a viscous
# flow; at three times this noise the oracle's own state leaves T > 0)
@pytest.mark.parametrize("n_wall,n_cut,nr", [(37, 8, 9), (63, 8, 14), (41, 8, 8), (39, 8, 11), (61, 8, 10),
                                             (35, 8, 13), (49, 8, 12)])
def test_cgrid_strips(L, n_wall, n_cut, nr):
    case = inputs.cgrid_case(n_wall, n_cut, nr, 0.6, 0.35, r_far=6.0, wake=4.0, length=1.2, re=1.0)
    M0 = inputs.initial_field(nr, case.ntheta, case.flow, noise=0.1, seed=n_wall)
    s = OS.Solver.from_case(OM.CGridMesh(case.X, n_cut), case, M0)
    m = L.Mesh.cgrid(case.X, n_cut, case.bodies, precision=L.FP32)
    m.init_fields(case.flow, M0[None])
    m.step(1)
    far = _far_rows((nr, case.ntheta))
    far[:, 0] = far[:, -1] = True
    _check(m, s, REST, far)


@pytest.mark.parametrize("kind,nr,nt", [("rings", 7, 26), ("rings", 12, 28), ("rings", 13, 30), ("rings", 11, 56),
                                        ("rings", 18, 58), ("section", 7, 24), ("section", 8, 26), ("section", 9, 28),
                                        ("section", 10, 52), ("section", 13, 54)])
@pytest.mark.parametrize("dof", [0, 1])
def test_ogrid_strips(L, kind, nr, nt, dof):
    body = inputs.BodySpec(dof=dof, r_in=0.75, r_out=2.5, m_star=3.0, v_r=5.0)
    if kind == "rings":
        case = inputs.cylinder_case(nr, nt, r_far=6.0, re=1.0, body=body)
        mesh = OM.ogrid_mesh(case.r, case.e)
        m = L.Mesh(case.r, case.e, case.bodies, precision=L.FP32)
    else:
        case = inputs.xy_case(inputs.ellipse_wall(nt, 0.6, 0.35), nr, r_far=6.0, length=1.2, re=1.0, body=body)
        mesh = OM.Q2Mesh(case.X)
        m = L.Mesh.xy(case.X, case.bodies, precision=L.FP32)
    M0 = inputs.initial_field(nr, nt, case.flow, noise=0.1, seed=nr * nt)
    s = OS.Solver.from_case(mesh, case, M0)
    m.init_fields(case.flow, M0[None])
    state = dict(REST, h=0.05, hdot=0.01) if dof else REST
    if dof:
        at = (state["h"], 0.0, state["hdot"], 0.0)
        m.blend_mesh([at], [at])
    m.step(1)
    _check(m, s, state, _far_rows((nr, nt)))


@pytest.mark.parametrize("ni,nj", [(8, 24), (10, 26), (12, 28), (14, 52), (8, 54)])
def test_box_strips(L, ni, nj):
    X, si, sj = inputs.box_mesh(ni, nj, float(ni), float(nj), skew=0.3)
    dt = 0.5
    flow = inputs.FlowSpec(ma=0.1, re=10.0, t_inf=1.0 / 3.0, gamma=1.4, pr=0.71, rho_inf=1.0, dt=dt, length=1.0)
    M0 = inputs.initial_field(ni, nj, flow, noise=0.1, seed=nj)
    s = OS.Solver(OM.periodic_box_mesh(ni, nj, float(ni), float(nj), skew=0.3), gamma=flow.gamma, Pr=flow.pr,
                  mu=flow.mu, dt=dt, rho_inf=1.0, u_inf=(flow.u_inf, 0.0), T_inf=flow.t_inf, bodies=[], M0=M0,
                  walls=False)
    m = L.Mesh.box(X, si, sj, precision=L.FP32)
    m.init_fields(flow, M0[None])
    m.step(1)
    _check(m, s, REST, np.zeros((ni, nj), bool))
