"""Float64 departure points on strongly skewed cells at large displacements: a
doubly periodic box whose element corners are moved at random by up to 0.6 of
their half width, against the oracle, whose Newton iteration runs to
convergence.  Tolerance as for every float64 field, 1e-12."""
import numpy as np
import pytest

import oracle.mesh as OM
import oracle.solver as OS
from paper_2107_01370_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2107_01370_gb300 import build, lbfsi
    build.build()
    lbfsi.load()
    return lbfsi


def _skewed_box(ni, nj, moved, seed):
    rng = np.random.default_rng(seed)
    ci, cj = ni // 2, nj // 2
    C = np.empty((ci + 1, cj + 1, 2))
    C[..., 0] = 2.0 * np.arange(ci + 1)[:, None]
    C[..., 1] = 2.0 * np.arange(cj + 1)[None, :]
    d = moved * rng.uniform(-1, 1, (ci, cj, 2))
    C[:ci, :cj] += d
    C[ci, :cj] += d[0]
    C[:ci, cj] += d[:, 0]
    C[ci, cj] += d[0, 0]
    X = np.empty((ni + 1, nj + 1, 2))
    X[::2, ::2] = C
    X[1::2, ::2] = 0.5 * (C[1:] + C[:-1])
    X[:, 1::2] = 0.5 * (X[:, 2::2] + X[:, :-1:2])
    return np.ascontiguousarray(X[:ni, :nj]), (float(ni), 0.0), (0.0, float(nj))


@pytest.mark.parametrize("moved,dt,cache", [(0.1, 0.45, True), (0.5, 0.45, True), (0.6, 0.35, True), (0.6, 0.35, False)])
def test_fp64_departures_on_skewed_cells(L, moved, dt, cache, monkeypatch):
    if not cache:
        monkeypatch.setenv("LBFSI_NO_DEPARTURE_CACHE", "1")
    X, si, sj = _skewed_box(24, 16, moved, 1)
    flow = inputs.FlowSpec(ma=0.1, re=10.0, t_inf=1.0 / 3.0, gamma=1.4, pr=0.71, rho_inf=1.0, dt=dt, length=1.0)
    M0 = inputs.initial_field(24, 16, flow, noise=0.3, seed=1)
    s = OS.Solver(OM.Q2Mesh(X, periodic_i=True, periodic_j=True, shift_i=si, shift_j=sj), gamma=flow.gamma, Pr=flow.pr,
                  mu=flow.mu, dt=dt, rho_inf=1.0, u_inf=(flow.u_inf, 0.0), T_inf=flow.t_inf, bodies=[], M0=M0,
                  walls=False)
    m = L.Mesh.box(X, si, sj, precision=L.FP64)
    m.init_fields(flow, M0[None])
    for _ in range(2):
        r = s.step()
    m.step(2)
    f = m.get_fields()[0].reshape(r.M.shape)
    m.close()
    scale = np.array([np.abs(r.M[0]).max(), np.hypot(r.M[1], r.M[2]).max(), np.hypot(r.M[1], r.M[2]).max(),
                      np.abs(r.M[3]).max()])
    assert (np.abs(f - r.M).max(axis=(1, 2)) / scale).max() < 1e-12
