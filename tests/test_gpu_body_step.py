"""A body's step against RK4 in extended precision, from the recorded state
before it and the recorded load: the new state is the old one plus an increment,
so it may be off by the rounding of that sum (half an ulp) and by that of the
increment, some 16 roundings (2^-53) of the terms it sums (64 where sines of
the prescribed pitch enter, each to about an ulp of an angle's own rounding)."""
import numpy as np
import pytest

from oracle.solver import body_dict
from paper_2107_01370_gb300 import inputs

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def L():
    from paper_2107_01370_gb300 import build, lbfsi
    build.build()
    lbfsi.load()
    return lbfsi


def _increment(acc, y, dt):
    """RK4 increment of (x..., v...) under acc(stage, y)."""
    n = len(y) // 2
    k, out = None, np.zeros(len(y), LD)
    for s, (at, w) in enumerate(((0.0, 1.0), (0.5, 2.0), (0.5, 2.0), (1.0, 1.0))):
        z = y if k is None else y + LD(at) * dt * k
        k = np.concatenate([z[n:], acc(s, z)])
        out += LD(w) * k
    return dt / LD(6.0) * out


def _columns(acc_of, nc, size, dt):
    """The increment as a matrix: one column per unit entry of (y, loads...)."""
    cols = []
    for c in range(nc):
        e = np.zeros(nc, LD)
        e[c] = 1.0
        cols.append(_increment(acc_of(e[size:]), e[:size], dt))
    return np.stack(cols, axis=1)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["transverse", "pitch-plunge", "forced"])
def test_body_step_rounds_once(L, kind, precision):
    body = {"transverse": inputs.BodySpec(dof=1, r_in=0.75, r_out=2.0, m_star=3.0, v_r=5.0, zeta=0.02),
            "pitch-plunge": inputs.BodySpec(dof=2, xp=-0.2, r_in=0.75, r_out=2.0, m_star=8.0, v_r=1.5, x_alpha=0.3,
                                            r_alpha=0.5, wh_wa=0.5),
            "forced": inputs.BodySpec(dof=2, xp=-0.2, r_in=0.75, r_out=2.0, m_star=8.0, v_r=1.5, x_alpha=0.3,
                                      r_alpha=0.5, wh_wa=0.5, pitch_amp=0.05, forced_periods=100.0)}[kind]
    case = inputs.cylinder_case(24, 32, r_far=8.0, body=body)
    m = L.Mesh(case.r, case.e, case.bodies, precision=L.FP64 if precision == "fp64" else L.FP32)
    m.init_fields(case.flow, inputs.initial_field(24, 32, case.flow, seed=3)[None])
    start = (0.03, 0.0 if kind != "pitch-plunge" else 0.02, 0.01, 0.0 if kind != "pitch-plunge" else -0.015)
    if kind != "forced":
        m.blend_mesh([start], [start])
    else:
        start = (0.0, 0.0, 0.0, 0.0)
    steps = 60
    loads, states = m.step_record(steps, states=True)
    m.close()
    got = np.asarray(states).reshape(steps, 4)
    b = {k: LD(v) for k, v in body_dict(body, case.flow.rho_inf, case.flow.u_inf).items()}
    dt = LD(case.flow.dt)
    worst = 0.0
    if kind == "transverse":
        rows, C = (0, 2), _columns(lambda F: lambda s, z: np.array([(F[0] - b["k"] * z[0] - b["c"] * z[1]) / b["m"]]), 3, 2, dt)
    elif kind == "pitch-plunge":
        det = b["m"] * b["i_a"] - b["s_a"] ** 2

        def acc_of(F):
            def acc(s, z):
                r0, r1 = F[0] - b["k_h"] * z[0], F[1] - b["k_a"] * z[1]
                return np.array([(b["i_a"] * r0 - b["s_a"] * r1) / det, (b["m"] * r1 - b["s_a"] * r0) / det])
            return acc
        rows, C = (0, 1, 2, 3), _columns(acc_of, 6, 4, dt)
    else:
        rows, C = (0, 2), _columns(
            lambda F: lambda s, z: np.array([(F[0] - b["k_h"] * z[0] - b["s_a"] * F[(1, 2, 2, 3)[s]]) / b["m"]]), 6, 2, dt)
    for n in range(steps):
        old = np.array(start if n == 0 else got[n - 1], LD)
        F = np.array(loads[n], LD).reshape(3)
        if kind == "forced":
            w = b["w_a"]
            x = [F[1]] + [-body.pitch_amp * w * w * np.sin(w * dt * (n + LD(t))) for t in (0.0, 0.5, 1.0)]
        else:
            x = [F[1]] + ([F[2]] if kind == "pitch-plunge" else [])
        x = np.concatenate([old[list(rows)], np.array(x, LD)])
        want = old[list(rows)] + C @ x
        tol = LD(0.5) * np.spacing(np.abs(want).astype(np.float64)) + (64 if kind == "forced" else 16) * LD(2.0) ** -53 * (np.abs(C) @ np.abs(x))
        err = np.abs(got[n][list(rows)].astype(LD) - want)
        worst = max(worst, float((err / tol).max()))
    assert worst <= 1.0
