"""Device memory of handles and batches: what a solve's state takes, and nothing
beside it that grows.  A node of a float64 solve: two population buffers of 18
values, two of 4 moments and 4 of staging, 384 bytes (without the departure
cache)."""
import numpy as np
import pytest

from paper_2107_01370_gb300 import inputs

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def L():
    from paper_2107_01370_gb300 import build, lbfsi
    build.build()
    lbfsi.load()
    return lbfsi


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _case(nr, nt):
    case = inputs.cylinder_case(nr, nt, r_far=max(8.0, 1.3 * nr * np.pi / nt))
    return case, inputs.initial_field(nr, nt, case.flow, seed=1)


def test_fp64_handle_holds_two_population_buffers(L, monkeypatch):
    monkeypatch.setenv("LBFSI_NO_DEPARTURE_CACHE", "1")
    case, M0 = _case(1024, 256)
    nb, N = 2, 1024 * 256
    for k in range(2):                    # (the first handle also loads the kernels)
        before = _free()
        m = L.Mesh(case.r, case.e, case.bodies * nb, precision=L.FP64)
        m.init_fields(case.flow, np.ascontiguousarray(np.broadcast_to(M0, (nb,) + M0.shape)))
        m.step(2)
        m.synchronize()
        took = before - _free()
        m.close()
    assert took <= 384 * N * nb + 16 * MB


def test_fp64_views_follow_the_state_from_the_start(L):
    """What is written through the populations' view before the first step is
    what the step streams."""
    import torch
    case, M0 = _case(24, 32)
    out = []
    for scale in (1.0, 1.0 + 2.0 ** -8):
        m = L.Mesh(case.r, case.e, case.bodies, precision=L.FP64)
        m.init_fields(case.flow, M0[None])
        p = torch.as_tensor(m.field_view(L.FIELD_POPULATIONS), device="cuda")
        f0 = m.get_populations(0)[0]
        assert np.array_equal(p[..., 0].cpu().numpy().reshape(f0.shape), f0)
        p *= scale                        # (density and energy alike: the velocity and T stay)
        torch.cuda.synchronize()
        m.step(1)
        out.append((m.get_fields()[0], m.get_populations(0)[0]))
        m.close()
    rho = out[1][0][0][4:-4] / out[0][0][0][4:-4]      # off the wall and far field, whose targets are moments
    assert np.abs(rho - (1.0 + 2.0 ** -8)).max() < 1e-12
