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


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_batch_allocates_nothing_after_its_creation(L, precision):
    """Solves of growing size admitted, stepped, read and removed one at a time
    (tile tables and kernels aside)."""
    prec = L.FP32 if precision == "fp32" else L.FP64
    cases = [_case(nr, nt) for nr, nt in (((128, 64), (512, 512), (2048, 1100), (2304, 1100)) if precision == "fp32"
                                          else ((128, 64), (512, 256), (768, 512)))]
    for k in range(2):                    # (the first batch also loads the kernels)
        b = L.Batch(640 * MB, precision=prec)
        before = _free()
        for case, M0 in cases:
            s = b.add(case.r, case.e, case.bodies[0], case.flow, 2, M0)
            b.step(2)
            assert np.isfinite(b.get(s)[0]).all()
            b.remove(s)
        took = before - _free()
        b.close()
    assert took <= 8 * MB


def test_batch_reads_do_not_disturb_the_run(L):
    """A float solve read between steps ends where one read at the end does."""
    case, M0 = _case(48, 64)
    got = []
    for reads in (False, True):
        b = L.Batch(64 * MB, precision=L.FP32)
        s = b.add(case.r, case.e, case.bodies[0], case.flow, 9, M0)
        if reads:
            b.get(s)
        for _ in range(9):
            b.step(1)
            if reads:
                b.get(s)
        f, loads, state = b.get(s)
        got.append((f, loads, state))
        b.close()
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1]) and got[0][2] == got[1][2]


@pytest.mark.parametrize("precision,node", [("fp32", 208), ("fp64", 384)])
def test_handle_runs_where_only_its_state_fits(L, precision, node):
    """With room for the populations, moments and staging alone (node bytes a
    node) a handle is made and gives the bits it gives with room to spare: the
    departure cache and the float correction field's buffer are left out."""
    import torch
    prec = L.FP32 if precision == "fp32" else L.FP64
    case, M0 = _case(4096, 1024)
    N = 4096 * 1024

    def run():
        m = L.Mesh(case.r, case.e, case.bodies, precision=prec)
        m.init_fields(case.flow, M0[None])
        m.step(1)
        m.step(1)
        f = m.get_fields()                # (float: through the staging)
        m.step(1)
        m.step(1)
        f = m.get_fields()
        m.close()
        return f

    want = run()
    torch.cuda.empty_cache()
    hold = torch.empty(_free() - node * N - 16 * MB, dtype=torch.uint8, device="cuda")
    try:
        got = run()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.array_equal(want, got)
