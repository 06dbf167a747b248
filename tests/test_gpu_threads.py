"""Several threads reading one batch or handle at once each get what a single
reader gets (the calls release the interpreter's lock)."""
import threading

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


def _case(nr, nt, seed):
    body = inputs.BodySpec(dof=1, r_in=0.75, r_out=2.0, m_star=2.0 + seed, v_r=3.0 + seed)
    case = inputs.cylinder_case(nr, nt, r_far=8.0, body=body)
    return case, inputs.initial_field(nr, nt, case.flow, noise=1e-2, seed=seed)


def _run(jobs, times):
    """Each job in a thread of its own; the calls whose result differs."""
    wrong = []
    go = threading.Barrier(len(jobs))

    def work(k, call, same):
        go.wait()
        for n in range(times):
            if not same(call()):
                wrong.append((k, n))

    threads = [threading.Thread(target=work, args=(k, *j)) for k, j in enumerate(jobs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return wrong


@pytest.mark.parametrize("fields", [False, True])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_threads_read_different_slots(L, precision, fields):
    b = L.Batch(64 << 20, precision=L.FP32 if precision == "fp32" else L.FP64)
    slots = []
    for k, (nr, nt) in enumerate(((32, 32), (48, 64), (64, 96), (40, 48))):
        case, M0 = _case(nr, nt, k + 1)
        slots.append(b.add(case.r, case.e, case.bodies[0], case.flow, 10, M0))
    b.step(7)
    want = [b.get(s, fields=True) for s in slots]

    def job(k):
        def same(got):
            return ((not fields or np.array_equal(got[0], want[k][0])) and np.array_equal(got[1], want[k][1])
                    and got[2] == want[k][2])
        return lambda: b.get(slots[k], fields=fields), same
    wrong = _run([job(k) for k in range(len(slots))], 400 if not fields else 100)
    b.close()
    assert not wrong, (len(wrong), wrong[:3])


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_threads_read_one_handle(L, precision):
    case, M0 = _case(48, 64, 3)
    m = L.Mesh(case.r, case.e, case.bodies, precision=L.FP32 if precision == "fp32" else L.FP64)
    m.init_fields(case.flow, M0[None])
    m.step(7)
    F, S, M = m.body_forces(), m.body_state(), m.get_fields()
    jobs = [(m.body_forces, lambda g: np.array_equal(g, F)), (m.body_state, lambda g: g == S),
            (m.get_fields, lambda g: np.array_equal(g, M)), (m.synchronize, lambda g: True)]
    wrong = _run(jobs, 100)
    m.close()
    assert not wrong, (len(wrong), wrong[:3])
