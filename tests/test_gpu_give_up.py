"""A block of a resident launch that gives up waiting for its group (SIC_WAIT_POLLS makes
its bounded wait short): the simulation ends with SIC_ETIMEOUT, now and at every later
call, and nothing else is affected.  A block that gave up has not written its tracers, so
whether or not the others completed the step, no call may report success on a state that
is not the one of single steps."""
import numpy as np
import pytest

from paper_1506_07207_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sic():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1506_07207_gb300 import sic as binding
    return binding


def _p(i=0):
    # 4 to 13 blocks, one item a warp: kept in shared memory until the last step
    return inputs.landau(0.1, 0.4 + 0.01 * i, 64 + 32 * (i % 3), 16 + 12 * (i % 4), 300, t_end=10.0)


def _code(sic, call):
    try:
        call()
        return sic.SIC_OK
    except sic.SicError as e:
        return e.code


def test_the_error_stays(sic, monkeypatch):
    monkeypatch.setenv("SIC_WAIT_POLLS", "1")
    sim = sic.Sim.from_problem(_p(3), history_len=4)
    try:
        monkeypatch.delenv("SIC_WAIT_POLLS")  # (read when the simulation's plan was built)
        sim.sic_step(200)
        for call in (sim.sic_sync, sim.sic_field, sim.sic_get_state, sim.sic_diagnostics):
            assert _code(sic, call) == sic.SIC_ETIMEOUT
        sim.sic_step(50)
        assert _code(sic, sim.sic_sync) == sic.SIC_ETIMEOUT
    finally:
        sim.sic_destroy()
    # the device is none the worse for it
    a, b = (sic.Sim.from_problem(_p(3), history_len=4) for _ in range(2))
    try:
        a.sic_step(20)
        for _ in range(20):
            b.sic_step(1)
        for p, q in zip(a.sic_get_state(), b.sic_get_state()):
            np.testing.assert_array_equal(p, q)
    finally:
        a.sic_destroy()
        b.sic_destroy()


def test_no_success_without_every_block(sic, monkeypatch):
    """One step a launch, so that the last step is where blocks give up: the recorder may
    have seen the count complete after another block's last poll."""
    probs = [_p(i) for i in range(32)]
    want = []
    for p in probs:
        sim = sic.Sim.from_problem(p, history_len=4)
        sim.sic_step(1)
        want.append(sim.sic_get_state())
        sim.sic_destroy()
    sims = [sic.Sim.from_problem(p, history_len=4) for p in probs]
    monkeypatch.setenv("SIC_WAIT_POLLS", "1")
    b = sic.Batch(sims)
    try:
        b.sic_batch_step(1)
        codes = [_code(sic, s.sic_sync) for s in sims]
        assert set(codes) <= {sic.SIC_OK, sic.SIC_ETIMEOUT}
        for s, c, w in zip(sims, codes, want):
            if c == sic.SIC_OK:
                for p, q in zip(s.sic_get_state(), w):
                    np.testing.assert_array_equal(p, q)
        b.sic_batch_step(1)  # those that gave up hold
        assert all(_code(sic, s.sic_sync) == sic.SIC_ETIMEOUT for s, c in zip(sims, codes) if c)
    finally:
        b.sic_batch_destroy()
        for s in sims:
            s.sic_destroy()
