"""Reading a member of a batch while its steps are in flight: the members after the first
have streams of their own, which nothing orders after the batch's steps.  What such a read
returns is of no certain step, but the steps must not notice it: states, fields, histories
and charges equal those of simulations that nobody read, bit for bit (integer sums, the
same order of FP32 sums)."""
import threading

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


# several blocks each (more than 8 items), so that the blocks of a member meet in the L2:
# one item a warp and several, one charge per sheet and one per tracer
def _problems():
    return [inputs.landau(0.1, 0.4, 128, 32, 1000, t_end=1.0),
            inputs.landau(0.2, 0.5, 96, 64, 1500, t_end=1.0),
            inputs.two_stream(1.5, 0.2, 0.3, 300, 300, 4000, t_end=1.0),
            inputs.tiny_problem(12, n_sheets=24, max_tracers=2500, nx=64, L=1.0, dt=0.001, vscale=0.2)]


READS = {
    "field": lambda s: s.sic_field(),
    "density spectrum": lambda s: s.sic_spectrum(0),
    "field spectrum": lambda s: s.sic_spectrum(1),
    "moments": lambda s: s.sic_moments(0),
    "first-order moments": lambda s: s.sic_moments(1),
}
CALLS, STEPS = 12, 40


def _final(sims):
    out = []
    for s in sims:
        out.append((*s.sic_get_state(), s.sic_field(), s.sic_history(32),
                    np.array([s.sic_diagnostics()["charge_fixed"]]), s.sic_deposit()[0]))
    return out


@pytest.fixture(scope="module")
def unread(sic):
    sims = [sic.Sim.from_problem(p, history_len=32) for p in _problems()]
    for s in sims:
        s.sic_step(CALLS * STEPS)
    out = _final(sims)
    for s in sims:
        s.sic_destroy()
    return out


def _check(sic, unread, read, threaded):
    sims = [sic.Sim.from_problem(p, history_len=32) for p in _problems()]
    b = sic.Batch(sims)
    try:
        stop = threading.Event()

        def reader():
            while not stop.is_set():
                for s in sims[1:]:
                    read(s)
        t = threading.Thread(target=reader) if threaded else None
        if t:
            t.start()
        try:
            for _ in range(CALLS):
                b.sic_batch_step(STEPS)
                if not threaded:
                    for s in sims[1:]:
                        read(s)
            sims[0].sic_sync()
        finally:
            stop.set()
            if t:
                t.join()
        b.sic_batch_destroy()
        for got, want in zip(_final(sims), unread):
            for p, q in zip(got, want):
                np.testing.assert_array_equal(p, q)
    finally:
        b.sic_batch_destroy()
        for s in sims:
            s.sic_destroy()


@pytest.mark.parametrize("threaded", [False, True])
@pytest.mark.parametrize("name", sorted(READS))
def test_reading_a_member_leaves_its_steps_alone(sic, unread, name, threaded):
    _check(sic, unread, READS[name], threaded)
