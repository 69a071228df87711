"""Piecewise-linear particles of items that a resident launch keeps in shared memory: the
tracers are written back there by whole lanes (8 words each) and the last lane publishes
the tracers after the item behind them, so the counts that matter are those where these
words belong to the next lane (0 and 7 modulo 8), beside full items and their neighbours.
Many steps in one launch equal the same steps one by one, bit for bit (integer charge, the
same order of FP32 sums)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

COUNTS = [7, 8, 15, 16, 248, 255, 256]


@pytest.fixture(scope="module")
def sic():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1506_07207_gb300 import sic as binding
    return binding


def _sheets(times, closed, per_tracer):
    rng = np.random.default_rng(5)
    L = 2.0
    counts = np.array(COUNTS * times, dtype=np.int32)
    x, v, w = [], [], []
    for n in counts:
        i = np.arange(n)
        x.append(rng.random() * L + L * i / n * (1.0 if closed else 0.9) + (rng.random(n) - 0.5) * L * min(0.3, 4.0 / n))
        v.append((rng.random(n) - 0.5) * 0.1)
        w.append((0.5 + rng.random(n) if per_tracer else np.full(n, 1.0)) * L / n)
    return L, counts, np.full(counts.size, int(closed)), np.full(counts.size, int(closed)), *map(np.concatenate, (x, v, w))


# (with the longer step some of these runs leave the position format, as they do in the
# oracle: piecewise-linear particles have no limiter.  Both sides then end with that error.)
@pytest.mark.parametrize("dt", [0.02, 0.001])
@pytest.mark.parametrize("order", [1, 4])
@pytest.mark.parametrize("per_tracer", [0, 1])
@pytest.mark.parametrize("closed", [0, 1])
@pytest.mark.parametrize("times", [1, 40])
def test_kept_items_equal_single_steps(sic, times, closed, per_tracer, order, dt):
    L, counts, cl, wd, x, v, w = _sheets(times, closed, per_tracer)
    got = []
    for many in (True, False):
        sim = sic.Sim.sic_create(100, L, dt, counts, cl, wd, x, v, w, half_step_init=False, history_len=32, order=order)
        try:
            for _ in range(1 if many else 24):
                sim.sic_step(24 if many else 1)
            got.append([*sim.sic_get_state(), sim.sic_field(), sim.sic_history(32), sim.sic_deposit()[0]])
        except sic.SicError as e:
            assert dt == 0.02 and order == 1 and e.code == sic.SIC_ERANGE
            got.append([np.array(e.code)])
        finally:
            sim.sic_destroy()
    assert len(got[0]) == len(got[1])
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
