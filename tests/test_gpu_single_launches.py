"""Steps on a stream that is being captured: any number of them goes into the capture, one
launch a step, and a replay advances the simulation (or the batch) by as many, bit for bit
as sic_step does (integer sums, the same order of FP32 sums)."""
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


def _problems():
    return [inputs.langmuir(n_tracers=900, nx=64),
            inputs.landau(0.1, 0.4, 128, 32, 3000, t_end=1.0),
            inputs.tiny_problem(12, n_sheets=4, max_tracers=2000, nx=64, L=1.0, vscale=0.5, dt=0.01)]


def _all(sim):
    return (*sim.sic_get_state(), sim.sic_history(64), sim.sic_field(), sim.sic_deposit()[0])


@pytest.mark.parametrize("steps", [1, 3, 8, 19])
@pytest.mark.parametrize("batch", [False, True])
def test_captured_steps_equal_plain_ones(sic, steps, batch):
    import torch
    stream = torch.cuda.Stream()
    plain = [sic.Sim.from_problem(p, history_len=64) for p in _problems()]
    sims = [sic.Sim.from_problem(p, history_len=64, stream=stream.cuda_stream) for p in _problems()]
    b = sic.Batch(sims) if batch else None
    step = (lambda n: b.sic_batch_step(n)) if batch else (lambda n: [s.sic_step(n) for s in sims])
    try:
        step(1)
        step(9)  # (and once through the ways that are not captured)
        for s in sims:
            s.sic_sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            step(steps)
        with torch.cuda.stream(stream):
            g.replay()
            g.replay()
        torch.cuda.synchronize()
        step(2)
        for s, p in zip(sims, plain):
            p.sic_step(12 + 2 * steps)
            for x, y in zip(_all(s), _all(p)):
                np.testing.assert_array_equal(x, y)
    finally:
        if b:
            b.sic_batch_destroy()
        for s in sims + plain:
            s.sic_destroy()
