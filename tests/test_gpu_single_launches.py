"""Steps of one launch each, the way of simulations too large for launches of many steps, of
single steps and of streams under capture.  SIC_STEPS_A_LAUNCH=1 sends small simulations
that way too: claims, blocks that move from one simulation to the next or arrive late,
graphs of 8 steps and what is left of them, alone and in a batch, against launches of many
steps (and, at the largest mesh, whichever way it goes against single steps).  Steps on a
stream that is being captured go into the capture, and a replay takes them again.  All are
equal bit for bit (integer sums, the same order of FP32 sums)."""
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


@pytest.fixture
def one_step_a_launch(monkeypatch):
    monkeypatch.setenv("SIC_STEPS_A_LAUNCH", "1")
    return monkeypatch


def _mixed():
    """One charge per sheet and one per tracer, every deposit; 19 steps: two graphs of 8 and three."""
    return [(inputs.landau(0.1, 0.4, 128, 32, 3000, t_end=1.0), 0),
            (inputs.two_stream(1.5, 0.2, 0.3, 512, 16, 5000, t_end=1.0), 0),
            (inputs.langmuir(nx=100), 0),
            (inputs.tiny_problem(12, n_sheets=4, max_tracers=2000, nx=64, L=1.0, vscale=0.5), 0),
            (inputs.landau(0.1, 0.5, 96, 20, 700, t_end=1.0), 1),
            (inputs.landau(0.1, 0.5, 96, 20, 700, t_end=1.0), 2),
            (inputs.landau(0.1, 0.5, 96, 20, 700, t_end=1.0), 3),
            (inputs.landau(0.1, 0.5, 96, 20, 700, t_end=1.0), 4)]


def _launches(sic, f):
    n = sic.sic_launch_count()
    f()
    return sic.sic_launch_count() - n


@pytest.mark.parametrize("grid", ["", "1", "7", "33"])
def test_single_launches_alone_equal_many_steps(sic, one_step_a_launch, grid):
    for p, order in _mixed():
        got = []
        for knob in ("1", "256"):
            one_step_a_launch.setenv("SIC_STEPS_A_LAUNCH", knob)
            one_step_a_launch.setenv("SIC_GRID", grid if knob == "1" else "")
            sim = sic.Sim.from_problem(p, history_len=64, order=order)
            try:
                assert _launches(sic, lambda: sim.sic_step(19)) == (19 if knob == "1" else 1)
                got.append(_all(sim))
            finally:
                sim.sic_destroy()
        for x, y in zip(*got):
            np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("members", ["mixed", "one charge", "many small"])
def test_single_launches_of_a_batch_equal_many_steps_alone(sic, one_step_a_launch, members):
    if members == "many small":
        probs = [(inputs.tiny_problem(100 + i, n_sheets=2, max_tracers=300, nx=[16, 37, 64][i % 3], L=1.0, vscale=0.2), 0)
                 for i in range(40)]
        probs += [(inputs.landau(0.1, 0.5, 128, 64, 4096, t_end=1.0), 0),
                  (inputs.two_stream(1.5, 0.2, 0.3, 256, 32, 8192, t_end=1.0), 0)]
    else:
        probs = [q for q in _mixed() if members == "mixed" or (q[1] == 0 and q[0].name != "tiny12")]
    steps = 25
    one_step_a_launch.setenv("SIC_STEPS_A_LAUNCH", "256")
    alone = []
    for p, order in probs:
        sim = sic.Sim.from_problem(p, history_len=64, order=order)
        assert _launches(sic, lambda: sim.sic_step(steps)) == 1
        alone.append(_all(sim))
        sim.sic_destroy()
    one_step_a_launch.setenv("SIC_STEPS_A_LAUNCH", "1")
    sims = [sic.Sim.from_problem(p, history_len=64, order=order) for p, order in probs]
    b = sic.Batch(sims)
    try:
        modes = 1 if members == "one charge" else 2
        assert _launches(sic, lambda: b.sic_batch_step(steps)) == steps * modes
        b.sic_batch_destroy()
        for s, want in zip(sims, alone):
            assert s.sic_diagnostics()["step"] == steps
            for x, y in zip(_all(s), want):
                np.testing.assert_array_equal(x, y)
    finally:
        b.sic_batch_destroy()
        for s in sims:
            s.sic_destroy()


def test_single_launches_with_step_counts_of_their_own(sic, one_step_a_launch):
    """sic_step_batch: members that leave the launches one after the other."""
    counts = [25, 3, 8, 0, 19, 1, 8, 24]
    got = []
    for knob in ("1", "256"):
        one_step_a_launch.setenv("SIC_STEPS_A_LAUNCH", knob)
        sims = [sic.Sim.from_problem(p, history_len=64, order=order) for p, order in _mixed()]
        try:
            sic.sic_step_batch(sims, counts)
            got.append([_all(s) for s in sims])
        finally:
            for s in sims:
                s.sic_destroy()
    for a, b in zip(*got):
        for x, y in zip(a, b):
            np.testing.assert_array_equal(x, y)


def test_the_server_takes_single_launches(sic, one_step_a_launch):
    """Served requests, refining as they fold, one launch a step and many."""
    probs = [r.problem() for r in inputs.serving_mix(n_requests=12, seed=77, max_sheets_exp=6, max_tracers_exp=11,
                                                     max_nx_exp=8)]
    got = []
    for knob in ("1", "256"):
        one_step_a_launch.setenv("SIC_STEPS_A_LAUNCH", knob)
        server = sic.Server(hbm_budget=1 << 30, max_active=5, chunk_steps=32)
        try:
            for p in probs:
                server.sic_server_submit_horizontal(p, n_steps=min(p.n_steps, 260), keep=True, history_len=64)
            while server.sic_server_tick():
                pass
            out = []
            for q, p in zip(sorted(server.sic_server_results(), key=lambda q: q["id"]), probs):
                out.append(np.array([q["status"], q["steps"], q["segment_updates"], q["charge_fixed"]]))
                out.append(np.array([q["field_energy"], q["kinetic_energy"], q["momentum"]]))
                sim = sic.adopt_sim(q["sim"], p.nx, p.counts)
                out += [sim.sic_history(64), sim.sic_field()]
                sim.sic_destroy()
            got.append(out)
        finally:
            server.sic_server_destroy()
    assert len(got[0]) == len(got[1]) == 4 * len(probs)
    for x, y in zip(*got):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("nx", [2049, 4096, 8192])
@pytest.mark.parametrize("knob", ["256", "1"])
def test_large_meshes_take_many_steps(sic, one_step_a_launch, knob, nx):
    """19 steps at once and one by one, alone and in a batch of two."""
    probs = [inputs.tiny_problem(77, n_sheets=4, max_tracers=9000, nx=nx, L=3.0, spread=0.05),
             inputs.landau(0.1, 0.5, nx, 24, 3000, t_end=1.0)]
    one_step_a_launch.setenv("SIC_STEPS_A_LAUNCH", knob)
    ones, alls, members = ([sic.Sim.from_problem(p, history_len=32) for p in probs] for _ in range(3))
    try:
        for s in ones:
            for _ in range(19):
                s.sic_step(1)
        for s in alls:
            s.sic_step(19)
        b = sic.Batch(members)
        b.sic_batch_step(19)
        b.sic_batch_destroy()
        for s, t, m in zip(ones, alls, members):
            want = _all(s)
            for got in (_all(t), _all(m)):
                for x, y in zip(got, want):
                    np.testing.assert_array_equal(x, y)
    finally:
        for s in ones + alls + members:
            s.sic_destroy()


def test_autotune_times_launches_of_many_steps_too(sic, one_step_a_launch):
    """A small batch (its steps are launch latencies, so that many to a launch take half
    the time): the launches of many steps are one of the candidates, in one launch each for
    the untimed and the timed steps, and stay.  A batch that does not take them times
    schedules only.  Both advance by the same steps, to the same bits."""
    probs = [inputs.landau(0.1, 0.4, 64, 16, 300, dt=1e-3), inputs.landau(0.1, 0.5, 128, 8, 600, dt=1e-3)]
    n, each = sic.SIC_AUTOTUNE_CANDIDATES, 100  # (0.6 and 1.2 ms: far more than a hiccup of the host)
    got = []
    for knob in ("256", "1"):
        one_step_a_launch.setenv("SIC_STEPS_A_LAUNCH", knob)
        sims = [sic.Sim.from_problem(p, history_len=300) for p in probs]
        b = sic.Batch(sims)
        try:
            tuned = _launches(sic, lambda: b.sic_batch_autotune(each))
            assert tuned == ((n - 1) * (each + 1) + 2 if knob == "256" else n * (each + 1))
            assert _launches(sic, lambda: b.sic_batch_step(12)) == (1 if knob == "256" else 12)
            b.sic_batch_destroy()
            assert all(s.sic_diagnostics()["step"] == n * (each + 1) + 12 for s in sims)
            got.append([(*s.sic_get_state(), s.sic_history(300)) for s in sims])
        finally:
            b.sic_batch_destroy()
            for s in sims:
                s.sic_destroy()
    for a, b in zip(*got):
        for x, y in zip(a, b):
            np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("members,rounds", [(1, 9), (1, 12), (4, 5), (4, 7)])
@pytest.mark.parametrize("nx", [3000, 4096])
def test_the_rule_on_rounds_of_items(sic, nx, members, rounds):
    """Where an SM holds one block of a launch of many steps and two of single steps (4096
    cells), fewer rounds of items (one per warp) go to launches of many steps; on 3000
    cells it holds two of each.  Either way: the steps of single launches."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    warps = 8 * sms * (2 if nx == 3000 else 1)
    sheets = int((rounds - 0.4) * warps / members) // 8        # of 8 items each
    p = inputs.landau(0.01, 0.5, nx, sheets, 2048, t_end=1.0)
    ones, many = ([sic.Sim.from_problem(p, history_len=16) for _ in range(members)] for _ in range(2))
    b = sic.Batch(many) if members > 1 else None
    try:
        step = b.sic_batch_step if b else many[0].sic_step
        takes_many = nx == 3000 or rounds <= (10 if members == 1 else 6)
        assert _launches(sic, lambda: step(9)) == (1 if takes_many else 9)
        if b:
            b.sic_batch_destroy()
        for s, t in zip(many, ones):
            for _ in range(9):
                t.sic_step(1)
            np.testing.assert_array_equal(s.sic_history(16), t.sic_history(16))
            np.testing.assert_array_equal(s.sic_deposit()[0], t.sic_deposit()[0])
    finally:
        if b:
            b.sic_batch_destroy()
        for s in ones + many:
            s.sic_destroy()
