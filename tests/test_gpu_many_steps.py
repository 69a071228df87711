"""Many steps in one launch against the same steps launched one by one: bit for bit the
same state, mesh, field, histories and scalars, where the two can part: one block and many,
meshes of 2 to 4096 cells (more and fewer cells than threads), partial items, open sheets,
weights per tracer, every deposit, the ring of history rows wrapping, a mode history, more
steps than one launch takes, and a hold (refinement, strict mode) in the middle.  Equality
is the tolerance: both are integer sums and the same order of FP32 sums."""
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


def _tiny(seed, sheets, tracers, nx):
    return inputs.tiny_problem(seed, n_sheets=sheets, max_tracers=tracers, nx=nx, L=1.0, dt=0.02, vscale=0.2)


PROBLEMS = {
    "two tracers, two cells": lambda: inputs.tiny_problem(4, 1, 2, 2, L=1.0, dt=0.01, vscale=0.1),
    "one block": lambda: _tiny(5, 3, 900, 37),
    "one block more": lambda: inputs.langmuir(n_tracers=4097, nx=64, n_steps=40),
    "ragged": lambda: _tiny(6, 40, 3000, 300),
    "fewer tracers than cells": lambda: _tiny(7, 6, 300, 4096),
    "more items than warps": lambda: inputs.landau(0.3, 0.5, 512, 330, 2300, t_end=1.0),
    "several rounds of items": lambda: inputs.landau(0.3, 0.5, 200, 1200, 1999, t_end=1.0),
}


def _all(sim, rows, mode):
    x, v = sim.sic_get_state()
    d = sim.sic_diagnostics()
    out = [x, v, sim.sic_history(rows), sim.sic_field(), np.array([d[k] for k in sorted(d)])]
    if mode:
        out.append(sim.sic_mode_history(rows))
    out.append(sim.sic_deposit()[0])
    return out


def _same(a, b):
    for p, q in zip(a, b):
        np.testing.assert_array_equal(p, q)


@pytest.mark.parametrize("order", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_many_steps_equal_single_ones(sic, name, order):
    p = PROBLEMS[name]()
    mode = 1 if p.nx >= 2 else 0
    got = []
    for many in (True, False):
        sim = sic.Sim.from_problem(p, history_len=5, order=order, mode_k=mode)
        try:
            if many:
                sim.sic_step(3)
                sim.sic_step(2)
                sim.sic_step(7)
            else:
                for _ in range(12):
                    sim.sic_step(1)
            got.append(_all(sim, 5, mode))
        finally:
            sim.sic_destroy()
    _same(*got)


def test_more_steps_than_one_launch_takes(sic):
    p = inputs.landau(0.05, 0.5, 64, 20, 700, dt=0.01, t_end=6.0)
    got = []
    for many in (True, False):
        sim = sic.Sim.from_problem(p, history_len=600)
        try:
            if many:
                sim.sic_step(515)
            else:
                for _ in range(515):
                    sim.sic_step(1)
            got.append(_all(sim, 600, 0))
        finally:
            sim.sic_destroy()
    _same(*got)


@pytest.mark.parametrize("kind", ["refine", "below a cell", "strict"])
def test_a_hold_stops_at_the_same_step(sic, kind):
    p = inputs.two_stream(2.4, 0.1, 0.2, 128, 32, 600, eps=0.3, dt=0.1, t_end=60.0)
    kw = dict(refine=0.0 if kind == "strict" else 0.02 * p.L if kind == "refine" else 0.5 * p.L / p.nx,
              strict=kind == "strict")
    got = []
    for many in (True, False):
        sim = sic.Sim.from_problem(p, history_len=700, **kw)
        try:
            n = 600
            try:
                if many:
                    sim.sic_step(n)
                else:
                    for _ in range(n):
                        sim.sic_step(1)
                x, v = sim.sic_get_state()
                d = sim.sic_diagnostics()
                assert 0 < d["step"] < n
                got.append([x, v, sim.sic_history(700), np.array([d[k] for k in sorted(d)])])
            except sic.SicError as e:
                assert kind == "strict" and e.code == sic.SIC_ESEGMENT_LONG
                got.append([np.array(e.code)])
        finally:
            sim.sic_destroy()
    _same(*got)
