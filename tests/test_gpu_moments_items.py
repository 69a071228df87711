"""sic_moments where its split of the work can go wrong: sheets that end before, on and
after a lane's 8 tracers and a warp's 256, open and closed, with one weight per sheet and
one per tracer, particles inside a cell, points, and particles of many cells (shared out
over a warp) up to more than a box, on meshes of 2 to 8192 cells, against the FP64 oracle
on the same state.

Tolerance: both sides are FP64 on the same positions, velocities and fixed-point charges
(the weights rounded to whole half units of sic_diagnostics' charge_unit, as sic.h states),
so n agrees within 1e-8 of max |n| and j within 1e-8 of max |n| max |v| (the bounds of
test_gpu_moments_pic.py)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sic():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1506_07207_gb300 import sic as binding
    return binding


def _sheets(per_tracer, L):
    rng = np.random.default_rng(17 + per_tracer)
    counts = np.array([2, 3, 7, 8, 9, 255, 256, 257, 263, 264, 512, 513, 1000, 2, 40], dtype=np.int32)
    closed = np.array([1, 0, 1, 0, 1, 0, 1, 0, 1, 1, 0, 1, 1, 0, 1], dtype=np.uint8)
    winding = np.where(closed == 1, np.array([1, 0, -1, 0, 1, 0, 1, 0, 0, 1, 0, 1, 1, 0, 1]), 0).astype(np.int32)
    x, v, w = [], [], []
    for s, n in enumerate(counts):
        i = np.arange(n)
        base = rng.random() * L + (winding[s] if winding[s] else 0.9 * (closed[s] == 0)) * L * i / n
        base = base + (rng.random(n) - 0.5) * L * min(0.4, 8.0 / n)
        if n > 5:
            base[4] = base[3]                       # a point
        if s == 13:
            base = np.array([0.25, 0.25 + 1.3]) * L  # longer than the box
        x.append(base)
        v.append(rng.normal(size=n) * 0.1)
        w.append((0.5 + rng.random(n) if per_tracer else np.full(n, 0.5 + rng.random())) * L / n)
    return counts, closed, winding, np.concatenate(x), np.concatenate(v), np.concatenate(w)


@pytest.mark.parametrize("weighting", [0, 1])
@pytest.mark.parametrize("nx", [2, 37, 512, 8192])
@pytest.mark.parametrize("per_tracer", [0, 1])
def test_moments_at_the_edges_of_the_work_split(sic, weighting, nx, per_tracer):
    L = 3.0
    counts, closed, winding, x, v, w = _sheets(per_tracer, L)
    sim = sic.Sim.sic_create(nx, L, 0.01, counts, closed, winding, x, v, w, half_step_init=False)
    try:
        n, j = sim.sic_moments(weighting)
        xs, vs = sim.sic_get_state()
        unit = sim.sic_diagnostics()["charge_unit"]
    finally:
        sim.sic_destroy()
    w = np.floor(w / (2 * unit) + 0.5) * 2 * unit
    n_ref, j_ref = oracle.moments(nx, L, counts, closed, winding, xs, vs, w, weighting)
    scale = np.abs(n_ref).max()
    np.testing.assert_allclose(n, n_ref, rtol=0, atol=1e-8 * scale)
    np.testing.assert_allclose(j, j_ref, rtol=0, atol=1e-8 * scale * np.abs(vs).max())


def test_a_state_is_the_same_after_moments(sic):
    """The moments' copies lie in the buffers that the next step writes: stepping on after
    them gives the same bits as without, on a mesh that takes many copies."""
    L = 3.0
    counts, closed, winding, x, v, w = _sheets(0, L)
    got = []
    for with_moments in (False, True):
        sim = sic.Sim.sic_create(37, L, 0.01, counts, closed, winding, x, v, w, half_step_init=False)
        try:
            for steps in (1, 2, 1):
                if with_moments:
                    sim.sic_moments(0)
                    sim.sic_moments(1)
                sim.sic_step(steps)
            got.append((*sim.sic_get_state(), sim.sic_field()))
        finally:
            sim.sic_destroy()
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
