"""The box deposit of short items, whose particles are dealt over the warp's lanes where most
of them cross a cell edge: a long sheet (full items, a lane's 8 tracers in order) against the
same sheet cut into sheets of 1 to 257 particles, around the sizes where the lanes and the
rule change (8, 32, 64, 96, 128), and closed sheets against open ones with the closing
particle written out.  Particles inside a cell, points, across one edge and many, on both
sides of the rule; one charge for all and one per tracer.  The charge is integers that do
not depend on how the work is cut: equality is the tolerance."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CUTS = [1, 2, 3, 7, 8, 9, 31, 32, 33, 63, 64, 65, 95, 96, 97, 126, 127, 128, 129, 130, 200, 255, 256, 257]


@pytest.fixture(scope="module")
def sic():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1506_07207_gb300 import sic as binding
    return binding


def _walk(n, step, L):
    """A sheet of n particles whose lengths are about `step`, back and forth, some points."""
    rng = np.random.default_rng(int(1e6 * step) + n)
    d = rng.normal(size=n) * step
    d[rng.random(n) < 0.05] = 0.0
    return 0.3 * L + np.concatenate([[0.0], np.cumsum(np.clip(d, -1.2 * L, 1.2 * L))])


def _mesh(sic, nx, L, sheets, closed):
    counts = [len(x) for x, _ in sheets]
    x, w = (np.concatenate([s[i] for s in sheets]) for i in (0, 1))
    flags = np.full(len(counts), int(closed))
    sim = sic.Sim.sic_create(nx, L, 1e-3, counts, flags, flags, x, np.zeros(x.size), w, half_step_init=False,
                             charge_unit=2.0 ** -27)
    try:
        return sim.sic_deposit()[0]
    finally:
        sim.sic_destroy()


@pytest.mark.parametrize("per_tracer", [False, True])
@pytest.mark.parametrize("nx,cells", [(5, 0.3), (64, 0.1), (64, 0.6), (64, 3.0), (300, 2.0), (300, 150.0), (4096, 2.5)])
def test_a_sheet_equals_its_pieces(sic, nx, cells, per_tracer):
    L = 2.0
    n = sum(CUTS)
    x = _walk(n, cells * L / nx, L)
    w = 0.5 + np.random.default_rng(3).random(n + 1) if per_tracer else np.ones(n + 1)
    ends = np.cumsum([0] + CUTS)
    pieces = [(x[a:b + 1], w[a:b + 1]) for a, b in zip(ends[:-1], ends[1:])]
    whole = _mesh(sic, nx, L, [(x, w)], False)
    np.testing.assert_array_equal(_mesh(sic, nx, L, pieces, False), whole)


@pytest.mark.parametrize("per_tracer", [False, True])
@pytest.mark.parametrize("nx,cells", [(5, 0.3), (64, 0.6), (300, 2.0)])
def test_a_closed_sheet_equals_its_open_one(sic, nx, cells, per_tracer):
    L = 2.0
    closed, opened = [], []
    rng = np.random.default_rng(9)
    for n in CUTS:
        if n < 2:
            continue
        x = np.linspace(0.0, L, n, endpoint=False) + rng.normal(size=n) * min(0.2 * L, cells * L / nx)
        w = 0.5 + rng.random(n) if per_tracer else np.ones(n)
        closed.append((x, w))
        opened.append((np.append(x, x[0] + L), np.append(w, w[0])))
    np.testing.assert_array_equal(_mesh(sic, nx, L, closed, True), _mesh(sic, nx, L, opened, False))
