"""Piecewise-linear particles of two cells each (quiet sheets: a lane takes its own) against
the same particles beside long ones (all cells are dealt over the warp): an open sheet, a
point, then long particles, against the sheet up to the point and the rest as sheets of
their own.  The point takes the gradient off both its neighbours, as an open end does, so
the charges are the same integers and add up exactly.  Up to 32 crossing particles (one
pass of a warp), forwards and backwards, around the periodic edge, one charge for all and
one per tracer."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sic():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1506_07207_gb300 import sic as binding
    return binding


def _mesh(sic, nx, L, x, w):
    sim = sic.Sim.sic_create(nx, L, 1e-3, [x.size], [0], [0], x, np.zeros(x.size), w, half_step_init=False, order=1,
                             charge_unit=2.0 ** -27)
    try:
        return sim.sic_deposit()[0]
    finally:
        sim.sic_destroy()


@pytest.mark.parametrize("per_tracer", [False, True])
@pytest.mark.parametrize("back", [False, True])
@pytest.mark.parametrize("quiet", [3, 12, 24, 28])
def test_pairs_equal_dealt_ones(sic, quiet, back, per_tracer):
    nx, L = 40, 1.0
    for seed in range(8):
        rng = np.random.default_rng(100 * quiet + seed)
        lengths = np.concatenate([0.55 + 0.4 * rng.random(quiet), [0.0], 2.2 + 3.0 * rng.random(4)])  # cells
        x = (rng.random() * nx + np.concatenate([[0.0], np.cumsum(lengths)])) * (L / nx) * (-1.0 if back else 1.0)
        w = 0.5 + rng.random(x.size) if per_tracer else np.ones(x.size)
        whole = _mesh(sic, nx, L, x, w)
        parts = _mesh(sic, nx, L, x[:quiet + 1], w[:quiet + 1]) + _mesh(sic, nx, L, x[quiet:], w[quiet:])
        np.testing.assert_array_equal(whole, parts)
