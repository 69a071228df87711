"""The whole cells inside a box particle, where their charge changes its way: none, one or
two (straight into the mesh), three and more (a difference array), starting in every cell
of a small mesh and around the ends of the largest, so that the cells inside wrap; forwards
and backwards along the sheet; one charge per sheet and one per tracer; deposited from rest
and after a step that leaves the tracers where they are.

Every whole cell gets floor(q 2^32 / length) units (positions are dyadic, so the length in
2^-32 cells is exact) and nothing outside the particle gets any: both exact.  The first and
last cells share the rest; the first one's share is one FP32 product with a reciprocal of
relative error 2^-23: within 2^-21 of q."""
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


def _expected(nx, a, b, q):
    """(exact charges of the whole cells as {cell: units}, lower end's cell, its exact
    share, upper end's cell) of q units between a < b in cells."""
    span = int((b - a) * 2 ** 32)
    ja, jb = int(np.floor(a)), int(np.floor(b))
    P = q * 2 ** 32 // span if jb > ja else 0
    return {c % nx: P for c in range(ja + 1, jb)}, ja % nx, q * (ja + 1 - a) / (b - a), jb % nx


@pytest.mark.parametrize("per_tracer", [False, True])
@pytest.mark.parametrize("nx", [8, 8192])
def test_whole_cells_inside_a_particle(sic, nx, per_tracer):
    L = 1.0
    starts = range(nx) if nx == 8 else [0, 1, 4095, nx - 5, nx - 4, nx - 3, nx - 2, nx - 1]
    for start in starts:
        for inside in (0, 1, 2, 3, 4):
            for back in (False, True):
                a = start + 1.0 - 0.375                    # 0.375 of the first cell
                b = start + 1.0 + inside + 0.6875          # and 0.6875 of the last one
                x = np.array([a, b]) * (L / nx)
                if back:
                    x = x[::-1].copy()
                w = np.array([1.0, 0.7]) if per_tracer else np.ones(2)
                sim = sic.Sim.sic_create(nx, L, 1e-9, [2], [0], [0], x, np.zeros(2), w, half_step_init=False)
                try:
                    unit = sim.sic_diagnostics()["charge_unit"]
                    q = int(sum(np.floor(w / unit * 0.5 + 0.5)))
                    inner, lo, share, hi = _expected(nx, a, b, q)
                    meshes = [sim.sic_deposit()[0]]
                    for steps in (1, 2):
                        sim.sic_step(steps)
                        meshes.append(sim.sic_deposit()[0])
                    for mesh in meshes:
                        assert mesh.sum() == q
                        for c, P in inner.items():
                            assert mesh[c] == P, (start, inside, back, c)
                        assert set(np.flatnonzero(mesh)) <= set(inner) | {lo, hi}
                        assert abs(int(mesh[lo]) - share) <= q * 2.0 ** -21 + 1
                finally:
                    sim.sic_destroy()
