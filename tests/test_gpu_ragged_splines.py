"""Spline shapes in periodic boxes whose last tile is narrower than the stencil: a particle that has moved to the rows
next to it deposits across it, three tiles from the tile it started in.  All particles in one tile row (column),
moving about a tile a step, FP64 with the time-centred solve, whose moments are cleared tile by tile before each
push: nodes that the step's tile lists miss keep the previous step's moments.  Against the oracle with the parity
tolerances of the FP64 form."""
import numpy as np
import pytest

from paper_1308_2590_gb300 import workloads as W
from tests.parity import compare_grid, compare_particles, run_pair
from tests.test_gpu_parity import small_uniform

pytestmark = pytest.mark.gpu

TILE, LONG = 8, 6 * 8 + 1


@pytest.mark.parametrize("up", [True, False])
@pytest.mark.parametrize("axis", ["x", "y"])
@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("order", [1, 2, 3, 4])
def test_moments_beyond_a_narrow_last_tile(order, extra, axis, up):
    cfg = small_uniform(n=LONG + extra, ppc=1, tile=TILE)
    n_long = LONG + extra
    cfg.nx, cfg.ny = (n_long, 24) if axis == "x" else (24, n_long)
    cfg.shape = order
    n = 60
    rng = np.random.default_rng(order)
    c = cfg.dt / cfg.dx                       # cells a step at the speed of light
    v = 8.0 / c
    u = v / np.sqrt(1.0 - v * v)
    # upwards: from rows 38.6 .. 39.9 (tile 4) to the last rows of tile 5; downwards: from tile 1 to the first of tile 0
    along = (38.6 + 1.3 * rng.random(n)) if up else (8.1 + 1.3 * rng.random(n))
    across = 4.0 + 2.0 * rng.random(n)
    P = dict(x=along * cfg.dx if axis == "x" else across * cfg.dx, y=across * cfg.dy if axis == "x" else along * cfg.dy,
             ux=np.zeros(n), uy=np.zeros(n), uz=0.05 * rng.standard_normal(n), w=np.full(n, 1e-6))
    P["u" + axis][:] = u if up else -u
    parts = [P, {k: a[:0] for k, a in P.items()}]
    for steps in (1, 2, 3):
        g, o = run_pair(cfg, steps, parts=parts)
        compare_particles(g, o, cfg)
        compare_grid(g, o, rho_scale=float(np.max(np.abs(o.M[0]))))
        g.close()
