"""Field kernels at the sizes where their strips, columns and ghost images change: sides below the ghost
ring, at and around the 30 columns a warp produces, rows at and around a strip's, periodic and walled boxes.
Random fields and a warm plasma over part of the box (touched and vacuum tiles): fields,
moments and particles against the oracle with the parity tolerances (1e-10, 1e-9)."""
import numpy as np
import pytest

from paper_1308_2590_gb300 import workloads as W
from tests.parity import compare_grid, compare_particles, density_scale, run_pair
from tests.test_gpu_parity import hot, small_uniform

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(2, 2), (2, 5), (5, 2), (3, 3), (29, 7), (30, 8), (31, 9), (60, 33), (61, 4),
                                   (90, 31), (33, 130)])
@pytest.mark.parametrize("field_mode", [W.FIELD_LITERAL, W.FIELD_CN])
@pytest.mark.parametrize("bc", [W.BC_PERIODIC, W.BC_ABSORBING])
def test_sizes(nx, ny, field_mode, bc):
    cfg = hot(small_uniform(ppc=2, tile=4, field_mode=field_mode, dt=0.05), 1.0).scaled(nx=nx, ny=ny, bc_x=bc)
    if nx >= 29:
        cfg.slab = (nx // 3, nx // 3 + 5)
    rng = np.random.default_rng(nx * 1000 + ny)
    nxn = nx if bc == W.BC_PERIODIC else nx + 1
    E, H = 0.1 * rng.standard_normal((3, ny, nxn)), 0.1 * rng.standard_normal((3, ny, nx))
    g, o = run_pair(cfg, 3, fields=(E, H))
    compare_particles(g, o, cfg)
    compare_grid(g, o, rho_scale=density_scale(cfg))
    g.close()
