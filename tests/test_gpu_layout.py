"""Layout of the bins over numbers of tiles around the parts its blocks take (8 tiles a thread, 8 blocks) and above
what they hold in one round, particles spread over the tiles or crowded in few of them: the particle order against the
oracle's and its moments within the parity tolerance (1e-9)."""
import numpy as np
import pytest

from paper_1308_2590_gb300 import workloads as W
from tests.parity import compare_particles, normwise, run_pair
from tests.test_gpu_parity import hot, small_uniform

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(2, 2), (9, 7), (8, 8), (13, 5), (64, 8), (513, 2), (300, 260)])
@pytest.mark.parametrize("dense", [False, True])
def test_tiles(nx, ny, dense):
    cfg = hot(small_uniform(ppc=1, tile=1, field_mode=W.FIELD_LITERAL, dt=0.05), 1.0).scaled(nx=nx, ny=ny)
    rng = np.random.default_rng(nx + ny)
    n = 3 * nx * ny
    parts = []
    for _ in cfg.species:
        x, y = rng.uniform(0, nx, n), rng.uniform(0, ny, n)
        if dense:   # every particle in one cell in eight
            x, y = np.floor(x / 8) * 8 + x % 1, np.floor(y)  + y % 1
        P = dict(x=x * cfg.dx, y=y * cfg.dy, w=rng.uniform(0.5, 1.0, n) * 1e-2)
        for k in ("ux", "uy", "uz"):
            P[k] = 0.1 * rng.standard_normal(n)
        parts.append({k: P[k] for k in ("x", "y", "ux", "uy", "uz", "w")})
    g, o = run_pair(cfg, 1, parts=parts)
    compare_particles(g, o, cfg)
    M = g.pic_moments()
    assert normwise(M[1:10], o.M[1:10]) < 1e-9 and normwise(M[10:13], o.M[10:13]) < 1e-9
    g.close()
