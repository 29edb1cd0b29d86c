"""CN solve at the sizes and plasmas where its paths change: sides that are powers of two, products of small
primes, odd, prime, at and above the largest prime of the spectral preconditioner; one cluster of blocks and a
grid; a uniform plasma (corrections by the preconditioner alone) and a dense slab in vacuum (BiCGSTAB around
it); a walled box (block-Jacobi).  Fields, moments and particles against the oracle's sparse LU solve with the
parity tolerances (1e-10, 1e-9), the solver's own residual below 1e-12."""
import pytest

from paper_1308_2590_gb300 import workloads as W
from tests.parity import compare_grid, compare_particles, density_scale, run_pair
from tests.test_gpu_parity import hot, small_uniform

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(16, 16), (2, 3), (3, 2), (24, 19), (30, 21), (61, 4), (6, 61), (67, 5), (48, 40),
                                   (96, 90), (128, 64)])
@pytest.mark.parametrize("slab", [False, True])
def test_sizes(nx, ny, slab):
    cfg = hot(small_uniform(ppc=3, tile=8), 5.0).scaled(nx=nx, ny=ny)
    if slab:
        if nx < 6:
            pytest.skip("no room for a slab")
        cfg.slab = (nx // 3, nx // 3 + max(1, nx // 4))
        cfg.species = [W.Species(s.q, s.m, s.ppc, 40.0, s.temperature_kev) for s in cfg.species]
    g, o = run_pair(cfg, 3)
    compare_particles(g, o, cfg)
    compare_grid(g, o, rho_scale=density_scale(cfg))
    assert g.pic_diagnostics()["cn_residual"] < 1e-12
    g.close()
