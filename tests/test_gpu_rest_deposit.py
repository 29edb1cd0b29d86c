"""Deposit at rest (its work items: runs of 32 segments per occupied bin) and the transposed spline deposit
at the sizes where they can go wrong: grids as narrow as the stencil and wrapping on themselves, tiles of one
segment and of several items, one particle in a large grid (nearly every bin empty), hot particles whose
segments spread over many stencils.  Moments after the load and after two steps against the oracle, with the
parity tolerances (FP64 1e-9, FP32 1e-5 normwise)."""
import numpy as np
import pytest

from paper_1308_2590_gb300 import workloads as W
from tests.parity import density_scale, normwise, run_pair
from tests.test_gpu_parity import hot, small_uniform

pytestmark = pytest.mark.gpu

CASES = [
    (4, 4, 2, 3, 1.0),      # nx, ny, tile, ppc, T (keV)
    (5, 4, 1, 2, 1.0),
    (16, 12, 8, 40, 30.0),  # 2560 particles a tile: three items
    (33, 17, 16, 3, 30.0),
]


@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32])
@pytest.mark.parametrize("order", [1, 2, 3, 4])
@pytest.mark.parametrize("nx,ny,tile,ppc,T", CASES)
def test_moments_after_load_and_steps(nx, ny, tile, ppc, T, order, precision):
    cfg = hot(small_uniform(ppc=ppc, tile=tile), T).scaled(nx=nx, ny=ny, precision=precision)
    cfg.species = [W.Species(s.q, s.m, ppc, s.density, s.temperature_kev) for s in cfg.species]
    cfg.shape = order
    tol = 1e-9 if precision == W.PREC_FP64 else 1e-5
    g, o = run_pair(cfg, 0)
    for k in range(2):
        M = g.pic_moments()
        assert normwise(M[0], o.M[0], density_scale(cfg)) < tol
        assert normwise(M[1:10], o.M[1:10]) < tol and normwise(M[10:13], o.M[10:13]) < tol
        if k == 0:
            g.pic_step(2)
            o.step(2)
            tol *= 5 if precision == W.PREC_FP32 and T > 5 else 1   # the fast plasma's FP32 positions (as elsewhere)
    g.close()


@pytest.mark.parametrize("order", [1, 3])
@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32])
def test_one_particle_in_a_large_grid(order, precision):
    cfg = small_uniform(ppc=1, tile=8).scaled(nx=300, ny=200, precision=precision)
    cfg.shape = order
    parts = [{k: np.ascontiguousarray(v[-1:]) for k, v in P.items()} for P in W.generate_particles(cfg)]
    g, o = run_pair(cfg, 0, parts=parts)
    tol = 1e-9 if precision == W.PREC_FP64 else 1e-5
    M = g.pic_moments()
    assert normwise(M[1:], o.M[1:]) < tol
    assert np.array_equal(np.any(M[1:] != 0, axis=0), np.any(o.M[1:] != 0, axis=0))
    g.close()
