"""Loads into species that already hold particles: tiles that order their bin and the new particles in one block
(up to 256 cells) and larger ones that take the sort; one new particle, counts around a segment of 32, many, all in
one cell.  Without a step between them two loads equal one load of both lists, bit for bit (the order is stable);
after steps the order is the oracle's and the state within the parity tolerances (1e-10, 1e-9)."""
import numpy as np
import pytest

from paper_1308_2590_gb300 import pic, workloads as W
from tests.parity import compare_grid, compare_particles, density_scale, run_pair, stream
from tests.test_gpu_parity import hot, small_foil

pytestmark = pytest.mark.gpu


def _new(cfg, n, one_cell, seed):
    rng = np.random.default_rng(seed)
    lo, hi = ((5 * cfg.dx, 6 * cfg.dx), (7 * cfg.dy, 8 * cfg.dy)) if one_cell else ((0, cfg.nx * cfg.dx),
                                                                                  (0, cfg.ny * cfg.dy))
    P = {"x": rng.uniform(lo[0], lo[1] if one_cell else hi[0], n),
         "y": rng.uniform(hi[0] if one_cell else 0.0, hi[1], n)}
    for k in ("ux", "uy", "uz"):
        P[k] = 0.1 * rng.standard_normal(n)
    P["w"] = rng.uniform(0.5, 1.0, n) * 1e-3
    return P


@pytest.mark.parametrize("tile", [1, 5, 16, 17])
@pytest.mark.parametrize("n,one_cell", [(1, False), (32, False), (33, True), (3000, False), (700, True)])
@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32])
def test_second_load(tile, n, one_cell, precision):
    cfg = hot(small_foil(tile=tile, precision=precision), 5.0)
    parts = W.generate_particles(cfg)
    new = _new(cfg, n, one_cell, n + tile)
    two, one = pic.Pic(cfg, stream=stream()), pic.Pic(cfg, stream=stream())
    two.load(0, parts[0])
    two.load(0, new)
    one.load(0, {k: np.concatenate([parts[0][k], new[k]]) for k in new})
    a, b = two.pic_get_particles(0), one.pic_get_particles(0)
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    two.close()
    one.close()
    if precision == W.PREC_FP32:
        return
    g, o = run_pair(cfg, 3, parts=parts)
    g.load(0, new)
    o.load_particles(0, **new)
    compare_particles(g, o, cfg)
    g.pic_step(2)
    o.step(2)
    compare_particles(g, o, cfg)
    compare_grid(g, o, rho_scale=density_scale(cfg))
    g.close()
