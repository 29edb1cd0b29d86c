"""The per-tile regroup's order (tile, cell, stayers before arrivals, previous order kept) and nothing lost,
exactly, in both forms, where its paths change: segments scattered over many cells (the staged FP32 copy),
more and fewer than 128 arrivals a tile, ragged tiles, tiles at and above the staging limit of cells, tiles of
several thousand particles, moves across several tiles (the full regroup).  Distinct weights tag the particles:
the order after a step must be the stable sort of the order before it by (tile, cell, came from another tile)
of the cells the particles are in now."""
import numpy as np
import pytest

from paper_1308_2590_gb300 import pic, workloads as W
from tests.parity import stream
from tests.test_gpu_parity import hot, small_uniform

pytestmark = pytest.mark.gpu

CASES = [
    (48, 40, 16, 40, 1.0),     # nx, ny, tile, ppc, T (keV); 10240 particles a tile: too many to stage in FP32
    (48, 40, 16, 12, 1.0),
    (33, 17, 16, 5, 1.0),
    (48, 48, 24, 6, 1.0),      # 576 cells: the largest staged tile
    (50, 50, 25, 6, 1.0),
    (40, 40, 8, 30, 50.0),
    (32, 32, 8, 3, 0.01),
]


@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32])
@pytest.mark.parametrize("nx,ny,tile,ppc,T", CASES)
def test_order_after_steps(nx, ny, tile, ppc, T, precision):
    cfg = hot(small_uniform(ppc=ppc, tile=tile), T).scaled(nx=nx, ny=ny, precision=precision)
    cfg.cn_tol = 1e-8
    cfg.species = [W.Species(s.q, s.m if k == 0 else 1.0, ppc, s.density, T) for k, s in enumerate(cfg.species)]
    parts = W.generate_particles(cfg)
    for P in parts:
        P["w"] = P["w"][0] * (1.0 + np.arange(P["w"].size) * 2.0 ** -22)
        assert np.unique(P["w"].astype(np.float32)).size == P["w"].size
    g = pic.Pic(cfg, stream=stream())
    g.pic_load_species(parts)
    tx, ty = min(tile, nx), min(tile, ny)
    ntx = -(-nx // tx)

    def keys(cell):
        cx, cy = cell % nx, cell // nx
        t = (cy // ty) * ntx + cx // tx
        return t, t * (tx * ty) + (cy % ty) * tx + cx % tx

    before = [g.pic_save_particles(s) for s in range(2)]
    for _ in range(3):
        g.pic_step(1)
        after = [g.pic_save_particles(s) for s in range(2)]
        for a, b in zip(after, before):
            assert a["w"].size == b["w"].size
            ia = np.argsort(a["w"], kind="stable")
            ib = np.argsort(b["w"], kind="stable")
            assert np.array_equal(a["w"][ia], b["w"][ib])
            new_cell = np.empty(ib.size, np.int64)
            new_cell[ib] = a["cell"][ia]                       # in the order before the step
            t_new, k_new = keys(new_cell)
            t_old, _ = keys(b["cell"].astype(np.int64))
            order = np.argsort(2 * k_new + (t_new != t_old), kind="stable")
            assert np.array_equal(a["w"], b["w"][order])
        before = after
    g.close()
