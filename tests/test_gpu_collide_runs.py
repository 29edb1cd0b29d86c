"""Collision pass: the shapes of a cell's pairs where the warp's batches can go wrong -- cells with more
pairs than lanes, a species with one or a few particles per cell against many (several rounds, either
species driving), cells with 1, 2 and 3 particles, fewer occupied cells than a batch, and bins that an
ionisation pass left with partly filled segments.  Against the oracle, 1e-12 of the largest |u| (the pair
arithmetic differs from the oracle's by the rounding of a few FP64 operations per pair)."""
import numpy as np
import pytest

from oracle import collide as ocol, ionize as ion
from paper_1308_2590_gb300 import workloads as W
from tests.parity import compare_grid, density_scale, run_pair
from tests.test_gpu_collide import KAPPA, LNL, _compare_u
from tests.test_gpu_ionize import FU, TU, _case, _load
from tests.test_gpu_parity import hot, small_uniform

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ppc,keep", [(70, 0.03), (70, 1.0), (3, 0.4), (1, 0.02)])
@pytest.mark.parametrize("pairs", [[(0, 1), (1, 1)], [(1, 0), (0, 0)]])
def test_rounds_and_odd_cells(ppc, keep, pairs):
    cfg = hot(small_uniform(ppc=ppc, tile=8), 5.0)
    parts = W.generate_particles(cfg)
    sel = np.random.default_rng(5).random(parts[0]["x"].size) < keep
    parts[0] = {k: np.ascontiguousarray(v[sel]) for k, v in parts[0].items()}
    g, o = run_pair(cfg, 1, parts=parts)
    n = ocol.collide(o, pairs, 11, LNL, KAPPA)
    assert g.pic_collide(pairs, 11, LNL, KAPPA) == n > 0
    _compare_u(g, o, len(cfg.species), 1e-12)
    compare_grid(g, o, rho_scale=density_scale(cfg))
    g.close()


def test_after_an_ionisation_pass():
    cfg, parts = _case(a0=6.0)
    chains = W.carbon_chains(1)   # nothing is appended to C0: its segments stay partly filled
    g, o = _load(cfg, parts)
    g.pic_step(8)
    o.step(8)
    assert g.pic_ionize(chains, 7, FU, TU) == ion.ionize(o, chains, 7, FU, TU) > 0
    pairs = [(1, 1), (0, 1), (1, 2)]
    n = ocol.collide(o, pairs, 3, LNL, 1e3 * KAPPA)
    assert g.pic_collide(pairs, 3, LNL, 1e3 * KAPPA) == n > 0
    _compare_u(g, o, 3, 1e-12)
    g.close()
