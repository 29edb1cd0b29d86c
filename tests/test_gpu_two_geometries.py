"""Runs of different tile sizes alive at the same time: the kernels' limit of dynamic shared memory belongs to the kernel,
not to the run, so a run set up later with smaller tiles must not take it below what an earlier one needs.  Each form
of the push, the regroup and the batched launches; with the exact deposit the bits of a run alone."""
import numpy as np
import pytest

from paper_1308_2590_gb300 import pic, workloads as W
from tests.parity import stream
from tests.test_gpu_parity import small_foil, small_uniform

pytestmark = pytest.mark.gpu


def _state(g, nsp):
    out = [g.pic_moments(), *g.pic_fields()]
    for s in range(nsp):
        P = g.pic_get_particles(s)
        out += [P[k] for k in ("x", "y", "ux", "uy", "uz", "w", "cell")]
    return out


def _make(kind, precision, deposit, shape, tile):
    cfg = small_foil(nx=48, ny=40, tile=tile, precision=precision) if kind == "foil" else \
        small_uniform(n=40, tile=tile, precision=precision)
    if precision == W.PREC_FP32:
        cfg.cn_tol = 1e-10
    cfg.deposit, cfg.shape = deposit, shape
    return cfg


def _loaded(cfg, parts):
    g = pic.Pic(cfg, stream=stream())
    for s, P in enumerate(parts):
        g.load(s, P)
    return g


@pytest.mark.parametrize("kind", ["foil", "uniform"])
@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32])
@pytest.mark.parametrize("deposit,shape", [(W.DEPOSIT_ATOMIC, 1), (W.DEPOSIT_DETERMINISTIC, 1), (W.DEPOSIT_ATOMIC, 3)])
def test_small_tiles_after_large_ones(kind, precision, deposit, shape):
    big, small = (_make(kind, precision, deposit, shape, t) for t in (16, 4))
    parts = W.generate_particles(big)
    with _loaded(big, parts) as alone:
        alone.pic_step(3)
        ref = _state(alone, len(big.species))
    a = _loaded(big, parts)
    b = _loaded(small, W.generate_particles(small))
    for g in (b, a):
        g.pic_step(2)
    if shape == 1:
        batch = pic.Batch(2, stream=stream())
        batch.step([a, b], 1)
        batch.step([b], 1)
        batch.close()
    else:
        a.pic_step(1)
    got = _state(a, len(big.species))
    if deposit == W.DEPOSIT_DETERMINISTIC:
        for x, y in zip(ref, got):
            assert np.array_equal(x.view(np.uint8), y.view(np.uint8))
    else:
        assert all(np.all(np.isfinite(x)) for x in got)
    a.close()
    b.close()
