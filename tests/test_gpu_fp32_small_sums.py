"""FP32 push: the particles that it adds to the node moments one by one (those few of a warp's that end in a cell of
their own) are summed apart from the bulk, so that they round at the size of their own sum.  Ions of weight 2, 32 at
rest in every cell centre, make 64 at every node, exactly; light electrons of weight 2^-10 run through them (576
tiles: more work items than blocks, so that most electrons meet the ions' sums).  Against the exact deposit of the
same step, whose sums are integers: an electron sum of size L over n electrons is off by at most n additions of
2^-24 L and, for sums made in registers or shared memory first, as many again.  (Added to the ions' 64, each would be
off by up to 2^-24 64.)"""
import numpy as np
import pytest

from paper_1308_2590_gb300 import pic, workloads as W
from tests.parity import stream
from tests.test_gpu_parity import small_uniform

pytestmark = pytest.mark.gpu


def test_few_particles_on_a_large_sum():
    n, heavy, light = 192, 32, 4
    cfg = small_uniform(n=n, ppc=1, tile=8, field_mode=W.FIELD_LITERAL, dt=0.125, precision=W.PREC_FP32)
    cfg.nx, cfg.ny, cfg.dx, cfg.dy = n, n, 0.25, 0.25
    cfg.species = [W.Species(1.0, 1e30, heavy, 1.0, 0.0), W.Species(-1.0, 1.0, light, 1.0, 0.0)]
    cell = np.repeat(np.arange(n * n), heavy)
    z = np.zeros(cell.size)
    ions = dict(x=(cell % n + 0.5) * cfg.dx, y=(cell // n + 0.5) * cfg.dy, ux=z, uy=z, uz=z, w=z + 2.0)
    rng = np.random.default_rng(4)
    m = n * n * light
    el = dict(x=n * cfg.dx * rng.random(m), y=n * cfg.dy * rng.random(m), ux=rng.standard_normal(m),
              uy=rng.standard_normal(m), uz=rng.standard_normal(m), w=np.full(m, 2.0 ** -10))
    rho = {}
    for deposit in (W.DEPOSIT_ATOMIC, W.DEPOSIT_DETERMINISTIC):
        with pic.Pic(cfg.scaled(deposit=deposit), stream=stream()) as g:
            g.load(0, ions)
            g.load(1, el)
            g.pic_step(1)
            rho[deposit] = g.pic_moments()[0] * cfg.dx * cfg.dy
            c = g.pic_get_particles(1)["cell"]
    exact = rho[W.DEPOSIT_DETERMINISTIC]
    L = 64.0 - exact
    assert 0.0 <= L.min() and 2.0 ** -10 < L.max() < 1.0
    near = np.bincount(c, minlength=n * n).reshape(n, n)
    near = near + np.roll(near, 1, 0)
    near = near + np.roll(near, 1, 1)   # electrons in the four cells of a node
    err = np.abs(rho[W.DEPOSIT_ATOMIC] - exact)
    assert err.max() <= near.max() * 2.0 ** -23 * L.max(), (err.max(), near.max(), L.max())
