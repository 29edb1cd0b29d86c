"""FP32 loads and the cell deposit at their edges: values whose rounding to FP32 takes each branch (ties, carries
into the exponent, denormals, underflow, the largest finite value), bit for bit; cells of 0 .. 70 particles, so that
runs of every length modulo the deposit's groups start at every lane, with ragged tiles and items of several
segments, moments against the oracle (1e-5 normwise, the FP32 parity tolerance)."""
import numpy as np
import pytest

from paper_1308_2590_gb300 import pic, workloads as W
from tests.parity import normwise, run_pair, stream
from tests.test_gpu_parity import small_uniform

pytestmark = pytest.mark.gpu


def test_values_round_to_nearest_even():
    rng = np.random.default_rng(8)
    tiny = 2.0 ** -149
    v = [0.0, -0.0, tiny, tiny / 2, np.nextafter(tiny / 2, 1), tiny * 1.5, tiny * 2.5, 5e-324, -2.0 ** -126,
         np.nextafter(2.0 ** -126, 0), 2.0 ** -126 - tiny / 2, 1 + 2.0 ** -24, 1 + 3 * 2.0 ** -24, 2 - 2.0 ** -25,
         -(1 + 2.0 ** -24 + 2.0 ** -52), 3.4028234663852886e38, -1.0000000596046448e38]
    v = np.array(v + list(rng.standard_normal(500) * 10.0 ** rng.uniform(-46, 30, 500)))
    n = v.size
    cfg = small_uniform(n=16, ppc=1, tile=4, precision=W.PREC_FP32)
    P = dict(x=np.full(n, 0.5 * cfg.dx), y=np.full(n, 0.5 * cfg.dy), ux=v, uy=v[::-1].copy(), uz=np.roll(v, 7),
             w=np.full(n, 1e-3))
    with pic.Pic(cfg, stream=stream(), capacity=[n, n]) as g:
        g.load(0, P)
        a = g.pic_get_particles(0)
        for k in ("ux", "uy", "uz"):
            assert np.array_equal(a[k], P[k].astype(np.float32).astype(np.float64)), k
            assert np.array_equal(np.signbit(a[k]), np.signbit(P[k])), k


@pytest.mark.parametrize("tile", [3, 8, 16])
@pytest.mark.parametrize("most", [5, 70])
def test_runs_of_every_length(tile, most):
    cfg = small_uniform(n=23, ppc=1, tile=tile, precision=W.PREC_FP32)
    rng = np.random.default_rng(most)
    count = np.arange(cfg.nx * cfg.ny) % (most + 1)
    rng.shuffle(count)
    cell = np.repeat(np.arange(cfg.nx * cfg.ny), count)
    parts = []
    for _ in cfg.species:
        n = cell.size
        P = dict(x=(cell % cfg.nx + rng.random(n)) * cfg.dx, y=(cell // cfg.nx + rng.random(n)) * cfg.dy,
                 w=rng.uniform(0.5, 1.0, n) * 1e-2)
        for k in ("ux", "uy", "uz"):
            P[k] = 0.3 * rng.standard_normal(n)
        parts.append({k: P[k] for k in ("x", "y", "ux", "uy", "uz", "w")})
    rngf = np.random.default_rng(2)
    fields = 0.1 * rngf.standard_normal((3, cfg.ny, cfg.nx)), 0.3 * rngf.standard_normal((3, cfg.ny, cfg.nx))
    g, o = run_pair(cfg, 0, parts=parts, fields=fields)
    M = g.pic_moments()
    assert normwise(M[0], o.M[0], np.max(np.abs(o.M[0]))) < 1e-5
    assert normwise(M[1:10], o.M[1:10]) < 1e-5 and normwise(M[10:13], o.M[10:13]) < 1e-5
    g.close()
