"""FP32 literal field step: E^{n+1} is E^n plus a small change and H^{n+3/2} is H^{n+1/2} plus one, so each rounds at its own
size and not at the size of intermediate sums.  Against FP64 arithmetic on the same FP32 values, with powers of two
for dx, dy and dt, so that every factor is exact, and fields of 1.5 +- 2^-9, so that differences of neighbours are
exact.  E: one rounding in [1, 2), 2^-24, and that of the change: sums of at most 2^-6 (2^-30 each, twice two of them
times hx = 2) and of the curl, at most 2^-4 (2^-29), times dt = 2^-3: below 2^-30.  H, from the E that the step made
(1.5 +- 2^-6): sums of at most 2^-4 (2^-29) times dt/(2 dx) = 2^-2, two of them: 2^-30; one rounding in [1, 2) for x
and y, two (an FMA for each derivative) for z.  Vacuum, and tiles marked by a particle too light to change a bit,
whose nodes take the full solve and must round alike."""
import numpy as np
import pytest

from paper_1308_2590_gb300 import pic, workloads as W
from tests.parity import stream
from tests.test_gpu_parity import small_uniform

pytestmark = pytest.mark.gpu


def _diff(c, axis, h, sign):
    """Centred difference along axis of c averaged along the other; sign +1: from the lower neighbours (cells to
    nodes), -1: to the upper ones (nodes to cells)."""
    s = c + np.roll(c, sign, axis=1 - axis)
    return sign * (s - np.roll(s, sign, axis=axis)) / (2 * h)


def _curl(cfg, F, sign):
    y, x = 0, 1
    return np.stack([_diff(F[2], y, cfg.dy, sign), -_diff(F[2], x, cfg.dx, sign),
                     _diff(F[1], x, cfg.dx, sign) - _diff(F[0], y, cfg.dy, sign)])


def _step(light):
    cfg = small_uniform(n=64, ppc=1, tile=8, field_mode=W.FIELD_LITERAL, dt=0.125, precision=W.PREC_FP32)
    cfg.nx, cfg.ny, cfg.dx, cfg.dy = 64, 40, 0.25, 0.25
    rng = np.random.default_rng(12)
    E, H = ((1.5 + rng.uniform(-1.0, 1.0, (3, cfg.ny, cfg.nx)) * 2.0 ** -9).astype(np.float32).astype(np.float64)
            for _ in range(2))
    with pic.Pic(cfg, stream=stream()) as g:
        if light:
            one = np.array([1.0])
            g.load(0, dict(x=4.1 * one, y=5.1 * one, ux=0 * one, uy=0 * one, uz=0 * one, w=1e-30 * one))
        g.pic_set_fields(E, H)
        g.pic_step(1)
        return cfg, E, H, *g.pic_fields()


def _in_range(new, old):
    return np.max(np.abs(new - old)) > 2.0 ** -11 and np.max(np.abs(new - 1.5)) < 2.0 ** -6


@pytest.mark.parametrize("light", [False, True])
def test_fp32_e_rounds_once(light):
    cfg, E, H, Eg, _ = _step(light)
    want = E + cfg.dt * _curl(cfg, H, 1)
    assert _in_range(want, E)
    assert np.max(np.abs(Eg - want)) <= 2.0 ** -24 + 2.0 ** -30


@pytest.mark.parametrize("light", [False, True])
def test_fp32_h_rounds_at_its_own_size(light):
    cfg, _, H, Eg, Hg = _step(light)
    want = H - cfg.dt * _curl(cfg, Eg, -1)
    assert _in_range(want, H)
    assert np.max(np.abs(Hg[:2] - want[:2])) <= 2.0 ** -24 + 2.0 ** -30
    assert np.max(np.abs(Hg[2] - want[2])) <= 2.0 ** -23 + 2.0 ** -30
