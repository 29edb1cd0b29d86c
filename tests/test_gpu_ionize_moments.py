"""Moments after an ionisation pass, which adds the new particles' and takes off those of the ions they came from,
against a deposit of every particle anew (forced by setting the same fields), and the next steps against the same
run with that deposit after every pass.  FP64: the sums differ by rounding, each term off by a few 2^-53 of the
largest moment (1e-13); FP32 and exact deposits take the full deposit (equal up to the order of FP32 sums, 1e-5,
and bit for bit).  Tiles that merge a load per tile and tiles that sort it."""
import numpy as np
import pytest

from paper_1308_2590_gb300 import pic, workloads as W
from tests.parity import normwise, stream
from tests.test_gpu_ionize import FU, TU, _case

pytestmark = pytest.mark.gpu


def _run(cfg, parts, anew):
    g = pic.Pic(cfg, stream=stream(), capacity=[parts[1]["x"].size] * len(parts))
    g.load(1, parts[1])
    moments, total = [], 0
    for _ in range(cfg.steps):
        g.pic_step(1)
        total += g.pic_ionize(W.carbon_chains(2), 2024, FU, TU)
        if anew:
            g.pic_set_fields(*g.pic_fields())
        moments.append(g.pic_moments())
    state = [g.pic_get_particles(s) for s in range(4)]
    g.close()
    return moments, state, total


@pytest.mark.parametrize("tile", [8, 20])
@pytest.mark.parametrize("precision,deposit", [(W.PREC_FP64, W.DEPOSIT_ATOMIC), (W.PREC_FP64, W.DEPOSIT_DETERMINISTIC),
                                               (W.PREC_FP32, W.DEPOSIT_ATOMIC)])
def test_moments_equal_a_deposit_anew(tile, precision, deposit):
    cfg, parts = _case(precision=precision)
    cfg = cfg.scaled(tile_nx=tile, tile_ny=tile, deposit=deposit)
    Ma, Sa, na = _run(cfg, parts, False)
    Mb, Sb, nb = _run(cfg, parts, True)
    assert na == nb > 100
    exact = deposit == W.DEPOSIT_DETERMINISTIC
    tol = 1e-5 if precision == W.PREC_FP32 else 1e-13
    for a, b in zip(Ma, Mb):
        if exact:
            assert np.array_equal(a, b)
            continue
        # rho is a difference of ion and electron charge: scaled by the ions' (40 n_c)
        assert normwise(a[0], b[0], 40.0) < tol
        assert normwise(a[1:10], b[1:10]) < tol and normwise(a[10:13], b[10:13]) < tol
    for a, b in zip(Sa, Sb):
        assert np.array_equal(a["w"], b["w"])   # the order
        for k in ("x", "y", "ux", "uy", "uz"):
            assert np.array_equal(a[k], b[k]) if exact else normwise(a[k], b[k], 10.0) < (1e-4 if tol > 1e-6 else 1e-10)
