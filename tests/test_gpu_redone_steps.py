"""Steps whose regroup fails every time, in the form whose moments are deposited after the regroup (FP32, linear shape,
time-centred solve, plain deposit): a step redone after the full sort leaves its own moments to the next one, which
must find them whether the steps were queued by pic_step, by pic_batch_step or by either in turn.

A thermal plasma with five particles that cross at least two tiles of four cells in every step (c dt / dx = 9).  The
fields start at zero and are made by the particles' currents, so a field solve without moments loses them whole
(errors of order one).  Tolerances against the FP64 oracle, normwise: moments 5e-5, the FP32 form's for particles
that move several cells a step (tests/test_gpu_fp32.py); fields 2e-4, four steps of such moments.  Two schedules of
one run differ by the order of FP32 sums only: the same bounds."""
import numpy as np
import pytest

from paper_1308_2590_gb300 import pic, workloads as W
from tests.parity import normwise, run_pair, stream
from tests.test_gpu_parity import small_uniform

pytestmark = pytest.mark.gpu

STEPS = 4
MOM_RTOL, FIELD_RTOL = 5e-5, 2e-4


def _case(far=5):
    cfg = small_uniform(n=32, ppc=1, tile=4, field_mode=W.FIELD_CN, dt=0.18, precision=W.PREC_FP32)
    cfg.cn_tol = 1e-10
    assert abs(cfg.dt / cfg.dx - 9.0) < 1e-12
    n = 400
    rng = np.random.default_rng(21)
    P = dict(x=32 * cfg.dx * rng.random(n), y=cfg.ny * cfg.dy * rng.random(n), ux=0.1 * rng.standard_normal(n),
             uy=0.1 * rng.standard_normal(n), uz=0.1 * rng.standard_normal(n), w=np.full(n, 1e-4))
    P["ux"][:far] = 40.0
    P["uy"][:far] = 0.0
    return cfg, [P, {k: v[:0] for k, v in P.items()}]


def _oracle_errors(g, o):
    M, (E, H) = g.pic_moments(), g.pic_fields()
    e = {"rho": normwise(M[0], o.M[0]), "S": normwise(M[1:10], o.M[1:10]), "dj": normwise(M[10:13], o.M[10:13])}
    scale = max(np.max(np.abs(o.E)), np.max(np.abs(o.H)))
    e["E"], e["H"] = normwise(E, o.E, scale), normwise(H, o.H, scale)
    return e


def _check(g, o):
    e = _oracle_errors(g, o)
    assert all(v < (FIELD_RTOL if k in "EH" else MOM_RTOL) for k, v in e.items()), e


# calls: (batched, steps)
@pytest.mark.parametrize("calls", [[(False, 4)], [(True, 4)], [(True, 1)] * 4, [(False, 1), (True, 3)], [(True, 2), (False, 2)],
                                   [(True, 3), (False, 1)], [(False, 2), (True, 1), (False, 1)]])
def test_moments_of_a_redone_step_reach_the_next(calls):
    cfg, parts = _case()
    quiet_cfg, quiet_parts = _case(far=0)
    g, o = run_pair(cfg, 0, parts=parts)
    q, oq = run_pair(quiet_cfg, 0, parts=quiet_parts)   # a run of the same batch without a failed regroup of its own
    o.step(STEPS)
    oq.step(STEPS)
    b = pic.Batch(2, stream=stream())
    for batched, n in calls:
        if batched:
            b.step([g, q], n)
        else:
            g.pic_step(n)
            q.pic_step(n)
    assert g.pic_diagnostics()["full_regroups"] == STEPS
    assert q.pic_diagnostics()["full_regroups"] == 0
    _check(g, o)
    _check(q, oq)
    b.close()
    g.close()
    q.close()
