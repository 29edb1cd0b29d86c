"""What a call that fails half way leaves behind, with failures that the checks build only reports (a launch check or an
allocation named by the test): the moments are those of the particles that are there, and later calls stay in bounds."""
import ctypes
import json
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from paper_1308_2590_gb300 import build as B, pic, workloads as W  # noqa: E402
from tests.parity import normwise, stream  # noqa: E402

pytestmark = pytest.mark.gpu


def _moments_of_state(g, cfg):
    """Moments of a new handle with the particles and fields of g."""
    with pic.Pic(cfg, stream=stream()) as h:
        for s in range(len(cfg.species)):
            P = g.pic_save_particles(s)
            if P["cell"].size:
                h.pic_restore_particles(s, P)
        h.pic_set_fields(*g.pic_fields())
        return h.pic_moments()


def ionisation(what, nth):
    """An ionisation pass whose nth check of this name fails, then a step."""
    from tests.test_gpu_ionize import FU, TU, _case
    cfg, parts = _case()
    with pic.Pic(cfg, stream=stream(), capacity=[parts[1]["x"].size] * len(parts)) as g:
        g.load(1, parts[1])
        for _ in range(9):   # every species holds particles by then
            g.pic_step(1)
            g.pic_ionize(W.carbon_chains(2), 2024, FU, TU)
        assert all(g.pic_particle_count(s) > 0 for s in range(4))
        g.pic_step(1)
        before = g.pic_particle_count(0)
        pic.lib().pic_checks_fail(what.encode(), nth)
        failed = False
        try:
            g.pic_ionize(W.carbon_chains(2), 2024, FU, TU)
        except pic.PicError:
            failed = True
        out = {"failed": failed, "electrons": g.pic_particle_count(0) - before}
        a, b = g.pic_moments(), _moments_of_state(g, cfg)
        # rho is a difference of ion and electron charge: scaled by the ions' (40 n_c)
        out["now"] = max(normwise(a[0], b[0], 40.0), normwise(a[1:10], b[1:10]), normwise(a[10:13], b[10:13]))
        g.pic_step(1)
        a, b = g.pic_moments(), _moments_of_state(g, cfg)
        out["step"] = max(normwise(a[0], b[0], 40.0), normwise(a[1:10], b[1:10]), normwise(a[10:13], b[10:13]))
    return out


def scratch(what, nth):
    """Particles in a species, a larger load whose sort scratch cannot be allocated, then a small load."""
    from tests.test_gpu_parity import small_uniform
    cfg = small_uniform(n=256, ppc=1, tile=2)
    rng = np.random.default_rng(9)

    def some(n):
        return dict(x=cfg.nx * cfg.dx * rng.random(n), y=cfg.ny * cfg.dy * rng.random(n),
                    **{k: 0.1 * rng.standard_normal(n) for k in ("ux", "uy", "uz")}, w=np.arange(1.0, n + 1))

    first, large, small = some(100), some(200000), some(20)
    out, states = {}, []
    for fail in (True, False):
        with pic.Pic(cfg, stream=stream()) as g:
            g.load(0, first)
            if fail:
                pic.lib().pic_checks_fail(what.encode(), nth)
                try:
                    g.load(0, large)
                except pic.PicError as e:
                    out["error"] = str(e)
            g.load(0, small)
            out["count"] = g.pic_particle_count(0)
            states.append(g.pic_save_particles(0))
    out["same"] = all(np.array_equal(states[0][k], states[1][k]) for k in states[0])
    return out


def _child(*args):
    r = subprocess.run([sys.executable, os.path.abspath(__file__), B.build(checks=True), *map(str, args)],
                       capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0, r.stdout + r.stderr
    return json.loads(r.stdout.splitlines()[-1])


# the deposits of the new target ions, electrons (two chains: C1+, C2+, electrons) and of the ions that have left
@pytest.mark.parametrize("what,nth", [("k_deposit_list", 1), ("k_deposit_list", 2), ("k_deposit_list", 4),
                                      ("k_cell_moments", 1), ("ionisation staging copies", 1)])
def test_moments_after_a_failed_ionisation_pass(what, nth):
    """FP64 sums of the same particles in another order: a few 2^-53 of the largest moment a term (1e-13)."""
    out = _child("ionisation", what, nth)
    assert out["failed"], out
    assert out["now"] < 1e-13 and out["step"] < 1e-13, out



def test_small_load_after_a_failed_allocation_of_the_sort_scratch():
    """More tiles (128 x 126) than the scratch of a sort of 20 particles has entries."""
    out = _child("scratch", "sort scratch", 1)
    assert "sort scratch" in out["error"] and out["count"] == 120 and out["same"], out


if __name__ == "__main__":
    pic.lib(sys.argv[1]).pic_checks_fail.argtypes = [ctypes.c_char_p, ctypes.c_int]
    print(json.dumps({"ionisation": ionisation, "scratch": scratch}[sys.argv[2]](sys.argv[3], int(sys.argv[4]))))
