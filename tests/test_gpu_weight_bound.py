"""The exact deposit's scale comes from the sum of the loaded weights, added up on the device (device, page-locked
and prefetched arrays) or the host (pageable ones): a total that is a power of two but for rounding, one particle,
and counts around a block's share give the same moments bit for bit from every kind of memory, and the oracle's
within the FP64 parity tolerance (1e-9)."""
import numpy as np
import pytest

from paper_1308_2590_gb300 import pic, workloads as W
from tests.parity import normwise, run_pair, stream
from tests.test_gpu_parity import small_uniform

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,w", [(1, 0.7), (255, 1e-3), (257, 0.1), (3 * 2 ** 14, 1.0 / 3.0), (70001, 1e-5)])
def test_memory_kinds_agree(n, w):
    torch = pytest.importorskip("torch")
    cfg = small_uniform(ppc=1, tile=8)
    cfg.deposit = W.DEPOSIT_DETERMINISTIC
    rng = np.random.default_rng(n)
    P = dict(x=rng.uniform(0, cfg.nx * cfg.dx, n), y=rng.uniform(0, cfg.ny * cfg.dy, n), w=np.full(n, w))
    for k in ("ux", "uy", "uz"):
        P[k] = 0.2 * rng.standard_normal(n)
    P = {k: P[k] for k in ("x", "y", "ux", "uy", "uz", "w")}
    pinned = {k: torch.from_numpy(v).pin_memory().numpy() for k, v in P.items()}
    empty = {k: v[:0] for k, v in P.items()}
    M = []
    for kind in ("pageable", "pinned", "prefetched"):
        with pic.Pic(cfg, stream=stream(), capacity=[n, n]) as g:
            if kind == "prefetched":
                g.pic_prefetch_species([pinned, empty])
                g.pic_load_prefetched()
            else:
                g.load(0, P if kind == "pageable" else pinned)
            M.append(g.pic_moments())
    assert np.array_equal(M[0], M[1]) and np.array_equal(M[0], M[2])
    g, o = run_pair(cfg, 0, parts=[P, empty])
    assert normwise(M[0][0], o.M[0], np.max(np.abs(o.M[0]))) < 1e-9
    assert normwise(M[0][1:10], o.M[1:10]) < 1e-9 and normwise(M[0][10:13], o.M[10:13]) < 1e-9
    g.close()
