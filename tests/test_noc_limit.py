"""The widest rows with NoC servers that the shared memory of a point holds: on the host (the kernel's source, a fiber
per lane) and on the GPU, against the oracle.  A point of NS one-CTA SMs with W warp slots, c LSU servers and k NoC
servers per SM takes 57 + NS (4 W + 7 + c + k) words (one HBM server), rounded up to four, of the 58,112 of 227 KB."""
import numpy as np
import pytest

from oracle import run as oracle_run
from paper_2607_11262_gb300 import workloads as W
from tests import gpu_helpers as H
from tests import tinygraphs as TG
from tests import warp_emulation as E

SMS, WARPS = 110, 128


def _batch():
    rng = np.random.default_rng(88)
    n = 330
    cta = np.sort(np.concatenate([np.arange(SMS), rng.integers(0, SMS, n - SMS)]))
    edges = sorted({(int(u), int(u + d), int(rng.integers(0, 2))) for u in range(n) for d in rng.integers(1, 9, 2) if u + d < n})
    edges = list({(u, v): (u, v, k) for u, v, k in edges}.values())
    g = TG.make(n, edges, [int(x) for x in rng.choice([W.DSMEM, W.DSMEM, W.SMEM], n)],
                [int(x) for x in rng.integers(0, WARPS, n)], [int(x) for x in cta], WARPS,
                work=[int(x) for x in rng.integers(1, 9, n)])
    rows = []
    for lsu, noc, group in ((6, 2, 1), (7, 1, 1), (6, 3, 2), (5, 3, 1), (6, 3, 1)):
        p = TG.unit_params(SMS, 1)
        p[W.P_CAP_LSU] = lsu
        p[W.P_NOC_BPC], p[W.P_NOC_LAT], p[W.P_CAP_NOC], p[W.P_CLUSTER_SMS] = 1, 2, noc, group
        rows.append(p)
    words = [57 + SMS * (4 * WARPS + 7 + p[W.P_CAP_LSU]) + -(-SMS // p[W.P_CLUSTER_SMS]) * p[W.P_CAP_NOC] for p in rows]
    assert [-(-w // 4) * 4 <= 58112 for w in words] == [True, True, True, True, False]
    return g, np.stack(rows)


def _check(g, rows, res):
    for q in range(len(rows) - 1):
        H.assert_point_equal(g, rows[q], res, q, oracle_run.simulate(g, rows[q]))
    assert res["status"][-1] == -9  # one word per SM too many


def test_on_the_host(warp):
    g, rows = _batch()
    rows = rows[[0, -1]]
    _check(g, rows, E.run(*warp, g, rows, lanes=False)[0])


@pytest.mark.gpu
def test_on_the_gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g, rows = _batch()
    _check(g, rows, H.run_gpu(g, rows))
