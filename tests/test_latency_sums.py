"""Base latencies that are sums of several parameters, each up to 2^31-1: a LOAD that misses in L2 has three, which
pass 2^32.  In both kernels, on the host (the kernels' source, a fiber per lane) and on the GPU, against the oracle."""
import numpy as np
import pytest

from oracle import run as oracle_run
from paper_2607_11262_gb300 import workloads as W
from tests import gpu_helpers as H
from tests import tinygraphs as TG
from tests import warp_emulation as E

BIG = 2**31 - 1


def _batch():
    g = TG.make(4, [(0, 1, W.DATA), (2, 3, W.DATA)], [W.LOAD, W.MMA] * 2, [0] * 4, [0, 0, 1, 1], 1, work=[2, 1, 2, 1])
    g.tile, g.n_tiles = np.array([0, W.NO_TILE, 1, W.NO_TILE], np.uint32), 2
    rows = []
    for tma, l2, dram in ((BIG, BIG, BIG), (BIG, BIG, 2), (BIG, BIG, 12), (BIG, 0, 1), (2**30, 2**30, 2**31 - 9),
                          (2**30, 2**30 - 20, 4), (3, 4, 5)):
        p = TG.unit_params(2, 1)
        p[W.P_TMA_LAT], p[W.P_L2_LAT], p[W.P_DRAM_LAT], p[W.P_MMA_LAT] = tma, l2, dram, 1
        p[W.P_L2_BYTES], p[W.P_L2_BPC] = 64, 1
        rows.append(p)
    rows = np.stack(rows)
    refs = [oracle_run.simulate(g, p) for p in rows]
    assert [r.status for r in refs] == [-6] * 5 + [0, 0]
    return g, rows, refs


@pytest.mark.parametrize("lanes", [False, True])
def test_on_the_host(warp, lanes):
    g, rows, refs = _batch()
    res, _ = E.run(*warp, g, rows, lanes=lanes)
    for q, ref in enumerate(refs):
        H.assert_point_equal(g, rows[q], res, q, ref)


@pytest.mark.gpu
@pytest.mark.parametrize("kernel", [1, 2])   # GTS_KERNEL_LANES, GTS_KERNEL_GENERAL
def test_on_the_gpu(kernel):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g, rows, refs = _batch()
    res = H.run_gpu(g, rows, kernel=kernel)
    assert res["plan"] & 1 == (kernel == 1)   # GTS_PLAN_LANES
    for q, ref in enumerate(refs):
        H.assert_point_equal(g, rows[q], res, q, ref)
