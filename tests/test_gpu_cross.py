"""Releases into heads of other CTAs, and NoC servers, against the oracle: CTAs
that sit in the slot of their rank, CTAs that do not (empty CTAs before them,
more CTAs than slots), heads that other CTAs release several times, and SM
groups whose NoC servers are all taken, or not."""
import numpy as np
import pytest

from oracle import run as oracle_run
from paper_2607_11262_gb300 import workloads as W
from tests import gpu_helpers as H
from tests import tinygraphs as TG

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2607_11262_gb300 import gts
    gts.load()


def _check(g, rows, res):
    for q in range(rows.shape[0]):
        H.assert_point_equal(g, rows[q], res, q, oracle_run.simulate(g, rows[q]))


@pytest.mark.parametrize("ctas,empty,slots", [(6, 0, 6), (6, 2, 8), (40, 0, 40), (40, 3, 43), (9, 0, 4), (9, 2, 5)])
def test_edges_between_ctas(ctas, empty, slots):
    rng = np.random.default_rng(8000 + 10 * ctas + empty)
    for k in range(4):
        g = TG.random_graph(rng, 160, W_=3, C=ctas, p_edge=0.05, cta_major=True,
                            types=(W.LOAD, W.STORE, W.MMA, W.EW, W.BAR))
        if empty:
            g.cta = np.where(g.cta >= ctas // 2, g.cta + empty, g.cta).astype(np.uint32)
            g.cta_kernel = np.zeros(ctas + empty, np.uint32)
            g.cta_off = np.array([0, ctas + empty], np.uint32)
        rows = np.stack([TG.small_params(rng, num_sms=-(-slots // c), cps=c) for c in (1, 2, 3)])
        _check(g, rows, H.run_gpu(g, rows))


@pytest.mark.parametrize("cap,group", [(1, 1), (1, 4), (2, 4), (16, 16), (32, 32)])
def test_noc_servers(cap, group):
    rng = np.random.default_rng(8100 + 40 * cap + group)
    for k in range(4):
        g = TG.random_graph(rng, 200, W_=4, C=20, p_edge=0.04, cta_major=bool(k % 2),
                            types=(W.DSMEM, W.DSMEM, W.DSMEM, W.EW, W.STORE, W.BAR))
        rows = []
        for cps in (1, 2):
            p = TG.small_params(rng, num_sms=20, cps=cps)
            p[W.P_NOC_BPC], p[W.P_NOC_LAT], p[W.P_CAP_NOC], p[W.P_CLUSTER_SMS] = 1, int(rng.integers(0, 4)), cap, group
            p[W.P_CAP_LSU] = 4
            rows.append(p)
        rows = np.stack(rows)
        _check(g, rows, H.run_gpu(g, rows))
