"""Memory order between the lanes of the lane-parallel kernel: its source runs on the host, a fiber per lane, under the
thread sanitizer, with __syncwarp as the only call that orders memory.  The lanes take turns upwards and downwards, so
that a read before an unordered write in one is a read after it in the other."""
import re

import numpy as np
import pytest

from oracle import run as oracle_run
from paper_2607_11262_gb300 import workloads as W
from tests import gpu_helpers as H
from tests import tinygraphs as TG
from tests import warp_emulation as E


def races(report):
    """The reports, less those of one statement by which several lanes store the same value."""
    out = []
    for r in report.split("=================="):
        if "data race" not in r:
            continue
        a, b = (re.search(r"([Rr]ead|[Ww]rite) of size.*?#0 (\S+).*?:(\d+)", x, re.S).groups()
                for x in re.split("Previous", r)[:2])
        a, b = (a[0].lower(),) + a[1:], (b[0].lower(),) + b[1:]
        if not (a == b and a[0] == "write" and a[1].startswith("lane_launch")):
            out.append((a, b))
    return out


@pytest.mark.parametrize("backwards", [False, True])
@pytest.mark.parametrize("rows", ["lowest_id", "l2", "policies"])
def test_lanes_are_kept_apart(warp, rows, backwards):
    rng = np.random.default_rng({"lowest_id": 61, "l2": 62, "policies": 63}[rows])
    for ctas, warps, tiles in ((40, 2, 7), (24, 3, 60)):
        g = TG.random_graph(rng, 220, W_=warps, C=ctas, p_edge=0.2, intra_cta=True, kernels=warps == 3,
                            types=(W.LOAD, W.LOAD, W.STORE, W.MMA, W.EW, W.BAR))
        g.work = np.maximum(g.work, 1).astype(np.uint32)
        g.tile = rng.integers(0, tiles, g.n_nodes).astype(np.uint32)
        g.n_tiles = tiles
        prm = []
        for k in range(4):
            p = TG.small_params(rng, num_sms=int(rng.choice([2, 7, 40])), cps=int(rng.integers(1, 3)))
            p[W.P_DRAM_LAT] = p[W.P_TMA_LAT] = 2
            p[W.P_CAP_HBM] = 1 + k % 2
            if rows == "l2":
                p[W.P_L2_BYTES], p[W.P_L2_LAT], p[W.P_L2_BPC] = [1, 8, 40, 10**6][k], 3, 2
            if rows == "policies":
                p[W.P_ISSUE_POLICY], p[W.P_SUBPARTITIONS] = 1 + k % 2, 1 + k
            prm.append(p)
        prm = np.stack(prm)
        res, report = E.run(*warp, g, prm, lanes=True, pad=warps == 3, backwards=backwards)
        assert not races(report), races(report)[:5]
        for q in range(len(prm)):
            H.assert_point_equal(g, prm[q], res, q, oracle_run.simulate(g, prm[q]))
        assert not res["scratch"].any()
