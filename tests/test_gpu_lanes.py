"""The lane-parallel kernel instance (one simulated SM per lane), which the
library can launch when the graph's ids are in CTA order with no edge between
CTAs and every valid row has up to 160 SMs of up to 32 warp slots: against the oracle where its tiles
end (SMs per lane round, slots read four at a time, the inline successors,
servers kept in registers up to four, L2 lists in shared memory), and against
the general instance on the same rows.  The tests hold their batches to the kernel
they mean and assert that it ran (H.run_gpu gives the plan); which one a batch gets
by itself has tests of its own.  Integer results, compared bit for bit."""
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


MIXES = ((W.LOAD, W.LOAD, W.STORE, W.MMA, W.EW, W.BAR), (W.LOAD, W.BAR, W.MMA), (W.LOAD, W.STORE),
         (W.LOAD, W.SMEM, W.MMA, W.EW, W.STORE, W.BAR, W.NOP))


def _graph(rng, n, ctas, warps, mix, kernels=False, max_work=9, p_edge=0.2, p_issue=0.3):
    g = TG.random_graph(rng, n, W_=warps, C=ctas, p_edge=p_edge, p_issue=p_issue, intra_cta=True, kernels=kernels,
                        types=MIXES[mix], max_work=max_work)
    g.work = np.maximum(g.work, 1).astype(np.uint32)
    g.lat_extra = np.where(g.type == W.NOP, 1, g.lat_extra).astype(np.uint32)  # no zero-latency node
    return g


def _row(rng, sms, cps, cap_hbm=1, cap_tma=1, cap_lsu=4):
    p = TG.small_params(rng, num_sms=sms, cps=cps)
    for k in (W.P_DRAM_LAT, W.P_TMA_LAT, W.P_SMEM_LAT, W.P_MMA_LAT, W.P_ALU_LAT):
        p[k] = max(1, int(p[k]))
    p[W.P_HBM_BPC] = int(rng.choice([1, 1, 2, 8]))
    p[W.P_TMA_BPC] = int(rng.choice([1, 3, 50]))
    p[W.P_CAP_HBM], p[W.P_CAP_TMA], p[W.P_CAP_LSU] = cap_hbm, cap_tma, cap_lsu
    return p


LANES = 1             # GTS_PLAN_LANES
IN_LANES, IN_GENERAL = 1, 2   # GTS_KERNEL_*


def _check(g, rows, res, lanes=True):
    assert bool(res["plan"] & LANES) == lanes, res["plan"]
    for q in range(rows.shape[0]):
        H.assert_point_equal(g, rows[q], res, q, oracle_run.simulate(g, rows[q]))


@pytest.mark.parametrize("sms", [2, 31, 32, 33, 64, 65, 160, 161])
def test_sm_counts(sms):
    """Around one to five SMs per lane, and one more than a lane looks after."""
    rng = np.random.default_rng(7000 + sms)
    for mix in range(4):
        g = _graph(rng, 700, 170, 2, mix, kernels=mix == 3)
        rows = np.stack([_row(rng, sms, 1, cap_hbm=c) for c in (1, 1, 3)])
        _check(g, rows, H.run_gpu(g, rows, kernel=IN_LANES), lanes=sms <= 160)


@pytest.mark.parametrize("sms", [1, 2, 40])
def test_rows_of_one_sm(sms):
    """A row of one SM, alone and beside another."""
    rng = np.random.default_rng(7050 + sms)
    g = _graph(rng, 300, 40, 3, 0)
    rows = np.stack([_row(rng, 1, 2, cap_hbm=2), _row(rng, sms, 1)])
    _check(g, rows, H.run_gpu(g, rows, kernel=IN_LANES))


@pytest.mark.parametrize("warps,cps", [(1, 1), (3, 1), (4, 1), (5, 1), (3, 3), (8, 4), (11, 3)])
def test_slots_per_sm(warps, cps):
    """1 to 33 slots per SM (a lane scans up to 32)."""
    rng = np.random.default_rng(7100 + warps * cps)
    g = _graph(rng, 300, 20, warps, 0, kernels=True)
    rows = np.stack([_row(rng, s, cps) for s in (2, 3, 5)])
    _check(g, rows, H.run_gpu(g, rows, kernel=IN_LANES), lanes=warps * cps <= 32)


@pytest.mark.parametrize("caps", [(1, 1, 1), (2, 2, 2), (4, 4, 4), (1, 5, 5), (32, 32, 32)])
def test_server_counts(caps):
    rng = np.random.default_rng(7200 + caps[0] * 40 + caps[1])
    for mix in (0, 3):
        g = _graph(rng, 260, 30, 4, mix)
        rows = np.stack([_row(rng, int(rng.choice([2, 7, 33])), int(rng.integers(1, 3)), *caps) for _ in range(6)])
        _check(g, rows, H.run_gpu(g, rows, kernel=IN_LANES))


@pytest.mark.parametrize("fan", [1, 2, 3, 6, 7, 8, 40])
def test_successor_counts(fan):
    """Successors kept beside the head (up to 6) and looked up (7 and more)."""
    rng = np.random.default_rng(7300 + fan)
    n, ctas = fan + 2, 5
    types = [W.LOAD] + [int(x) for x in rng.choice([W.MMA, W.EW, W.SMEM, W.BAR], fan)] + [W.STORE]
    warps = [0] + [int(x) for x in rng.integers(0, 3, fan)] + [1]
    edges = [(0, v, int(rng.integers(0, 2))) for v in range(1, fan + 1)] + [(v, n - 1, W.DATA) for v in range(1, fan + 1)]
    g = TG.make(n * ctas, [(c * n + u, c * n + v, k) for c in range(ctas) for u, v, k in edges], types * ctas,
                warps * ctas, [c for c in range(ctas) for _ in range(n)], 3,
                work=[int(x) for x in rng.integers(1, 9, n * ctas)])
    rows = np.stack([_row(rng, s, c) for s, c in ((2, 1), (3, 2), (8, 1))])
    _check(g, rows, H.run_gpu(g, rows, kernel=IN_LANES))


@pytest.mark.parametrize("mix", range(4))
def test_nodes_without_work(mix):
    """Nodes that hold their unit for no cycle; their latency is positive."""
    rng = np.random.default_rng(7350 + mix)
    g = _graph(rng, 300, 40, 3, mix, kernels=mix == 1)
    g.work[rng.random(g.n_nodes) < 0.4] = 0
    rows = np.stack([_row(rng, s, c, h) for s, c, h in ((2, 1, 1), (5, 2, 2), (33, 1, 1), (40, 1, 3))])
    _check(g, rows, H.run_gpu(g, rows, kernel=IN_LANES))


@pytest.mark.parametrize("seed", range(6))
def test_agrees_with_the_general_instance(seed):
    """Rows over all forms the rule takes, in either kernel."""
    rng = np.random.default_rng(7400 + seed)
    g = _graph(rng, 400, int(rng.integers(20, 60)), int(rng.integers(1, 7)), seed % 4, kernels=seed % 2 == 1,
               max_work=[2, 6, 60][seed % 3], p_issue=[0.0, 0.3, 0.9][seed % 3])
    g.lat_extra[::5] += 1
    rows = np.stack([_row(rng, int(rng.choice([2, 5, 31, 40, 130])), int(rng.choice([1, 2, 4])),
                          int(rng.choice([1, 1, 2, 4])), int(rng.choice([1, 1, 2, 5])), int(rng.integers(1, 9)))
                     for _ in range(24)])
    rows[7, W.P_TMA_BPC] = 0                    # refused
    rows[11, W.P_DRAM_LAT] = 2**31 - 40         # overflows
    lanes = H.run_gpu(g, rows, kernel=IN_LANES)
    assert lanes["plan"] & LANES
    both = H.run_gpu(g, rows, kernel=IN_GENERAL)
    assert not both["plan"] & LANES
    n = rows.shape[0]
    for k in ("status", "makespan"):
        assert np.array_equal(lanes[k], both[k][:n]), k
    ok = lanes["status"] == 0
    assert ok.sum() >= n - 2
    for k in ("start", "finish", "digest", "cta_sm", "busy"):
        assert np.array_equal(lanes[k][ok], both[k][:n][ok]), k


def test_empty_ctas_and_gates():
    """Empty CTAs before, between and after the others, over three kernels."""
    rng = np.random.default_rng(7500)
    g = _graph(rng, 120, 12, 2, 0)
    remap = np.array([1, 2, 4, 5, 6, 9, 10, 11, 13, 15, 16, 18], np.uint32)
    g.cta = remap[g.cta]
    g.cta_kernel = np.array([0] * 5 + [1] * 6 + [2] * 10, np.uint32)
    g.cta_off = np.array([0, 21], np.uint32)
    rows = np.stack([_row(rng, s, c) for s, c in ((2, 1), (3, 2), (30, 1))])
    _check(g, rows, H.run_gpu(g, rows, kernel=IN_LANES))


def test_points_taken_by_cost_class():
    """More points than the scratch holds rows: the classes hand out every point once."""
    import torch

    from paper_2607_11262_gb300 import gts
    w = W.workload("wsgemm_small", points=120)
    dg = gts.DeviceGraph(w.graph)
    dp = gts.DeviceParams(dg, w.params)
    gts.gts_params_set_kernel(dp.handle, IN_LANES)
    row = (dg.row_nodes + 1) // 2 * 16
    assert gts.gts_batch_plan(dg.handle, dp.handle, 0, 120) & LANES
    few = torch.zeros(gts.GTS_SCRATCH_HEADER_BYTES + 7 * row, dtype=torch.uint8, device="cuda")
    full = gts.simulate(dg, dp, flags=gts.GTS_WANT_DIGEST)
    part = gts.simulate(dg, dp, first_point=11, n_points=90, flags=gts.GTS_WANT_DIGEST | gts.GTS_SCRATCH_CLEAN,
                        scratch=few)
    torch.cuda.synchronize()
    assert int(full.status.abs().sum()) == 0 and int(part.status.abs().sum()) == 0
    assert torch.equal(full.digest[11:101], part.digest) and torch.equal(full.makespan[11:101], part.makespan)
    assert int(torch.count_nonzero(few[gts.GTS_SCRATCH_HEADER_BYTES:])) == 0


@pytest.mark.parametrize("k", [64, 192])
def test_dense_slots_agree_with_padded_ones(k):
    """A batch of two waves runs with unpadded slots (3 per SM); its rows in batches of one wave do not."""
    import torch

    from paper_2607_11262_gb300 import gts
    g = W.ws_gemm(1024, 1024, k, 132, "ws")
    p = W.sweep_params(77, 3000, [W.AX_SMS, W.AX_HBM, W.AX_TMA_LAT, W.AX_MMA_RATE], 1)
    p[0, W.P_NUM_SMS] = 132
    dg = gts.DeviceGraph(g)
    dp = gts.DeviceParams(dg, p)
    gts.gts_params_set_kernel(dp.handle, IN_LANES)
    flags = gts.GTS_WANT_DIGEST | gts.GTS_WANT_BUSY
    assert gts.gts_batch_plan(dg.handle, dp.handle, 0, 3000) == LANES
    whole = gts.simulate(dg, dp, flags=flags)
    for lo in range(0, 3000, 600):
        assert gts.gts_batch_plan(dg.handle, dp.handle, lo, 600) == LANES | gts.GTS_PLAN_PADDED
        part = gts.simulate(dg, dp, first_point=lo, n_points=600, flags=flags)
        torch.cuda.synchronize()
        for f in ("status", "makespan", "digest", "busy"):
            assert torch.equal(getattr(whole, f)[lo:lo + 600], getattr(part, f)), (f, lo)
    assert int(whole.status.abs().sum()) == 0


def _with_l2(rng, p, tiles_bytes):
    p = p.copy()
    p[W.P_L2_BYTES], p[W.P_L2_LAT], p[W.P_L2_BPC] = int(rng.choice(tiles_bytes)), int(rng.integers(1, 9)), int(rng.choice([1, 2, 5]))
    return p


@pytest.mark.parametrize("tiles", [1, 7, 64, 3000])
def test_l2_lists(tiles):
    """The L2 list in shared memory."""
    rng = np.random.default_rng(7600 + tiles)
    for mix in (0, 2):
        g = _graph(rng, 220, 24, 3, mix, kernels=mix == 2)
        g.tile = rng.integers(max(0, tiles - 40), tiles, g.n_nodes).astype(np.uint32)
        g.tile[::6] = W.NO_TILE
        g.n_tiles = tiles
        rows = [_row(rng, int(rng.choice([2, 5, 40])), int(rng.integers(1, 3)), int(rng.integers(1, 3))) for _ in range(5)]
        rows = np.stack([rows[0]] + [_with_l2(rng, p, [1, 6, 30, 10**6]) for p in rows[1:]])
        _check(g, rows, H.run_gpu(g, rows, kernel=IN_LANES))


@pytest.mark.parametrize("tiles", [28906, 28907])
def test_l2_list_limit(tiles):
    """The longest list of a point with two SMs of three warps (299 other words, 58,112 in all), and one more tile,
    which the general instance runs."""
    rng = np.random.default_rng(7650)
    g = _graph(rng, 400, 30, 3, 0)
    g.tile = rng.integers(tiles - 90, tiles, g.n_nodes).astype(np.uint32)
    g.tile[::6] = W.NO_TILE
    g.n_tiles = tiles
    rows = np.stack([_with_l2(rng, _row(rng, 2, 1), [1, 30, 200, 10**6]) for _ in range(4)])
    rows[:, W.P_CAP_TENSOR:W.P_CAP_HBM + 1] = 1
    _check(g, rows, H.run_gpu(g, rows, kernel=IN_LANES), lanes=tiles == 28906)


@pytest.mark.parametrize("schedulers", [1, 2, 3, 4, 7, 32])
@pytest.mark.parametrize("policy", [W.POLICY_GTO, W.POLICY_RR])
def test_issue_policies(policy, schedulers):
    """Schedulers of a policy in the lanes, beside lowest-id rows and rows with an L2 list."""
    rng = np.random.default_rng(7700 + 40 * policy + schedulers)
    for mix in range(4):
        g = _graph(rng, 260, 30, 4, mix, kernels=mix == 1, p_issue=[0.0, 0.3, 0.8, 0.3][mix])
        g.tile = rng.integers(0, 9, g.n_nodes).astype(np.uint32)
        g.n_tiles = 9
        rows = []
        for k in range(6):
            p = _row(rng, int(rng.choice([2, 3, 8, 33])), int(rng.choice([1, 2, 4])), int(rng.choice([1, 2])),
                     int(rng.choice([1, 3])))
            if k:
                p[W.P_ISSUE_POLICY], p[W.P_SUBPARTITIONS] = policy, schedulers
            rows.append(_with_l2(rng, p, [8, 40]) if k == 5 else p)
        rows = np.stack(rows)
        _check(g, rows, H.run_gpu(g, rows, kernel=IN_LANES))


@pytest.mark.parametrize("seed", range(4))
def test_policies_agree_with_the_general_instance(seed):
    rng = np.random.default_rng(7800 + seed)
    g = _graph(rng, 500, 50, int(rng.integers(2, 6)), seed, max_work=[2, 6, 60, 6][seed])
    rows = []
    for k in range(24):
        p = _row(rng, int(rng.choice([2, 5, 31, 40])), int(rng.choice([1, 2])), int(rng.choice([1, 2, 4])))
        p[W.P_ISSUE_POLICY], p[W.P_SUBPARTITIONS] = 1 + k % 2, int(rng.choice([1, 2, 4]))
        rows.append(p)
    rows = np.stack(rows)
    lanes = H.run_gpu(g, rows, kernel=IN_LANES)
    assert lanes["plan"] & LANES
    both = H.run_gpu(g, rows, kernel=IN_GENERAL)
    assert not both["plan"] & LANES
    assert np.all(lanes["status"] == 0)
    for k in ("status", "makespan", "start", "finish", "digest", "cta_sm", "busy"):
        assert np.array_equal(lanes[k], both[k][:rows.shape[0]]), k


def _ws_rows(n, sms, cps, hbm=None, policy=0, schedulers=0):
    p = W.sweep_params(7, n, [W.AX_SMS, W.AX_HBM, W.AX_TMA_LAT, W.AX_MMA_RATE], 1)
    p[:, W.P_NUM_SMS], p[:, W.P_CTAS_PER_SM] = sms, cps
    if hbm:
        p[:, W.P_HBM_BPC] = hbm
    p[:, W.P_ISSUE_POLICY], p[:, W.P_SUBPARTITIONS] = policy, schedulers
    return p


@pytest.mark.parametrize("rows,lanes", [
    ((12, 132, 1), True), ((12, 132, 10), True), ((12, 2, 1), True), ((12, 4, 10), True), ((12, 1, 1), False),
    ((12, 2, 10), False), ((12, 4, 10, 32), False), ((12, 132, 1, 0, W.POLICY_RR, 1), True),
    ((12, 3, 1, 0, W.POLICY_GTO, 4), True), ((12, 132, 10, 64, W.POLICY_RR, 1), False),
    ((12, 2, 10, 0, W.POLICY_GTO, 4), False)])
def test_the_kernel_that_takes_less_time_runs(rows, lanes):
    """Rows on both sides of the estimate: SMs that a lane walks 30 slots of, few SMs, HBM that feeds one, policies."""
    g = W.ws_gemm(2048, 1024, 128, 132, "ws")
    p = _ws_rows(*rows)
    res = H.run_gpu(g, p)
    assert bool(res["plan"] & LANES) == lanes
    other = H.run_gpu(g, p, kernel=IN_GENERAL if lanes else IN_LANES)
    assert bool(other["plan"] & LANES) != lanes
    for k in ("status", "makespan", "start", "finish", "digest", "cta_sm", "busy"):
        assert np.array_equal(res[k], other[k]), k


def test_one_row_does_not_decide_for_the_table():
    """A sweep that starts at one SM runs in the lanes; scratch from the whole table serves any part of it."""
    import torch

    from paper_2607_11262_gb300 import gts
    g = W.ws_gemm(2048, 1024, 128, 132, "ws")
    p = np.concatenate([_ws_rows(40, 1, 1), _ws_rows(400, 132, 1)])
    dg = gts.DeviceGraph(g)
    dp = gts.DeviceParams(dg, p)
    assert gts.gts_batch_plan(dg.handle, dp.handle, 0, 440) & LANES
    assert not gts.gts_batch_plan(dg.handle, dp.handle, 0, 40) & LANES
    scratch = gts.alloc_scratch(dg, dp)
    flags = gts.GTS_WANT_DIGEST | gts.GTS_SCRATCH_CLEAN
    whole = gts.simulate(dg, dp, flags=flags, scratch=scratch)
    for lo, n in ((0, 40), (30, 300), (200, 240)):
        part = gts.simulate(dg, dp, first_point=lo, n_points=n, flags=flags, scratch=scratch)
        torch.cuda.synchronize()
        assert torch.equal(whole.digest[lo:lo + n], part.digest) and torch.equal(whole.makespan[lo:lo + n], part.makespan)
    assert int(whole.status.abs().sum()) == 0
    assert int(torch.count_nonzero(scratch[gts.GTS_SCRATCH_HEADER_BYTES:])) == 0
