"""The kernels of the simulator and of the goodput pass on the CPU (simlanes), the lanes of a warp as far
apart as its barriers allow: every row the oracle's, and no access to shared
structures that only a lockstep warp would keep in order."""
import numpy as np
import pytest

import simlanes
from paper_2609_16206_gb300 import workloads as W

ALL_FIVE = list(W.ALL_POLICIES) + [W.POLICY_LEARNED_P2]


@pytest.fixture(scope="module")
def lanes(tmp_path_factory):
    return simlanes.build(str(tmp_path_factory.mktemp("simlanes")))


def check(orc, lanes, sc, sets, pols, traces, order, **kw):
    res, races, stuck = simlanes.simulate(lanes, sc, sets, pols, traces, order=order, **kw)
    assert (races, stuck) == (0, 0)
    row = 0
    for tr in traces:
        for cc in sets:
            for pol in pols:
                o = orc.simulate(sc, cc, pol, tr)
                assert res["status"][row] == o["status"], (row, pol)
                if o["status"] == 0:
                    assert int(res["hash"][row]) == o["hash"], (row, pol)
                    for key in ("t_first_us", "t_done_us", "i_pre", "i_dec"):
                        assert np.array_equal(res[key][row], o[key]), (row, pol, key)
                row += 1
    return res


@pytest.mark.parametrize("order", [0, 1, 7])
@pytest.mark.parametrize("sc,deployed", [
    (W.SimCfg(), 0), (W.SimCfg(n_prefill=2, n_decode=7), 1),
    (W.SimCfg(n_prefill=2, n_decode=2, kv_cap_tokens=16_000), 0),  # requests wait in the FIFO
    (W.SimCfg(n_decode=1, pre_base_us=1, pre_us_per_tok=0), 0),  # heaps of more than 33 keys
    (W.SimCfg(n_prefill=2, n_decode=2, kv_cap_tokens=16_000, cap_active=9, cap_waiting=8, cap_pending=8), 1)],
    ids=["1p3d", "2p7d", "scarce", "deep", "small_caps"])
def test_block_per_row(orc, lanes, sc, deployed, order):
    tc = W.replica_sweep().trace.replace(rate_mreq=(8_000, 60_000), prompt_max=min(8192, sc.kv_cap_tokens // 2))
    sets = [W.as_deployed(W.CALIBRATED) if deployed else W.CALIBRATED]
    check(orc, lanes, sc, sets, ALL_FIVE, [orc.gen_trace(tc, 150)], order)


@pytest.mark.parametrize("order", [0, 1, 7])
@pytest.mark.parametrize("sc,ws_rows", [
    (W.SimCfg(prefill_batch_tokens=2048), None), (W.SimCfg(n_prefill=3, n_decode=5, prefill_batch_tokens=900), 1),
    (W.SimCfg(n_prefill=2, n_decode=2, kv_cap_tokens=16_000, cap_active=9, cap_waiting=8, prefill_batch_tokens=4096), 1),
    (W.SimCfg(n_prefill=2, n_decode=6), 1), (W.SimCfg(n_prefill=4, n_decode=13), None)],
    ids=["batched", "batched_packed", "batched_small_caps", "packed", "4p13d"])
def test_rows_in_warps(orc, lanes, sc, ws_rows, order):
    """A row or (ws_rows=1: a workspace of one slot) several to a warp; with batched prefill the decode lanes read the
    prefill lanes' rings."""
    tc = W.replica_sweep().trace.replace(rate_mreq=(8_000, 60_000), prompt_max=min(8192, sc.kv_cap_tokens // 2))
    sets = [W.CALIBRATED, W.as_deployed(W.CALIBRATED)]
    check(orc, lanes, sc, sets, ALL_FIVE, [orc.gen_trace(tc, 90)], order, ws_rows=ws_rows)


def _two_failures(max_steps, burst_at=40):
    """Round robin on two decode instances: the even requests run instance 0 out of its steps, then a burst at one
    instant has more requests pending than either instance may hold."""
    k = np.arange(burst_at + 20)
    tr = {"arrival_us": np.minimum(k, burst_at) * 10_000, "prompt_len": np.full(k.size, 10), "true_out": np.where(k % 2, 1, 8),
          "pred_out": np.full(k.size, 4), "slo_class": k % 2}
    return W.SimCfg(n_prefill=1, n_decode=2, pre_base_us=100, pre_us_per_tok=0, xfer_us_per_tok=1, dec_base_us=1_000,
                    cap_pending=4, max_steps_per_instance=max_steps), tr


@pytest.mark.parametrize("max_steps,status", [(100, -4), (152, -4), (153, -4), (161, -3), (1 << 20, -3)])
@pytest.mark.parametrize("ws_rows", [None, 1])
def test_first_failure_is_the_rows(orc, lanes, max_steps, status, ws_rows):
    """A row's status is that of its first failure, in a block per row (where round-robin warps do not meet) as in a
    warp."""
    sc, tr = _two_failures(max_steps)
    res = check(orc, lanes, sc, [W.CALIBRATED], [W.POLICY_RR] * 3 + [W.POLICY_JSQ] * 2, [tr] * 4, 0, ws_rows=ws_rows)
    assert (res["status"].reshape(4, 5)[:, :3] == status).all()


def _trace(rows):
    """(arrival, prompt, output) per request."""
    a = np.array(rows).T
    return {"arrival_us": a[0], "prompt_len": a[1], "true_out": a[2], "pred_out": a[2] % 512, "slo_class": a[0] * 0}


# two decode instances in turns, 1 ms steps; every request KV-ready at once
_BASE = W.SimCfg(n_prefill=1, n_decode=2, pre_base_us=1, pre_us_per_tok=0, xfer_us_per_tok=0, dec_base_us=1_000,
                 dec_us_per_seq=0, dec_kv_tokens_per_us=1 << 31, kv_cap_tokens=5_000)


@pytest.mark.parametrize("name,sc,rows,status", [
    # instance 0 runs out of steps in the middle of a long run, then a burst overflows the pending heap of instance 1
    ("budget_in_a_run", _BASE.replace(max_steps_per_instance=50, cap_pending=3, pre_base_us=500),
     [(0, 1, 2000), (0, 1, 1)] + [(200_000, 1, 1)] * 12, -4),
    # instance 0's FIFO overflows behind a request that fills its KV, long before instance 1 runs out of steps
    ("fifo_behind_its_head", _BASE.replace(max_steps_per_instance=900, cap_waiting=2),
     [(0, 1, 4500), (0, 1, 2000)] + [(10_000 + 1000 * k, 1, 800 if k % 2 == 0 else 1) for k in range(12)] +
     [(3_000_000, 1, 1)], -3),
    # the same FIFO, filled to its last place: instance 0 runs out of steps
    ("fifo_full", _BASE.replace(max_steps_per_instance=900, cap_waiting=6),
     [(0, 1, 4500), (0, 1, 2000)] + [(10_000 + 1000 * k, 1, 800 if k % 2 == 0 else 1) for k in range(12)] +
     [(3_000_000, 1, 1)], -4),
    # a FIFO overflow at the very step end at which the budget is used up
    ("both_at_one_step_end", _BASE.replace(max_steps_per_instance=40, cap_waiting=3),
     [(0, 1, 40), (0, 1, 1)] + [(39_500, 1, 30), (39_500, 1, 1)] * 4, -3)], ids=lambda v: v if isinstance(v, str) else "")
@pytest.mark.parametrize("ws_rows", [None, 1])
def test_failure_inside_a_run_of_steps(orc, lanes, name, sc, rows, status, ws_rows):
    """What fails between two events of an instance fails before what another instance does later."""
    tr = _trace(rows)
    res = check(orc, lanes, sc, [W.CALIBRATED], [W.POLICY_RR] * 5, [tr] * 2, 0, ws_rows=ws_rows)
    assert (res["status"] == status).all(), res["status"]
    sc = sc.replace(prefill_batch_tokens=1)
    check(orc, lanes, sc, [W.CALIBRATED], [W.POLICY_RR, W.POLICY_LEARNED], [tr], 0, ws_rows=ws_rows)


@pytest.mark.parametrize("order", [0, 1, 7])
@pytest.mark.parametrize("N", [1, 130, 1500, 3001])
@pytest.mark.parametrize("shape", ["spread", "narrow", "tie_below", "equal", "small", "negative", "wide"])
def test_goodput(orc, lanes, shape, N, order):
    """The goodput pass with both P99s: thresholds of spread, crowded and equal values, bins of a single value with more
    members than are counted out (small), and rows that are selected from memory."""
    rng = np.random.default_rng(N)
    R, u = 2, rng.random((2, N))
    v = {"spread": rng.integers(1, 10**7, (R, N)), "narrow": np.floor(15_500 * np.exp(0.008 * rng.standard_normal((R, N)))),
         "tie_below": np.where(u < 0.88, rng.integers(14_000, 15_000, (R, N)), np.where(u < 0.975, 15_204, 15_290)),
         "equal": np.full((R, N), 15_204), "small": rng.integers(1, 9, (R, N)), "negative": rng.integers(-500, 3, (R, N)),
         "wide": (1 << 33) + rng.integers(0, 1000, (R, N))}[shape].astype(np.int64)
    o = rng.integers(1, 400, (R, N))
    tr = {"arrival_us": np.sort(rng.integers(0, 10**9, (R, N)), axis=1), "prompt_len": np.ones((R, N)), "true_out": o,
          "pred_out": np.ones((R, N)), "slo_class": rng.integers(0, 2, (R, N))}
    tf = tr["arrival_us"] + v
    td = tf + rng.permutation(v.T).T * np.maximum(o - 1, 0)
    (met, p99, tpot), races, stuck = simlanes.goodput(lanes, W.SimCfg(), tr, tf, td, order)
    assert (races, stuck) == (0, 0)
    for r in range(R):
        assert (met[r], p99[r]) == orc.goodput(W.SimCfg(), {k: x[r] for k, x in tr.items()}, tf[r], td[r])
        assert tpot[r] == orc.p99_tpot({"true_out": o[r]}, tf[r], td[r])
