"""Parity: the fp32 GPU scorer against the fp64 brute-force oracle -- relative
error <= 1e-6 per cost, identical argmin except where the oracle's top-two gap
is below 1e-5 relative (there the GPU's pick must itself be within 1e-5 of
the minimum)."""
import json
import os

import numpy as np
import pytest
import torch

from conftest import GOLDEN
from gpuutil import need_gpu
from paper_2609_16206_gb300 import workloads as W

pytestmark = pytest.mark.gpu
REL_COST = 1e-6
REL_GAP = 1e-5


def _run(ctr, p, oh, cls, Q, A, kap, consts, offset=0):
    dev = "cuda"

    def t(a, dt):  # optional element offset to break 16-byte alignment
        buf = torch.zeros(a.size + offset, dtype=dt, device=dev)
        buf[offset:] = torch.from_numpy(np.ascontiguousarray(a))
        return buf[offset:]
    n = p.size
    am = torch.full((n + offset,), -9, dtype=torch.int32, device=dev)[offset:]
    cost = torch.full((n + offset,), -9.0, dtype=torch.float32, device=dev)[offset:]
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    ctr.ctr_score_batch(t(p, torch.float32), t(oh, torch.float32), t(cls, torch.uint8), t(Q, torch.float32),
                        t(A, torch.float32), t(kap, torch.float32), consts, am, cost, status=status)
    torch.cuda.synchronize()
    assert int(status[0]) == 0
    return am.cpu().numpy(), cost.cpu().numpy()


def _check(orc, p, oh, cls, Q, A, kap, consts, am, cost):
    ref_am, best, second = orc.score_batch(p, oh, cls, Q, A, kap, consts)
    bad_cls = cls >= 4
    assert np.all(am[bad_cls] == -1) and np.all(np.isnan(cost[bad_cls]))
    ok = ~bad_cls
    with np.errstate(divide="ignore", invalid="ignore"):  # a zero minimum: inf (strict) or nan (a tie)
        gap = (second - best) / best
    strict = ok & (gap >= REL_GAP)
    assert np.array_equal(am[strict], ref_am[strict]), np.flatnonzero(am[strict] != ref_am[strict])[:5]
    idx = np.flatnonzero(ok)
    if idx.size == 0:
        return 0
    chosen = orc.score_pairs(p, oh, cls, idx, am[idx], Q, A, kap, consts)
    assert np.all(chosen <= best[idx] * (1 + REL_GAP) + 1e-30)
    rel = np.abs(cost[idx].astype(np.float64) - chosen) / np.maximum(chosen, 1e-30)
    assert rel.max() <= REL_COST, rel.max()
    return int((ok & ~strict).sum())


def test_standalone_batch_full_size(orc):
    """2^20 requests x 64 instances, the standalone scoring workload."""
    ctr = need_gpu()
    p, oh, cls = W.score_requests(1 << 20, seed=0)
    Q, A, kap = W.score_state(64, seed=1)
    am, cost = _run(ctr, p, oh, cls, Q, A, kap, W.SCORE_CONSTS)
    near = _check(orc, p, oh, cls, Q, A, kap, W.SCORE_CONSTS, am, cost)
    assert near < 1000


@pytest.mark.parametrize("n", [0, 1, 3, 5, 4097, 100_003])
@pytest.mark.parametrize("offset", [0, 1])
def test_ragged_and_misaligned(orc, n, offset):
    ctr = need_gpu()
    p, oh, cls = W.score_requests(n, seed=n + 3)
    Q, A, kap = W.score_state(64, seed=4)
    am, cost = _run(ctr, p, oh, cls, Q, A, kap, W.SCORE_CONSTS, offset=offset)
    _check(orc, p, oh, cls, Q, A, kap, W.SCORE_CONSTS, am, cost)


@pytest.mark.parametrize("n_inst", [1, 2, 7, 63, 64, 65, 256])
def test_instance_counts(orc, n_inst):
    ctr = need_gpu()
    p, oh, cls = W.score_requests(20_000, seed=n_inst)
    Q, A, kap = W.score_state(n_inst, seed=n_inst + 1)
    am, cost = _run(ctr, p, oh, cls, Q, A, kap, W.SCORE_CONSTS)
    _check(orc, p, oh, cls, Q, A, kap, W.SCORE_CONSTS, am, cost)


def test_degenerate_states(orc):
    ctr = need_gpu()
    p, oh, cls = W.score_requests(30_000, seed=77)
    cls = cls.copy()
    cls[::97] = 4
    cls[::101] = 255
    Q, A, kap = W.score_state(16, seed=78)
    cases = [
        (np.repeat(Q[:4], 4), np.repeat(A[:4], 4), np.repeat(kap[:4], 4)),   # duplicated instances
        (Q, A, np.zeros_like(kap)),                                            # no KV pressure
        (np.zeros_like(Q), np.zeros_like(A), kap),                             # idle pool
        (np.full_like(Q, 5.0), np.full_like(A, 3.0), np.full_like(kap, 0.5)),  # all equal
    ]
    for Qc, Ac, kc in cases:
        am, cost = _run(ctr, p, oh, cls, Qc, Ac, kc, W.SCORE_CONSTS)
        _check(orc, p, oh, cls, Qc, Ac, kc, W.SCORE_CONSTS, am, cost)
    zero_rho = W.SCORE_CONSTS.copy()
    zero_rho[3] = 0.0
    am, cost = _run(ctr, p, oh, cls, Q, A, kap, zero_rho)
    _check(orc, p, oh, cls, Q, A, kap, zero_rho, am, cost)


@pytest.mark.parametrize("n_inst", [9, 33, 64, 65, 130])
def test_every_line_on_the_envelope(orc, n_inst):
    """A state whose lower envelope holds every instance (queued tokens convex in
    the index, KV occupancy falling linearly): breakpoints at about 23 (2d + 1)
    tokens of o_hat, so the requests cross every segment, past the branch-free
    count of 8 segments and past 32 (the second register slot of the warp
    walk), and through the all-thread path for wider pools."""
    ctr = need_gpu()
    d = np.arange(n_inst)
    Q = (37.0 * d * d * (64.0 / n_inst) ** 2).astype(np.float32)
    A = np.zeros(n_inst, np.float32)
    kap = ((n_inst - d) / n_inst).astype(np.float32)
    n = 20_000
    rng = np.random.default_rng(n_inst)
    oh = np.floor(rng.random(n) * 3300.0).astype(np.float32)
    p = np.floor(rng.random(n) * 4000.0 + 16.0).astype(np.float32)
    cls = rng.integers(0, 4, n).astype(np.uint8)
    ref_am, _, _ = orc.score_batch(p, oh, cls, Q, A, kap, W.SCORE_CONSTS)
    assert np.unique(ref_am).size >= n_inst - 1  # the case exercises what it claims
    am, cost = _run(ctr, p, oh, cls, Q, A, kap, W.SCORE_CONSTS)
    _check(orc, p, oh, cls, Q, A, kap, W.SCORE_CONSTS, am, cost)


@pytest.mark.parametrize("n_inst", [64, 65, 95, 96, 97, 255, 256])
@pytest.mark.parametrize("state", ["random", "twins", "every_line", "one_slope", "falling"])
def test_wide_pool_envelopes(orc, n_inst, state):
    """Both sides of the 64-instance line and of whole warps: random lines, pairs of equal ones, an envelope of every
    line, parallel lines (one segment), and lines each below the one before it at every o_hat (the last one wins)."""
    ctr = need_gpu()
    rng = np.random.default_rng(n_inst)
    d = np.arange(n_inst)
    Q = rng.integers(0, 65536, n_inst).astype(np.float32)
    A = rng.integers(0, 256, n_inst).astype(np.float32)
    kap = rng.random(n_inst, dtype=np.float32)
    if state == "twins":
        Q, A, kap = (np.repeat(v[:(n_inst + 1) // 2], 2)[:n_inst] for v in (Q, A, kap))
    elif state == "every_line":
        Q, A = (37.0 * d * d * (64.0 / n_inst) ** 2).astype(np.float32), np.zeros(n_inst, np.float32)
        kap = ((n_inst - d) / n_inst).astype(np.float32)
    elif state == "one_slope":
        kap[:] = 0.25
    elif state == "falling":
        Q, A = (1000.0 * (n_inst - d)).astype(np.float32), np.zeros(n_inst, np.float32)
        kap = ((n_inst - d) / n_inst).astype(np.float32)
    n = 6_001
    oh = np.floor(rng.random(n) * 3300.0).astype(np.float32)
    p = np.floor(rng.random(n) * 4000.0 + 16.0).astype(np.float32)
    cls = rng.integers(0, 4, n).astype(np.uint8)
    am, cost = _run(ctr, p, oh, cls, Q, A, kap, W.SCORE_CONSTS)
    _check(orc, p, oh, cls, Q, A, kap, W.SCORE_CONSTS, am, cost)


def test_hand_computed_exact(orc):
    ctr = need_gpu()
    with open(os.path.join(GOLDEN, "score_hand.json")) as f:
        h = json.load(f)
    r, s, e = h["requests"], h["state"], h["expect"]
    f32 = lambda x: np.array(x, np.float32)
    am, cost = _run(ctr, f32(r["p"]), f32(r["oh"]), np.array(r["cls"], np.uint8), f32(s["Q"]), f32(s["A"]),
                    f32(s["kappa"]), np.array(h["consts"], np.float32))
    assert am[3] == -1 and np.isnan(cost[3])
    # requests 0..2 tie between instances 2 and 3: either is a valid argmin, the cost is exact
    assert set(am[:3].tolist()) <= {2, 3}
    assert cost[:3].tolist() == e["best"][:3]


def test_invalid_arguments():
    ctr = need_gpu()
    x = torch.zeros(8, device="cuda")
    c = torch.zeros(8, dtype=torch.uint8, device="cuda")
    am = torch.zeros(8, dtype=torch.int32, device="cuda")
    bad = W.SCORE_CONSTS.copy()
    bad[0] = -1.0
    with pytest.raises(ctr.CtrError):
        ctr.ctr_score_batch(x, x, c, x, x, x, bad, am, x)
    big = torch.zeros(257, device="cuda")
    with pytest.raises(ctr.CtrError):
        ctr.ctr_score_batch(x, x, c, big, big, big, W.SCORE_CONSTS, am, x)


@pytest.mark.parametrize("seed", range(48))
def test_random_scoring_problems(orc, seed):
    """Seeded random problems: 1-256 instances (duplicated ones give exact ties), constants with zero
    weights, classes including invalid ones, aligned and misaligned buffers."""
    ctr = need_gpu()
    rng = np.random.default_rng(500 + seed)
    n_inst = int(rng.choice([1, 2, 5, 17, 64, 65, 130, 256]))
    n = int(rng.choice([0, 1, 7, 1000, 20_001]))
    p = np.floor(rng.exponential(800.0, n)).astype(np.float32)
    oh = np.floor(rng.exponential(400.0, n) + rng.integers(0, 2, n)).astype(np.float32)
    cls = rng.integers(0, 5 if seed % 3 == 0 else 4, n).astype(np.uint8)
    Q = rng.integers(0, 1 << int(rng.integers(1, 17)), n_inst).astype(np.float32)
    A = rng.integers(0, 1 << int(rng.integers(1, 9)), n_inst).astype(np.float32)
    kap = rng.random(n_inst, dtype=np.float32)
    if n_inst > 1 and seed % 4 == 1:  # duplicated instances: exact ties broken by index
        j = rng.integers(0, n_inst, n_inst // 2)
        Q[j], A[j], kap[j] = Q[0], A[0], kap[0]
    consts = W.SCORE_CONSTS.copy()
    consts[:9] *= rng.choice([0.0, 0.5, 1.0, 3.0], 9).astype(np.float32)
    consts[8] = np.float32(1.0 / float(rng.choice([1e4, 2e5, 1e6])))
    consts[9:] = rng.choice([0.5, 1.0, 2.0], 4).astype(np.float32)
    if consts[:8].max() == 0:
        consts[0] = 1.0
    am, cost = _run(ctr, p, oh, cls, Q, A, kap, consts, offset=int(seed % 2))
    if n:
        _check(orc, p, oh, cls, Q, A, kap, consts, am, cost)


def test_chained_launches_read_completed_outputs():
    """The scorer is launched as a programmatic dependent launch: a call that
    reads the previous call's output on the same stream (no host sync in
    between) must see it complete.  Call 1's costs are call 2's prompt
    lengths; a fill kernel clobbers both output buffers first, so a read that
    ran ahead of its producer would see NaN or stale values."""
    ctr = need_gpu()
    n = 1 << 20
    p, oh, cls = W.score_requests(n, seed=5)
    Q, A, kap = W.score_state(64, seed=6)
    d = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)
    dp, dcls, dQ, dA, dk = d(p, torch.float32), d(cls, torch.uint8), d(Q, torch.float32), d(A, torch.float32), \
        d(kap, torch.float32)
    am1 = torch.empty(n, dtype=torch.int32, device="cuda")
    am2 = torch.empty_like(am1)
    c1 = torch.empty(n, dtype=torch.float32, device="cuda")
    c2 = torch.empty_like(c1)
    for it in range(8):
        doh = d(oh * (1 + it % 3), torch.float32)
        c1.fill_(float("nan"))
        c2.fill_(float("nan"))
        ctr.ctr_score_batch(dp, doh, dcls, dQ, dA, dk, W.SCORE_CONSTS, am1, c1)
        ctr.ctr_score_batch(c1, doh, dcls, dQ, dA, dk, W.SCORE_CONSTS, am2, c2)
        torch.cuda.synchronize()
        ref_am = torch.empty_like(am2)
        ref_c = torch.empty_like(c2)
        ctr.ctr_score_batch(c1.clone(), doh, dcls, dQ, dA, dk, W.SCORE_CONSTS, ref_am, ref_c)
        torch.cuda.synchronize()
        assert not torch.isnan(c1).any() and not torch.isnan(c2).any(), it
        assert torch.equal(am2, ref_am) and torch.equal(c2, ref_c), it


@pytest.mark.parametrize("n_inst", [65, 200, 256])
def test_wide_pool_slopes_past_2_to_126(n_inst):
    """Slopes so far apart that a division which flushes the reciprocals of denominators above 2^126 puts the crossing of
    the first two lines at 0 (the cost is 1e37 against 2e36 there)."""
    ctr = need_gpu()
    consts = np.array([1, 1, 0, 1, 0, 1, 1, 0, 0, 1, 0.5, 1, 1], np.float32)
    Q, kap = np.full(n_inst, 2e38, np.float32), np.zeros(n_inst, np.float32)
    i, j = n_inst // 3, n_inst - 2
    Q[i], kap[i], Q[j], kap[j] = 0, 2e38, 1e37, 1e37
    oh = np.linspace(0, 0.2, 4_001, dtype=np.float32)
    p, A, cls = np.ones_like(oh), np.zeros(n_inst, np.float32), (np.arange(oh.size) % 4).astype(np.uint8)
    am, cost = _run(ctr, p, oh, cls, Q, A, kap, consts)
    c64 = Q.astype(np.float64)[None] + p[:, None] + oh[:, None].astype(np.float64) * (1 + kap.astype(np.float64)[None])
    c64 *= np.where(cls == 1, 0.5, 1.0)[:, None]
    best = c64.min(1)
    assert np.all(c64[np.arange(oh.size), am] <= best * (1 + 1e-6))  # a tie within fp32 roundings may go either way
    assert np.max(np.abs(cost - best) / best) <= 2e-6
