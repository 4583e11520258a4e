"""Which tokens a stopped trajectory keeps: all up to the turn (token) that
fired and none after, also where the threshold lies within a rounding of the
recorded sum, where a window begins inside a turn, and where tokens after the
stop are masked."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import oracle_batch, run_batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stride():
    import paper_2609_14636_gb300 as s

    return s


def _layout(rng, rows):
    lens, left = [], rows
    while left > 0:
        turns = []
        for _ in range(int(rng.integers(3, 12))):
            n = min(left, 1 if rng.random() < 0.2 else int(rng.integers(2, 130)))
            left -= n
            if n:
                turns.append(n)
        lens.append(turns)
    return synth.layout_from_turn_lengths(lens)


def _cuts(rows, k):
    return [(rows * i // k, rows * (i + 1) // k) for i in range(k)]


def _kept_rows(st, lay, mode):
    """Rows kept according to the recorded stop."""
    n = np.diff(lay.traj_row_off)
    if mode == oracle.TOKEN_SUM:
        return np.where(st["stopped"] != 0, st["stop_row"] + 1, n)
    turn = np.minimum(lay.traj_turn_off[:-1] + st["stop_turn"] + 1, lay.n_turns)
    return np.where(st["stopped"] != 0, lay.turn_row_off[turn] - lay.traj_row_off[:-1], n)


ROUTES = [("split", 700, 64), ("split", 1900, 64), ("stream", 1500, 64), ("stream", 50_000, 16), ("stream", 300, 57_344),
          ("rows", 900, 64), ("scan", 250, 0), ("scan", 9000, 0), ("scan", 60_000, 0), ("scan", 4096 * 512 + 700, 0)]


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("route, rows, V", ROUTES)
def test_threshold_at_a_recorded_sum(stride, route, rows, V, mode):
    """lambda = the running sum after one of the trajectory's turns, rounded to fp32 (1e-8 to 6e-8 off, either way), or,
    where the log-probs' grid and the turn's length allow it, the sum itself but for the rounding of its quotients."""
    import torch

    rng = np.random.default_rng(rows + mode)
    lay = _layout(rng, rows)
    off = [torch.from_numpy(a).cuda() for a in (lay.traj_row_off, lay.turn_row_off, lay.traj_turn_off)]
    ws = torch.empty(stride.stride_score_batch_workspace_size(rows), dtype=torch.uint8, device="cuda")
    lt = torch.from_numpy(-rng.exponential(4.0, rows).astype(np.float32) - np.float32(0.05)).cuda()
    ls = torch.clamp(lt + 0.5 * torch.from_numpy(rng.standard_normal(rows).astype(np.float32)).cuda(), max=-0.05)
    if V:
        x = torch.from_numpy(rng.standard_normal((rows, V), dtype=np.float32)).cuda()
        y = x + 0.3 * torch.from_numpy(rng.standard_normal((rows, V), dtype=np.float32)).cuda()
        tok = torch.from_numpy(rng.integers(0, V, rows).astype(np.int32)).cuda()

    def run(lam, windows):
        st, ts = stride.new_state(lay.n_traj), stride.new_turn_stats(lay.n_turns)
        for a, b in windows:
            if V:
                stride.stride_score_batch(x[a:b], y[a:b], tok[a:b], *off, a, b, mode, lam, st, turn_stats=ts, workspace=ws)
            else:
                stride.stride_scan_logprobs(ls[a:b], lt[a:b], *off, a, b, mode, lam, st, turn_stats=ts, workspace=ws)
        torch.cuda.synchronize()
        return stride.state_to_numpy(st)[:lay.n_traj], stride.turn_stats_to_numpy(ts)[:lay.n_turns]

    if V:
        stride.stride_force_batch_kernel(route)
    try:
        for windows in (_cuts(rows, 1), _cuts(rows, 2), _cuts(rows, 5)):
            cum = run(-1e30, windows)[1]["cum"]
            for _ in range(3 if rows > 1_000_000 else 12):
                pick = lay.traj_turn_off[:-1] + (rng.random(lay.n_traj) * np.diff(lay.traj_turn_off)).astype(int)
                lam = cum[pick].astype(np.float32)
                st, _ = run(torch.from_numpy(lam).cuda(), windows)
                assert lay.n_traj < 9 or (st["stopped"] != 0).sum() > lay.n_traj // 4
                np.testing.assert_array_equal(st["loss_tokens"], _kept_rows(st, lay, mode))
    finally:
        stride.stride_force_batch_kernel("auto")


@pytest.mark.parametrize("route, rows, V", ROUTES[1:6])
def test_threshold_equal_to_a_sum(stride, route, rows, V):
    """Every log pi_T is the same number p, so every turn's mean is p, and the running sum after two turns is the fp32
    number 2 p but for the rounding of the quotients p / n: equal to lambda, not below it.  The third turn stops.  (The
    cluster scan rounds the quotients to fp32, so there only the kept tokens agree with the stop.)"""
    import torch

    rng = np.random.default_rng(rows)
    lay = _layout(rng, rows)
    x = torch.from_numpy(rng.standard_normal((rows, V), dtype=np.float32)).cuda()
    y = torch.zeros((rows, V), device="cuda")
    tok = np.zeros(rows, np.int32)
    stride.stride_force_batch_kernel(route)
    try:
        p = run_batch(stride, x, y, tok, lay, 0, np.float32(-1e30))["logp_t"]
        assert np.all(p == p[0])
        for k in (1, 2, 5):
            st = run_batch(stride, x, y, tok, lay, 0, np.float32(2 * p[0]), windows=_cuts(rows, k))["state"]
            if route != "split":
                third = np.minimum(2, np.diff(lay.traj_turn_off) - 1)
                np.testing.assert_array_equal(st["stop_turn"], np.where(third == 2, 2, -1))
            np.testing.assert_array_equal(st["loss_tokens"], _kept_rows(st, lay, 0))
    finally:
        stride.stride_force_batch_kernel("auto")


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("low", [-np.inf, np.finfo(np.float32).min])
@pytest.mark.parametrize("route, rows, V", [r for r in ROUTES if r[2]])
def test_masked_tokens_after_a_stop(stride, route, rows, V, low, mode):
    """Sampled tokens with a masked teacher logit, once to three times in a turn, most of them after the stop."""
    rng = np.random.default_rng(rows + V + mode)
    lay = _layout(rng, rows)
    S = rng.standard_normal((rows, V), dtype=np.float32)
    T = S + rng.standard_normal((rows, V), dtype=np.float32) * np.float32(0.3)
    tok = rng.integers(0, V, rows).astype(np.int32)
    for k in range(lay.n_turns):
        a, b = lay.turn_row_off[k], lay.turn_row_off[k + 1]
        for r in a + np.unique(rng.integers(0, b - a, [0, 0, 1, 2, 3][k % 5])):
            T[r, tok[r]] = low
    lam = rng.uniform(-40.0, -6.0, lay.n_traj).astype(np.float32)
    o = oracle_batch(S, T, tok, lay, mode, lam)
    stride.stride_force_batch_kernel(route)
    try:
        for k in (1, 2, 5):
            g = run_batch(stride, S, T, tok, lay, mode, lam, windows=_cuts(rows, k))
            assert g["status"] == 0
            np.testing.assert_array_equal(g["state"]["stop_row"], o["stop_row"])
            np.testing.assert_array_equal(g["state"]["stop_turn"], o["stop_turn"])
            np.testing.assert_array_equal(g["state"]["loss_tokens"], o["traj_loss_tokens"])
    finally:
        stride.stride_force_batch_kernel("auto")
