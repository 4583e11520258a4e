"""Sampled tokens masked with the lowest finite logit (-3.4e38, the usual
mask where -inf is avoided): their log-probs, and every sum over them, are
finite in fp64, whichever kernel scans the window."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import SUM_RTOL, oracle_batch, run_batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stride():
    import paper_2609_14636_gb300 as s

    return s


def _masked(rng, rows, V, f32, turns):
    """Trajectories of `turns`; in each, one turn (the third, fourth, ... in
    rotation) with masked sampled tokens: once in T, twice, once in S, once in
    both."""
    assert rows % sum(turns) == 0
    lay = synth.layout_from_turn_lengths([list(turns)] * (rows // sum(turns)))
    S32 = rng.standard_normal((rows, V), dtype=np.float32)
    T32 = S32 + rng.standard_normal((rows, V), dtype=np.float32) * np.float32(0.3)
    S, T = (S32, T32) if f32 else (synth.bf16_bits_from_f32(S32), synth.bf16_bits_from_f32(T32))
    low = np.finfo(np.float32).min if f32 else np.uint16(0xFF7F)
    tok = rng.integers(0, V, rows).astype(np.int32)
    for i in range(lay.n_traj):
        k = lay.traj_turn_off[i] + 2 + i % (len(turns) - 2)
        a, b = lay.turn_row_off[k], lay.turn_row_off[k + 1]
        in_s, in_t = [((), (0,)), ((), (0, 2)), ((1,), ()), ((3,), (3,))][i % 4]
        for x, at in ((S, in_s), (T, in_t)):
            for j in at:
                if a + j < b:
                    x[a + j, tok[a + j]] = low
    return lay, S, T, tok


def _compare(g, o, lay, mode):
    """Stops and counts exact (no test is near lambda); sums within 1e-5 of the summed magnitudes (one log-prob's
    rounding is 2 ulp of its log-sum-exp)."""
    lt, d = o["logp_t"], o["d"]
    ls = lt + d
    fin = [np.abs(v) + 1.0 for v in (lt, d)] + [np.abs(ls * d) + np.abs(ls) + np.abs(d) + 1.0]
    mag = [np.add.reduceat(v, lay.turn_row_off[:-1]) for v in fin]
    ts, st = g["turn_stats"], g["state"]
    for f, ref, m in zip(("sum_t", "sum_d", "sum_l"), ("turn_sum_t", "turn_sum_d", "turn_sum_l"), mag):
        assert np.all(np.isfinite(ts[f])), f
        assert np.all(np.abs(ts[f] - o[ref]) <= SUM_RTOL * m), f
    np.testing.assert_allclose(ts["mean_t"], o["turn_mean"], rtol=SUM_RTOL)
    np.testing.assert_allclose(ts["cum"], o["turn_cum"], rtol=SUM_RTOL)
    np.testing.assert_allclose(st["cum"], o["traj_cum"], rtol=SUM_RTOL)
    for f in ("stop_row", "stop_turn"):
        assert np.array_equal(st[f], o[f]), f
    assert np.array_equal(st["loss_tokens"], o["traj_loss_tokens"])
    loss = np.add.reduceat(fin[2], lay.traj_row_off[:-1])
    assert np.all(np.abs(st["loss"] - o["traj_loss"]) <= SUM_RTOL * loss)
    prof = [np.sum(v) for v in fin[:2]]
    for k in range(2):
        assert np.all(np.abs(g["profile"][:, 1 - k] - o["profile"][:, 1 - k]) <= SUM_RTOL * prof[k]), k


# Up to 1,216 rows a window takes the small-window kernel and the cluster scan (tiles of 128 rows).  From there on, below
# 57,344 logits the scan follows the persistent kernel, else it runs inside.  Windows of both kinds carry state across.
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("rows, V, f32", [(1300, 32_000, False), (2600, 4_099, True), (1300, 57_343, False),
                                          (1300, 57_344, False), (80_000, 64, False), (100, 64, True), (700, 32_000, False),
                                          (1200, 4_099, False)])
def test_lowest_finite_logit(stride, rows, V, f32, mode):
    rng = np.random.default_rng(rows + V + mode)
    lay, S, T, tok = _masked(rng, rows, V, f32, (7, 20, 33, 4, 36))
    lam = np.float32(-1e6)  # only a masked log-prob crosses it
    o = oracle_batch(S, T, tok, lay, mode, lam)
    half = rows // 2 - 13
    for windows in (None, [(0, half), (half, rows)], [(0, half), (half, half + 30), (half + 30, rows)]):
        g = run_batch(stride, S, T, tok, lay, mode, lam, windows=windows)
        assert g["status"] == 0
        _compare(g, o, lay, mode)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("rows", [300, 1300, 80_000])  # one tile, some, two rows per thread
def test_lowest_finite_log_probs(stride, rows, mode):
    """The same on given log-probs."""
    import torch

    rng = np.random.default_rng(rows + mode)
    lay, _, _, _ = _masked(rng, rows, 64, False, (7, 20, 33, 4, 36))
    lt = -rng.exponential(4.0, rows).astype(np.float32) - np.float32(0.05)
    ls = np.minimum(lt + rng.normal(0.0, 0.5, rows), -0.05).astype(np.float32)
    low = np.finfo(np.float32).min
    for i in range(lay.n_traj):
        a = lay.turn_row_off[lay.traj_turn_off[i] + 2 + i % 3]
        for x, at in ((lt, ((0,), (0, 2), (), (3,))[i % 4]), (ls, ((), (), (1,), (3,))[i % 4])):
            for j in at:
                if a + j < rows:
                    x[a + j] = low
    lam = np.float32(-1e6)
    d = (ls - lt).astype(np.float64)
    o = oracle.scan_batch(lt.astype(np.float64), d, lay.traj_row_off, lay.turn_row_off, lay.traj_turn_off, mode,
                          np.float64(lam), logp_s=ls.astype(np.float64))
    o.update(logp_t=lt.astype(np.float64), d=d)
    off = [torch.from_numpy(a).cuda() for a in (lay.traj_row_off, lay.turn_row_off, lay.traj_turn_off)]
    gs, gt = torch.from_numpy(ls).cuda(), torch.from_numpy(lt).cuda()
    ws = torch.empty(stride.stride_score_batch_workspace_size(rows), dtype=torch.uint8, device="cuda")
    for edges in ((0, rows), (0, rows // 2 - 13, rows)):
        st, ts, pr = stride.new_state(lay.n_traj), stride.new_turn_stats(lay.n_turns), stride.new_profile()
        for a, b in zip(edges[:-1], edges[1:]):
            stride.stride_scan_logprobs(gs[a:b], gt[a:b], *off, a, b, mode, float(lam), st, turn_stats=ts, workspace=ws,
                                        profile=pr)
        torch.cuda.synchronize()
        _compare({"turn_stats": stride.turn_stats_to_numpy(ts)[:lay.n_turns], "state": stride.state_to_numpy(st)[:lay.n_traj],
                  "profile": pr.cpu().numpy()}, o, lay, mode)
