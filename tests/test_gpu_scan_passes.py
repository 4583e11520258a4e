"""The scan on given log-probs at the sizes where its tiles can go wrong:
windows that end inside, at and just past a tile of one row per thread (256)
and of two (512, from 152 x 256 rows on), turns of one row, empty
trajectories, one trajectory over all tiles, and more tiles than a tile folds
by itself.  Against the sums in 64 bits; sums that no rounding of a term
touches to the accuracy that the scan states, and the same after a scoring
kernel, against the sums of the log-probs that it returned."""
from __future__ import annotations

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stride():
    import paper_2609_14636_gb300 as s

    return s


ONE_WAVE = 152 * 256


def _layout(rng, rows, shape):
    if shape == "one":
        return synth.layout_from_turn_lengths([[rows]])
    if shape == "turns":  # one trajectory of turns of 1 to 3,000 rows
        cut = np.unique(np.concatenate([rng.integers(1, rows, max(rows // 700, 1)), [rows]])) if rows > 1 else np.array([rows])
        return synth.layout_from_turn_lengths([np.diff(np.concatenate([[0], cut])).tolist()])
    lens, left = [], rows  # "mixed": 1-4 turns of 1-300 rows (half of them 1), now and then empty trajectories
    while left > 0:
        turns = []
        for _ in range(int(rng.integers(1, 5))):
            n = min(left, 1 if rng.random() < 0.5 else int(rng.integers(2, 301)))
            if n:
                turns.append(n)
            left -= n
        lens.append(turns)
        if rng.random() < 0.05:
            lens.extend([[]] * 30)
    return synth.layout_from_turn_lengths(lens)


def _reference(ls, lt, lay, mode, lam):
    ls, lt = ls.astype(np.float64), lt.astype(np.float64)
    d = ls - lt
    tr, tu, first = lay.traj_row_off, lay.turn_row_off, lay.traj_turn_off
    n = np.diff(tu)
    sums = [np.add.reduceat(v, tu[:-1]) for v in (lt, d, ls * d)]
    cum, loss = np.zeros(lay.n_turns), np.zeros(lay.n_traj)
    stop = np.full(lay.n_traj, -1, np.int64)
    total, margin = np.zeros(lay.n_traj), np.full(lay.n_traj, np.inf)
    for i in range(lay.n_traj):
        k0, k1, r0, r1 = first[i], first[i + 1], tr[i], tr[i + 1]
        if r0 == r1:
            continue
        if mode == 0:
            c = np.cumsum(sums[0][k0:k1] / n[k0:k1])
            cum[k0:k1], at = c, tu[k0 + 1:k1 + 1] - 1
        else:
            c = np.cumsum(lt[r0:r1])
            cum[k0:k1], at = c[tu[k0 + 1:k1 + 1] - 1 - r0], np.arange(r0, r1)
        total[i], margin[i] = c[-1], np.min(np.abs(c - lam) / np.abs(lam))
        hit = np.nonzero(c < lam)[0]
        end = r1
        if len(hit):
            stop[i] = at[hit[0]] - r0
            end = at[hit[0]] + 1
        loss[i] = np.sum((ls * d)[r0:end])
    prof = np.zeros((10, 3))
    pos = np.arange(len(lt)) - np.repeat(tu[:-1], n)
    for j, v in enumerate((d, lt, np.ones(len(lt)))):
        prof[:, j] = np.bincount(10 * pos // np.repeat(n, n), v, 10)
    return sums, n, cum, total, loss, stop, prof, margin


def _profile_t(lt, lay):
    """The profile's log pi_T column."""
    n = np.diff(lay.turn_row_off)
    tenth = 10 * (np.arange(len(lt)) - np.repeat(lay.turn_row_off[:-1], n)) // np.repeat(n, n)
    return np.array([lt[tenth == j].sum(dtype=np.longdouble) for j in range(10)])


CASES = [(r, s) for r in (1, 31, 255, 256, 257, 5000) for s in ("one", "mixed")]
CASES += [(ONE_WAVE + d, s) for d in (-1, 0, 1) for s in ("turns", "mixed")]
CASES += [(512 * 79 + d, s) for d in (0, 1, 511) for s in ("one", "mixed")]
CASES += [(4096 * 512 + 1, s) for s in ("turns", "mixed")]
CASES += [(1024 * 512 + d, "turns") for d in (0, 1)]  # the longest trajectory that each tile folds by itself


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("rows, shape", CASES)
def test_scan_passes(stride, rows, shape, mode):
    import torch

    rng = np.random.default_rng(rows + 7 * mode)
    lay = _layout(rng, rows, shape)
    lt = -rng.exponential(4.5, rows).astype(np.float32)
    ls = np.minimum(lt + rng.normal(0.0, 0.5, rows), 0.0).astype(np.float32)
    # a threshold that stops about half of the trajectories on the way
    lam = float(np.float32(-4.5 * 1.9 if mode == 0 else -4.5 * max(1.0, 0.6 * rows / max(lay.n_traj, 1)) - 0.37))
    sums, n, cum, total, loss, stop, prof, margin = _reference(ls, lt, lay, mode, lam)
    off = [torch.from_numpy(a).cuda() for a in (lay.traj_row_off, lay.turn_row_off, lay.traj_turn_off)]
    gs, gt = torch.from_numpy(ls).cuda(), torch.from_numpy(lt).cuda()
    ws = torch.empty(stride.stride_score_batch_workspace_size(rows), dtype=torch.uint8, device="cuda")
    ws.fill_(0xA5)  # nothing in it is taken for granted
    for cut in ((), (rows // 3, rows // 3 + 1), (2 * rows // 5,)):
        st, ts, pr = stride.new_state(lay.n_traj), stride.new_turn_stats(lay.n_turns), stride.new_profile()
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        opd = torch.empty(rows, device="cuda")
        edges = sorted({0, rows, *cut})
        for a, b in zip(edges[:-1], edges[1:]):
            stride.stride_scan_logprobs(gs[a:b], gt[a:b], *off, a, b, mode, lam, st, opd=opd[a:b], turn_stats=ts,
                                        dev_status=status, workspace=ws, profile=pr)
        torch.cuda.synchronize()
        assert int(status) == 0
        assert np.array_equal(opd.cpu().numpy(), ls - lt)
        state = stride.state_to_numpy(st)[:lay.n_traj]
        stats = stride.turn_stats_to_numpy(ts)[:lay.n_turns]
        # The terms d and logp_S * d are rounded to fp32 (6e-8 each), their sums are good to 2^-45: 1e-6 of the summed
        # magnitudes bounds the difference.
        mag = [np.add.reduceat(np.abs(v.astype(np.float64)), lay.turn_row_off[:-1]) for v in (lt, ls - lt, ls * (ls - lt))]
        for k, f in enumerate(("sum_t", "sum_d", "sum_l")):
            assert np.all(np.abs(stats[f] - sums[k]) <= 1e-6 * mag[k] + 1e-9), f
        assert np.array_equal(stats["n"], n)
        np.testing.assert_allclose(stats["mean_t"], sums[0] / n, rtol=1e-6)
        np.testing.assert_allclose(stats["cum"], cum, rtol=1e-6)
        full = np.diff(lay.traj_row_off) > 0
        np.testing.assert_allclose(state["cum"][full], total[full], rtol=1e-6)
        np.testing.assert_allclose(pr.cpu().numpy(), prof, rtol=1e-6, atol=1e-6 * np.abs(prof).max())
        # Sums of log pi_T itself: pairs inside a tile (2^-45 of the summed magnitudes) and fp64 across tiles; the token
        # sum fp64 throughout, a tree of some 60 levels at most.
        exact = np.add.reduceat(lt.astype(np.longdouble), lay.turn_row_off[:-1])
        assert np.all(np.abs(stats["sum_t"] - exact) <= 2.0**-44 * mag[0])
        if mode == 1:
            run = np.cumsum(lt.astype(np.longdouble))
            run = run[lay.turn_row_off[1:] - 1] - np.repeat(np.concatenate([[0], run])[lay.traj_row_off[:-1]],
                                                            np.diff(lay.traj_turn_off))
            # (the difference of two running sums: 2^-63 of the whole)
            assert np.all(np.abs(stats["cum"] - run) <= 2.0**-47 * np.abs(run) + 2.0**-60 * np.abs(lt.sum(dtype=np.float64)))
        # (and one fp64 addition per warp and decile)
        assert np.all(np.abs(pr.cpu().numpy()[:, 1] - _profile_t(lt, lay)) <= (2.0**-45 + rows / 32 * 2.0**-53) * np.abs(prof[:, 1]))
        sure = full & (margin > 1e-5)
        assert np.array_equal(np.where(state["stopped"] != 0, state["stop_row"], -1)[sure], stop[sure])
        size = np.add.reduceat(np.abs((ls * (ls - lt)).astype(np.float64)), lay.traj_row_off[:-1][full])
        assert np.all(np.abs(state["loss"] - loss)[sure] <= 1e-6 * size[sure[full]] + 1e-9)
        assert np.array_equal(state["turn_idx"][full], np.diff(lay.traj_turn_off)[full])
        assert np.array_equal(state["rows_seen"][full], np.diff(lay.traj_row_off)[full])


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("rows, V, cuts", [(5000, 16, (1700,)), (ONE_WAVE - 1, 16, ()), (ONE_WAVE, 16, ()), (ONE_WAVE + 1, 16, ()),
                                           (90_000, 16, (ONE_WAVE + 300,)), (1057, 57_344, (500,))])
def test_sums_after_a_scoring_kernel(stride, rows, V, cuts, mode):
    """The persistent kernel's rows, scanned in two passes (one row per thread, or two: V < 57,344) or inside it.  Every
    sum is that of the returned log-probs, products and quotients included: pairs inside a tile, 2^-45 of the summed
    magnitudes, and fp64 for the rest; the retained loss has one fp64 addition per warp more."""
    import torch

    rng = np.random.default_rng(rows + V + mode)
    lay = _layout(rng, rows, "mixed")
    x = torch.from_numpy(rng.standard_normal((rows, V), dtype=np.float32)).cuda()
    y = x + 0.3 * torch.from_numpy(rng.standard_normal((rows, V), dtype=np.float32)).cuda()
    tok = torch.from_numpy(rng.integers(0, V, rows).astype(np.int32)).cuda()
    off = [torch.from_numpy(a).cuda() for a in (lay.traj_row_off, lay.turn_row_off, lay.traj_turn_off)]
    st, ts, pr = stride.new_state(lay.n_traj), stride.new_turn_stats(lay.n_turns), stride.new_profile()
    out = {k: torch.empty(rows, device="cuda") for k in ("logp_s", "logp_t", "opd")}
    ws = torch.full((stride.stride_score_batch_workspace_size(rows),), 0xA5, dtype=torch.uint8, device="cuda")
    lam = torch.from_numpy(rng.uniform(-60.0, -3.0, lay.n_traj).astype(np.float32)).cuda()
    stride.stride_force_batch_kernel("stream")
    try:
        for a, b in zip((0, *cuts), (*cuts, rows)):
            stride.stride_score_batch(x[a:b], y[a:b], tok[a:b], *off, a, b, mode, lam, st,
                                      out={k: v[a:b] for k, v in out.items()}, turn_stats=ts, workspace=ws, profile=pr)
        torch.cuda.synchronize()
    finally:
        stride.stride_force_batch_kernel("auto")
    ls, lt, d = (out[k].cpu().numpy().astype(np.longdouble) for k in ("logp_s", "logp_t", "opd"))
    assert np.array_equal(d.astype(np.float32), (ls - lt).astype(np.float32))
    state = stride.state_to_numpy(st)[:lay.n_traj]
    stats = stride.turn_stats_to_numpy(ts)[:lay.n_turns]
    tu, n = lay.turn_row_off, np.diff(lay.turn_row_off)
    for f, v in (("sum_t", lt), ("sum_d", d), ("sum_l", ls * d)):
        assert np.all(np.abs(stats[f] - np.add.reduceat(v, tu[:-1])) <= 2.0**-44 * np.add.reduceat(np.abs(v), tu[:-1])), f
    for i in range(lay.n_traj):
        k0, k1, r0, r1 = *lay.traj_turn_off[i:i + 2], *lay.traj_row_off[i:i + 2]
        if r0 == r1:
            continue
        if mode == 0:
            cum = np.cumsum(np.add.reduceat(lt, tu[:-1])[k0:k1] / n[k0:k1])
            tests = cum
        else:
            tests = np.cumsum(lt[r0:r1])
            cum = tests[tu[k0 + 1:k1 + 1] - 1 - r0]
        assert np.all(np.abs(stats["cum"][k0:k1] - cum) <= 2.0**-47 * np.abs(cum))
        assert abs(state["cum"][i] - cum[-1]) <= 2.0**-47 * abs(cum[-1])
        hit = np.nonzero(tests < float(lam[i]))[0]
        end = r1 if not len(hit) else (tu[k0 + hit[0] + 1] if mode == 0 else r0 + hit[0] + 1)
        assert state["stopped"][i] == bool(len(hit)) and state["loss_tokens"][i] == end - r0
        term = (ls * d)[r0:end]
        assert abs(state["loss"][i] - term.sum()) <= (2.0**-44 + len(term) / 16 * 2.0**-53) * np.abs(term).sum()
    tenth = 10 * (np.arange(rows) - np.repeat(tu[:-1], n)) // np.repeat(n, n)
    prof = pr.cpu().numpy()
    for j in range(10):
        for k, v in enumerate((d, lt)):
            v = v[tenth == j]
            assert abs(prof[j, k] - v.sum()) <= (2.0**-45 + rows / 32 * 2.0**-53) * np.abs(v).sum()
        assert prof[j, 2] == (tenth == j).sum()
