"""GPU parity of the persistent kernel's scan at the sizes where it can go
wrong: windows that end inside, at and just past a tile, turns of one row (a
tile full of turns), runs of more empty trajectories than a tile stages, and
very short rows.  From 57,344 logits on the scan runs inside the kernel, in
32-row tiles; below that it follows in two passes.

And rows at every alignment through the same kernel: S and T starting on
different element offsets from a 16-byte boundary, strides that move the
offset from row to row, vocabularies of less than a vector, around one and
two vectors, and around one full stage (16,384 bf16 or 8,192 fp32 logits)."""
from __future__ import annotations

import numpy as np
import pytest

import synth
from gpu_helpers import compare_rows, compare_scan, oracle_batch, run_batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stride():
    import paper_2609_14636_gb300 as s

    return s


def _layout(rng, rows):
    """Turns of one row (half of them) or 2-70 rows, 1-4 per trajectory,
    and now and then 40 trajectories without turns in a row."""
    lens, left = [], rows
    while left > 0:
        turns = []
        for _ in range(int(rng.integers(1, 5))):
            n = min(left, 1 if rng.random() < 0.5 else int(rng.integers(2, 71)))
            if n:
                turns.append(n)
            left -= n
        lens.append(turns)
        if rng.random() < 0.1:
            lens.extend([[]] * 40)
    return synth.layout_from_turn_lengths(lens)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("rows, V", [(1, 64), (31, 64), (32, 64), (33, 64), (95, 264), (1024, 264), (1057, 64),
                                     (20_000, 16), (1, 57_344), (31, 57_344), (33, 57_343), (33, 57_344),
                                     (95, 57_344), (1057, 57_344)])
def test_warp_tiles(stride, rows, V, mode):
    rng = np.random.default_rng(rows * 2 + mode)
    lay = _layout(rng, rows)
    # Unit logits: compare_scan bounds a running sum's error by 1e-5 of the sum, and a single log-prob's rounding is
    # about 2 ulp of its log-sum-exp (<= 5e-7 below 8), so |log-prob| has to stay above 0.05.  With N(0, 1) logits and
    # 16 entries it does; N(0, 3^2) rows have entries of probability 0.999 (log-prob -1e-3: 5e-4 relative).
    S = synth.bf16_bits_from_f32(rng.standard_normal((rows, V), dtype=np.float32))
    T = synth.bf16_bits_from_f32(synth.f32_from_bf16_bits(S) + rng.standard_normal((rows, V), dtype=np.float32) * np.float32(0.3))
    tok = rng.integers(0, V, rows).astype(np.int32)
    lam = rng.uniform(-60.0, -3.0, lay.n_traj).astype(np.float32)
    o = oracle_batch(S, T, tok, lay, mode, lam)
    assert o["logp_t"].max() < -0.05
    stride.stride_force_batch_kernel("stream")
    try:
        for windows in (None, [w for w in ((0, rows // 3), (rows // 3, rows)) if w[0] < w[1]]):
            g = run_batch(stride, S, T, tok, lay, mode, lam, windows=windows)
            assert g["status"] == 0
            compare_rows(g, o)
            compare_scan(g, o, lay, mode, lam)
    finally:
        stride.stride_force_batch_kernel("auto")


@pytest.mark.parametrize("off_s, off_t", [(0, 0), (1, 1), (3, 0), (0, 7), (5, 2)])
@pytest.mark.parametrize("f32", [False, True])
def test_unaligned_rows(stride, f32, off_s, off_t):
    import torch

    stage = 8192 if f32 else 16_384
    rng = np.random.default_rng(100 + 10 * off_s + off_t + f32)
    for V in (1, 3, 7, 8, 9, 15, 16, 17, 31, 33, 1001, stage - 1, stage, stage + 1, stage + 7, stage + 8, 2 * stage + 9):
        rows = 70 if V < 2000 else 9
        lay = synth.layout_from_turn_lengths([[3, 2], [rows - 5]])
        # (unit logits, as above; V = 1 has log-prob 0, an exact 0 on both sides)
        S32 = rng.standard_normal((rows, V), dtype=np.float32)
        T32 = S32 + rng.standard_normal((rows, V), dtype=np.float32) * np.float32(0.3)
        S, T = (S32, T32) if f32 else (synth.bf16_bits_from_f32(S32), synth.bf16_bits_from_f32(T32))
        tok = (S32 * -1.0).argmax(1).astype(np.int32)  # an unlikely token: log-probs well away from 0
        o = oracle_batch(S, T, tok, lay, 0, np.float32(-1e6))
        for ld in (V, V + 3):
            dev = []
            for a, off in ((S, off_s), (T, off_t)):
                flat = np.full(16 + rows * ld, np.nan, np.float32) if f32 else np.full(16 + rows * ld, 0x7FC0, np.uint16)
                np.lib.stride_tricks.as_strided(flat[off:], (rows, V), (ld * flat.itemsize, flat.itemsize))[:] = a
                t = torch.from_numpy(flat if f32 else flat.view(np.int16)).cuda()
                dev.append((t if f32 else t.view(torch.bfloat16)).as_strided((rows, V), (ld, 1), off))
            stride.stride_force_batch_kernel("stream")
            try:
                g = run_batch(stride, *dev, tok, lay, 0, np.float32(-1e6), V=V)
            finally:
                stride.stride_force_batch_kernel("auto")
            assert g["status"] == 0, V
            compare_rows(g, o)
            compare_scan(g, o, lay, 0, np.float32(-1e6))
