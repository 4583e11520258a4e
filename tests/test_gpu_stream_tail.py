"""The streaming loop's end: rows whose share per thread is any number of
16-byte vectors around its batches of four, through the three kernels that
stream with it (decode step, small windows, shard pass), decode steps of row counts
at the edges of the launch-shape rule, and shard passes on both sides of the
persistent kernel's.  Against the log-softmax in 64 bits."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stride():
    import paper_2609_14636_gb300 as s

    return s


def _logits(rows, V, f32, seed):
    import torch

    g = torch.Generator(device="cuda").manual_seed(seed)
    S = 3.0 * torch.randn((rows, V), generator=g, device="cuda")
    T = S + 0.5 * torch.randn((rows, V), generator=g, device="cuda")
    if not f32:
        S, T = S.bfloat16(), T.bfloat16()
    tok = torch.randint(0, V, (rows,), generator=g, device="cuda", dtype=torch.int32)
    S[:, V // 2] = -float("inf")  # masked entries, among them the last
    S[:, V - 1] = -float("inf")
    tok[tok == V - 1] = 0
    tok[tok == V // 2] = 1
    return S, T, tok


def _exact(x, tok):
    x = x.double()
    return (x.gather(1, tok.long()[:, None])[:, 0] - x.logsumexp(1)).cpu().numpy()


def _close(got, x, tok):
    # one fp32 exp-sum of up to 152,000 terms and the rounding of numbers near 20: a few 1e-6
    np.testing.assert_allclose(got.cpu().numpy(), _exact(x, tok), rtol=0, atol=1e-5)


def _step(stride, S, T, tok, compact):
    import torch

    n = S.shape[0]
    out = {k: torch.full((n,), float("nan"), device="cuda") for k in ("logp_s", "logp_t")}
    end = torch.zeros(n, dtype=torch.uint8, device="cuda")
    if compact:
        idx = torch.arange(n - 1, -1, -1, dtype=torch.int32, device="cuda")
        stride.stride_score_step_compact(S, T, tok, end, idx, 0, -1e9, stride.new_state(n), out=out)
    else:
        stride.stride_score_step(S, T, tok, end, 0, -1e9, stride.new_state(n), out=out)
    _close(out["logp_s"], S, tok)
    _close(out["logp_t"], T, tok)


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("batches", [0, 1, 2])
@pytest.mark.parametrize("left", [0, 1, 2, 3])
def test_rows_around_a_batch(stride, batches, left, f32):
    import torch

    per_vec = 4 if f32 else 8
    for d in (-1, 0, 1):
        for tail in (0, 3):
            vecs = 128 * (4 * batches + left) + d
            if vecs < 1:
                continue
            V = vecs * per_vec + tail
            S, T, tok = _logits(5, V, f32, 10 * vecs + tail)
            stride.stride_force_step_shape(128, 1)
            try:
                _step(stride, S, T, tok, True)
            finally:
                stride.stride_force_step_shape(0, 0)
            parts = torch.empty((1, 5, 6), device="cuda")
            stride.stride_partial_lse(S, T, tok, 0, parts[0])
            ls, lt = torch.empty(5, device="cuda"), torch.empty(5, device="cuda")
            stride.stride_combine_partials(parts, ls, lt)
            _close(ls, S, tok)
            _close(lt, T, tok)
            off = [torch.tensor(a, dtype=t, device="cuda") for a, t in (([0, 5], torch.int64), ([0, 5], torch.int64),
                                                                        ([0, 1], torch.int32))]
            ws = torch.empty(stride.stride_score_batch_workspace_size(5), dtype=torch.uint8, device="cuda")
            out = {"logp_s": torch.empty(5, device="cuda"), "logp_t": torch.empty(5, device="cuda")}
            stride.stride_force_batch_kernel("split1")
            try:
                stride.stride_score_batch(S, T, tok, *off, 0, 5, 0, -1e9, stride.new_state(1), out=out, workspace=ws)
            finally:
                stride.stride_force_batch_kernel("auto")
            _close(out["logp_s"], S, tok)
            _close(out["logp_t"], T, tok)


@pytest.mark.parametrize("compact", [False, True])
@pytest.mark.parametrize("V", [33, 4099, 32_000])
def test_every_launch_shape(stride, compact, V):
    rows = (1, 2, 13, 14, 15, 17, 18, 21, 22, 23, 28, 30, 31, 36, 41, 44, 45, 52, 53, 63, 64, 72, 73, 84, 99, 108, 121, 136, 137,
            152, 153, 182, 217, 218, 273, 274, 300, 305, 400, 1216, 1300)
    S, T, tok = _logits(max(rows), V, False, V)
    for n in rows:
        _step(stride, S[:n], T[:n], tok[:n], compact)


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("rows", [1, 7, 456, 457, 700, 760, 1065])
@pytest.mark.parametrize("kb", [11, 32, 128])
def test_shard_pass_routes(stride, rows, kb, f32):
    """Shard rows around the sizes from which the persistent kernel takes the pass, and row counts on both sides of the
    other's two shapes (five loads from 760 rows on, not at 1,065), aligned and not, the second shard with and without
    the row's token."""
    import torch

    W = kb * 1024 // (4 if f32 else 2)
    for w0, w1 in ((W, W), (W + 3, W - 1)):
        S, T, tok = _logits(rows, w0 + w1, f32, rows + w1)
        parts = torch.full((2, rows, 6), -7.0, device="cuda")
        for k, (a, b) in enumerate(((0, w0), (w0, w0 + w1))):
            stride.stride_partial_lse(S[:, a:b], T[:, a:b], tok, a, parts[k], V_shard=b - a)
        mine = [(tok < w0).cpu().numpy(), (tok >= w0).cpu().numpy()]
        for k in range(2):
            assert np.array_equal(~np.isnan(parts[k, :, 4].cpu().numpy()), mine[k])
            assert np.array_equal(~np.isnan(parts[k, :, 5].cpu().numpy()), mine[k])
        o = [torch.empty(rows, device="cuda") for _ in range(2)]
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        stride.stride_combine_partials(parts, *o, dev_status=status)
        assert int(status) == 0
        _close(o[0], S, tok)
        _close(o[1], T, tok)
