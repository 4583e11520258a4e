"""The Python module's two routes into the library -- native marshalling for
plain arguments, the general ctypes code for the rest -- give the same
results bit for bit, and refuse the same calls in the same way."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stride():
    import paper_2609_14636_gb300 as s

    return s


class _General:
    """Stands for the native module and leaves every call to the general code."""

    def __getattr__(self, name):
        return lambda *args: None


class _Counting:
    """The native module, counting the calls that it took."""

    def __init__(self, native):
        self.native, self.taken = native, 0

    def __getattr__(self, name):
        fn = getattr(self.native, name)

        def call(*args):
            rc = fn(*args)
            self.taken += rc is not None
            return rc

        return call


ROWS, V, TRAJ, TURNS = 24, 40, 3, 2


def _all_calls(stride, int_=int, float_=float, stream=None):
    """Every entry point once, options given; all outputs as numpy arrays."""
    import torch

    g = torch.Generator(device="cuda").manual_seed(1)
    S = torch.randn((ROWS, V), generator=g, device="cuda")
    T = S + 0.3 * torch.randn((ROWS, V), generator=g, device="cuda")
    tok = torch.randint(0, V, (ROWS,), generator=g, device="cuda", dtype=torch.int32)
    lay = [torch.tensor(a, device="cuda", dtype=d) for a, d in (
        ([0, 8, 16, 24], torch.int64), ([0, 3, 8, 12, 16, 20, 24], torch.int64), ([0, 2, 4, 6], torch.int32))]
    lam = torch.tensor([-3.0, -1e9, -5.0], device="cuda")
    res = []

    def fresh():
        out = {k: torch.empty(ROWS, device="cuda") for k in stride.ROW_OUTPUT_KEYS}
        r = dict(state=stride.new_state(TRAJ), turn_stats=stride.new_turn_stats(TRAJ * TURNS), profile=stride.new_profile(),
                 dev_status=torch.zeros(1, dtype=torch.int32, device="cuda"))
        stride.stride_state_init(r["state"], int_(TRAJ), stream)
        res.extend([*out.values(), *r.values()])
        return out, r

    ws = torch.empty(stride.multi_teacher_workspace_size(ROWS), dtype=torch.uint8, device="cuda")
    for mode, lm in ((0, lam), (1, float_(-9.0))):
        out, r = fresh()
        stride.stride_score_batch(S, T, tok, *lay, int_(0), int_(ROWS), int_(mode), lm, out=out, workspace=ws, stream=stream, **r)
        ts = r["turn_stats"]
        out, r = fresh()
        stride.stride_score_batch_noalloc(S, T, tok, *lay, int_(0), int_(ROWS), int_(mode), lm, out=out, V=int_(V - 3),
                                          stream=stream, **r)
        out, r = fresh()
        dom = torch.tensor([1, 0, 1], dtype=torch.uint8, device="cuda")
        row0 = torch.tensor([0, 0, 8], dtype=torch.int64, device="cuda")
        stride.stride_score_batch_multi_teacher(S, [T[8:16], T.flip(0)], dom, row0, tok, *lay, int_(0), int_(ROWS), int_(mode),
                                                lm, out=out, workspace=ws, stream=stream, **r)
        out, r = fresh()
        stride.stride_scan_logprobs(S[0, :ROWS].neg().abs().neg(), T[0, :ROWS].abs().neg(), *lay, int_(0), int_(ROWS),
                                    int_(mode), lm, opd=out["opd"].zero_(), workspace=ws, stream=stream, **r)
        for k in stride.ROW_OUTPUT_KEYS:
            if k != "opd":
                out[k].zero_()
    B = TRAJ
    end = torch.tensor([0, 1, 0], dtype=torch.uint8, device="cuda")
    for compact in (False, True):
        st = stride.new_state(B)
        out = {"logp_s": torch.zeros(B, device="cuda"), "opd": torch.zeros(B, device="cuda")}
        now = torch.zeros(B, dtype=torch.uint8, device="cuda")
        turn = torch.zeros((B, 40), dtype=torch.uint8, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        kw = dict(out=out, stopped_now=now, turn_out=turn, dev_status=status, V=int_(V), stream=stream)
        if compact:
            idx = torch.tensor([2, 0], dtype=torch.int32, device="cuda")
            stride.stride_score_step_compact(S[:B], T[:B], tok[:B], end, idx, int_(1), lam, st, n_rows=int_(2), **kw)
        else:
            stride.stride_score_step(S[:B], T[:B], tok[:B], end, int_(0), lam, st, **kw)
        res.extend([st, *out.values(), now, turn, status])
    parts = torch.empty((2, ROWS, 6), device="cuda")
    for k in range(2):
        stride.stride_partial_lse(S[:, 20 * k:20 * k + 20], T[:, 20 * k:20 * k + 20], tok, int_(20 * k), parts[k],
                                  V_shard=int_(20), stream=stream)
    o = [torch.empty(ROWS, device="cuda") for _ in range(4)]
    stride.stride_combine_partials(parts, *o, stream=stream)
    mean, n = torch.zeros((5, 4), device="cuda"), torch.ones(5, dtype=torch.int32, device="cuda")
    task = torch.tensor([4, 0, 2], dtype=torch.int32, device="cuda")
    stride.stride_buffer_record(mean, n, task, None, ts, lay[2], stream=stream)
    ok = torch.ones((5, 4), dtype=torch.uint8, device="cuda")
    ks = [torch.empty(5, dtype=torch.int32, device="cuda") for _ in range(2)]
    stride.stride_select_restart(mean, n, ok, float_(-6.0), *ks, stream=stream)
    torch.cuda.synchronize()
    return [x.cpu().numpy().copy() for x in (*res, parts, *o, mean, n, *ks)]


def test_routes_agree(stride, monkeypatch):
    import torch

    native = stride._native()
    counting = _Counting(native)
    monkeypatch.setattr(stride, "_NATIVE", counting)
    plain = _all_calls(stride)
    assert counting.taken > 20
    side = torch.cuda.Stream()
    for kw in (dict(stream=torch.cuda.current_stream()), dict(stream=torch.cuda.current_stream().cuda_stream),
               dict(int_=np.int64, float_=np.float32)):
        assert all(np.array_equal(a, b, equal_nan=a.dtype.kind == "f") for a, b in zip(plain, _all_calls(stride, **kw)))
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):  # the current stream is looked up on each call
        assert all(np.array_equal(a, b, equal_nan=a.dtype.kind == "f") for a, b in zip(plain, _all_calls(stride)))
    torch.cuda.current_stream().wait_stream(side)
    monkeypatch.setattr(stride, "_NATIVE", _General())
    assert all(np.array_equal(a, b, equal_nan=a.dtype.kind == "f") for a, b in zip(plain, _all_calls(stride)))


def test_routes_refuse_alike(stride, monkeypatch):
    import torch

    f = lambda *s, dt=torch.float32: torch.zeros(s, dtype=dt, device="cuda")  # noqa: E731
    S, tok, end, st = f(4, 8), f(4, dt=torch.int32), f(4, dt=torch.uint8), stride.new_state(4)
    good = dict(S=S, T=S, tokens=tok, turn_end=end, stop_mode=0, lam=-1.0, state=st)
    bad = [dict(S=S.cpu()), dict(T=f(4, 9)), dict(S=S.half(), T=S.half()), dict(T=f(8, 4).t()), dict(S=f(4), T=f(4)),
           dict(tokens=tok.long()), dict(tokens=tok[:3]), dict(tokens=f(4, 2, dt=torch.int32)[:, 0]), dict(tokens=None),
           dict(state=st[:3]), dict(state=None), dict(lam=f(3)), dict(lam="x"), dict(lam=None), dict(stop_mode=7),
           dict(lam=float("nan")), dict(out={"nope": f(4)}), dict(out={"opd": f(3)}), dict(out={"opd": f(4).double()}),
           dict(stopped_now=f(3, dt=torch.uint8)), dict(turn_out=f(4, 39, dt=torch.uint8)), dict(dev_status=f(1)),
           dict(V=9), dict(V=0), dict(V="x"), dict(stream="x")]
    native = stride._native()
    for change in bad:
        got = []
        for route in (native, _General()):
            monkeypatch.setattr(stride, "_NATIVE", route)
            with pytest.raises(Exception) as e:
                stride.stride_score_step(**{**good, **change})
            got.append((type(e.value), str(e.value)))
        assert got[0] == got[1], change
