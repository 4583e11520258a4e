"""The measured cases of the scoring library: what a training loop asks of it, through the Python entry points.

Six kinds of pass, each with its own outputs:

* ``batch``   ragged trajectories in one or several row windows with carried state (stride_score_batch, or the
              no-allocation entry point), optionally followed by the prefix-buffer record and the restart choice;
* ``domains`` the same with one teacher buffer per domain (stride_score_batch_multi_teacher);
* ``shards``  vocabulary-sharded logits: one partial pass per shard, the merge, the scan on the log-probs;
* ``scan``    the scan on log-probs that the caller already has, then record and restart choice over a large buffer;
* ``steps``   decode steps of all rollouts, stopped ones masked (stride_score_step);
* ``live``    decode steps over the live rollouts' rows only (stride_score_step_compact), as plain calls or as one
              CUDA graph.

Logits follow the repository's workload generators: student N(0, sigma^2), a teacher that tracks it (noise 0.3) up to a
first-error turn of each trajectory and drifts after it (noise 2.5), tokens sampled from the student by Gumbel-max.
"""
import math

import numpy as np
import torch

import paper_2609_14636_gb300 as stride

V0 = 151_936  # the vocabulary of the repository's bf16 workloads
ROW_KEYS = ("logp_s", "logp_t", "opd", "lse_s", "lse_t", "x_s", "x_t")
GEN_ROWS = 512  # rows generated at a time
MAX_BYTES = 2 * 20_000 * V0 * 2  # logit bytes of the largest listed case: no drawn case reads more


def listed():
    return [
        # The end of a decode sweep: a handful of live rollouts, one call per generated token.  The smallest call;
        # launch and host time are all of it.
        dict(name="live_8_one_step", kind="live", rows=8, rollouts=256, steps=1, ring=1, graph=False, V=V0, ld=V0,
             dtype="bf16", mode=0, sigma=3.0),
        # A decode turn of 256 rollouts as plain calls, thresholds that stop some of them on the way (masked).
        dict(name="steps_256_masked", kind="steps", rows=256, rollouts=256, steps=16, ring=4, graph=False, V=V0, ld=V0,
             dtype="bf16", mode=1, sigma=3.0),
        # A rollout engine that captured its decode loop: an odd number of live rollouts, steps replayed as a graph.
        dict(name="live_61_graph", kind="live", rows=61, rollouts=256, steps=32, ring=4, graph=True, V=V0, ld=V0,
             dtype="bf16", mode=0, sigma=3.0),
        # The tiny reference: one 512-token trajectory, fp32 logits, token-sum rule.
        dict(name="tiny_512_f32", kind="batch", entry="batch", rows=512, traj=1, turns=4, window=0, V=32_000, ld=32_000,
             dtype="f32", mode=1, sigma=3.0, outputs=3, profile=False, tasks=0),
        # One window of a host-fed stream (the end-to-end path scores 1,024 rows per copied window).
        dict(name="window_1024", kind="batch", entry="batch", rows=1024, traj=1, turns=4, window=0, V=V0, ld=V0,
             dtype="bf16", mode=0, sigma=4.0, outputs=3, profile=False, tasks=0),
        # A batch of a few short trajectories: more rows than one wave, far fewer than a full batch.
        dict(name="batch_3001", kind="batch", entry="noalloc", rows=3001, traj=6, turns=4, window=0, V=V0, ld=V0,
             dtype="bf16", mode=0, sigma=4.0, outputs=7, profile=True, tasks=0),
        # Long agentic trajectories streamed in 16,384-row windows with carried state (the second window is what is
        # left), recorded in the prefix buffer, then the restart choice: one pass of the training loop.  The largest.
        dict(name="agentic_20000_windows", kind="batch", entry="batch", rows=20_000, traj=5, turns=12, window=16_384,
             V=V0, ld=V0, dtype="bf16", mode=0, sigma=4.0, outputs=3, profile=False, tasks=64),
        # A vocabulary that is not a multiple of a vector, rows packed without padding: no row start is aligned.
        dict(name="packed_odd_6000", kind="batch", entry="batch", rows=6000, traj=8, turns=4, window=0, V=151_933,
             ld=151_933, dtype="bf16", mode=0, sigma=4.0, outputs=3, profile=False, tasks=0),
        # A 32,000-entry vocabulary: many short rows, single-turn math rollouts (token-sum rule).
        dict(name="vocab_32000_bf16", kind="batch", entry="batch", rows=30_011, traj=64, turns=1, window=0, V=32_000,
             ld=32_000, dtype="bf16", mode=1, sigma=3.0, outputs=3, profile=False, tasks=0),
        # Cross-domain scoring, each trajectory against the teacher of its own domain, rows in per-domain buffers.
        dict(name="domains_8192", kind="domains", rows=8192, traj=12, turns=6, V=V0, ld=V0, dtype="bf16", mode=0,
             sigma=4.0, outputs=3, profile=False, domains=2),
        # Tensor-parallel logits: four column shards, merge, scan.
        dict(name="shards_4x6000", kind="shards", rows=6000, traj=8, turns=6, V=V0, ld=V0 // 4, dtype="bf16", mode=0,
             sigma=4.0, shards=4, profile=False),
        # Log-probs that the trainer already has, for a whole batch (64 trajectories of 8 turns), then the record and
        # the restart choice over a 10,000-record prefix buffer.
        dict(name="scan_148909", kind="scan", rows=148_909, traj=64, turns=8, mode=0, profile=True, tasks=10_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["batch", "batch", "batch", "domains", "shards", "scan", "steps", "live", "live"])
    mode = rng.randint(0, 1)
    if kind == "scan":
        traj = _log_int(rng, 1, 128)
        turns = rng.randint(1, 12) if mode == 0 else 1
        return dict(kind=kind, rows=max(_log_int(rng, 300, 148_909), 4 * traj * turns), traj=traj, turns=turns, mode=mode,
                    profile=rng.random() < 0.5, tasks=max(traj, _log_int(rng, 16, 10_000)))
    dtype = "f32" if rng.random() < 0.25 else "bf16"
    elt = 4 if dtype == "f32" else 2
    V = rng.choice([V0, V0, 32_000, _log_int(rng, 32_000, 152_064)])
    if rng.random() < 0.3:
        V -= rng.randint(1, 7)  # not a whole number of vectors ...
    ld = V if rng.random() < 0.6 else (V + 63) // 64 * 64  # ... packed, or padded to aligned rows
    sigma = rng.choice([3.0, 4.0])
    if kind in ("steps", "live"):
        rollouts = rng.choice([64, 128, 256])
        rows = rollouts if kind == "steps" else min(rollouts, _log_int(rng, 1, 256))
        return dict(kind=kind, rows=rows, rollouts=rollouts, steps=rng.randint(2, 32), ring=4, graph=rng.random() < 0.5,
                    V=V, ld=ld, dtype=dtype, mode=mode, sigma=sigma)
    most = MAX_BYTES // (2 * ld * elt)
    traj = _log_int(rng, 1, 24)
    turns = rng.randint(1, 10) if mode == 0 else 1
    rows = min(max(_log_int(rng, 64, 40_000), 4 * traj * turns), most)
    c = dict(kind=kind, rows=rows, traj=traj, turns=turns, V=V, ld=ld, dtype=dtype, mode=mode, sigma=sigma,
             profile=rng.random() < 0.3)
    if kind == "shards":
        n = rng.choice([2, 4, 8])
        c.update(shards=n, V=V // n * n, ld=V // n if rng.random() < 0.5 else (V // n + 63) // 64 * 64,
                 rows=min(rows, 10_000))
        return c
    c.update(outputs=rng.choice([0, 3, 7]))
    if kind == "domains":
        c.update(domains=rng.randint(1, 3))
        return c
    c.update(entry=rng.choice(["batch", "batch", "noalloc"]), window=rng.choice([0, 0, 1024, 4096, 16_384]),
             tasks=rng.choice([0, 64]))
    return c


# ---------------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------------
def _layout(case, seed):
    """traj_row_off, turn_row_off, traj_turn_off: case-given counts, turn lengths within a factor of eight."""
    n = case["traj"] * case["turns"]
    w = np.random.default_rng([seed, 7]).uniform(64.0, 512.0, n)
    cut = np.floor(np.cumsum(w) / w.sum() * (case["rows"] - n)).astype(np.int64)
    cut[-1] = case["rows"] - n
    turn = np.concatenate([[0], cut + np.arange(1, n + 1)]).astype(np.int64)
    first = np.arange(0, n + 1, case["turns"]).astype(np.int32)
    return turn[first].copy(), turn, first


def _sigma_t(case, seed, traj, turn, first):
    """Teacher noise of each row: 0.3 before the trajectory's first-error turn, 2.5 from it on."""
    err = np.random.default_rng([seed, 8]).integers(0, case["turns"] + 1, case["traj"])
    sig = np.full(case["rows"], 0.3, np.float32)
    for i, e in enumerate(err):
        sig[turn[first[i] + min(e, case["turns"])]:traj[i + 1]] = 2.5
    return torch.from_numpy(sig).cuda()


def _logits(rows, V, ld, dtype, sigma, sig_t, g):
    """S, T [rows, ld] and the sampled tokens [rows]."""
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    S, T = (torch.empty((rows, ld), dtype=dt, device="cuda") for _ in range(2))
    tok = torch.empty(rows, dtype=torch.int32, device="cuda")
    if ld > V:
        S[:, V:] = 0
        T[:, V:] = 0
    for a in range(0, rows, GEN_ROWS):
        b = min(rows, a + GEN_ROWS)
        x = torch.randn((b - a, V), generator=g, device="cuda").mul_(sigma).to(dt)
        S[a:b, :V] = x
        x = x.float()
        noise = torch.randn((b - a, V), generator=g, device="cuda").mul_(sig_t[a:b, None])
        T[a:b, :V] = noise.add_(x)
        x.sub_(noise.exponential_(generator=g).log_())  # Gumbel-max: -log of an exponential is Gumbel
        tok[a:b] = x.argmax(1)
        del x, noise
    return S, T, tok


def _lam(case):
    """Thresholds that stop some of the trajectories (per token about -4.5, as the generators score)."""
    if case["mode"] == stride.TURN_MEAN:
        return -4.8 * max(1.0, 0.7 * case["turns"])
    return -4.8 * 0.7 * case["rows"] / case["traj"]


def _state_views(st, n):
    f, i8, i4 = st[:n].view(torch.float64), st[:n].view(torch.int64), st[:n].view(torch.int32)
    return {"cum": f[:, 0], "open_sums": f[:, 1:4], "loss": f[:, 4], "counts": i8[:, 5:8], "turns": i4[:, 16:20]}


def _stats_views(ts, n):
    f, f4, i4 = ts[:n].view(torch.float64), ts[:n].view(torch.float32), ts[:n].view(torch.int32)
    return {"sum_t": f[:, 0], "sum_d": f[:, 1], "sum_l": f[:, 2], "cum": f[:, 3], "mean_t": f4[:, 8], "n": i4[:, 9]}


class _State:
    pass


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + 17)


def _logprob_inputs(case, seed):
    g = _gen(seed)
    lt = -torch.empty(case["rows"], device="cuda").exponential_(generator=g).mul_(4.5)
    ls = lt + torch.randn(case["rows"], generator=g, device="cuda").mul_(0.5)
    return ls.clamp_(max=0.0), lt


def _buffer_inputs(case, seed):
    """A prefix buffer with earlier records of up to 12 turns (or the case's), and a correctness mask."""
    g = _gen(seed + 500)
    T_max = max(12, case["turns"])
    mean = torch.randn((case["tasks"], T_max), generator=g, device="cuda").mul_(1.5).sub_(4.5)
    n = torch.randint(1, T_max + 1, (case["tasks"],), generator=g, device="cuda", dtype=torch.int32)
    task = torch.randperm(case["tasks"], generator=g, device="cuda")[:case["traj"]].to(torch.int32)
    ok = (torch.rand((case["tasks"], T_max), generator=g, device="cuda") < 0.9).to(torch.uint8)
    return mean, n, task, ok


def _step_inputs(case, seed):
    g = _gen(seed)
    rng = np.random.default_rng([seed, 9])
    rows, n = case["rows"], case["rollouts"]
    sig = torch.full((case["ring"] * rows,), 0.5, device="cuda")
    S, T, tok = _logits(case["ring"] * rows, case["V"], case["ld"], case["dtype"], case["sigma"], sig, g)
    end = (rng.random((case["steps"], rows)) < 0.2).astype(np.uint8)
    idx = rng.permutation(n)[:rows].astype(np.int32)
    if case["kind"] == "live":
        lam = np.full(n, -np.inf, np.float32)  # the caller packs live rollouts; none of them stops in this stretch
    elif case["mode"] == stride.TURN_MEAN:
        lam = rng.uniform(-40.0, -5.0, n).astype(np.float32)
    else:
        lam = rng.uniform(-400.0, -10.0, n).astype(np.float32)
    return S, T, tok, torch.from_numpy(end).cuda(), torch.from_numpy(idx).cuda(), torch.from_numpy(lam).cuda()


def _step_calls(s):
    case = s.case
    if case["steps"] > 1:
        stride.stride_state_init(s.state, case["rollouts"])
    for k in range(case["steps"]):
        a = s.slabs[k % case["ring"]]
        if case["kind"] == "live":
            stride.stride_score_step_compact(a[0], a[1], a[2], s.end[k], s.idx, case["mode"], s.lam, s.state,
                                             out=s.out[k], stopped_now=s.now[k], turn_out=s.turn[k], V=case["V"])
        else:
            stride.stride_score_step(a[0], a[1], a[2], s.end[k], case["mode"], s.lam, s.state, out=s.out[k],
                                     stopped_now=s.now[k], turn_out=s.turn[k], V=case["V"])


def prepare(case, seed):
    s = _State()
    s.case, kind = case, case["kind"]
    if kind in ("steps", "live"):
        rows, steps = case["rows"], case["steps"]
        S, T, tok, end, s.idx, s.lam = _step_inputs(case, seed)
        s.slabs = [(S[a:a + rows], T[a:a + rows], tok[a:a + rows]) for a in range(0, case["ring"] * rows, rows)]
        s.end = [end[k] for k in range(steps)]
        s.state = stride.new_state(case["rollouts"])
        row = {k: torch.empty((steps, rows), device="cuda") for k in ROW_KEYS[:3]}
        s.out = [{k: v[i] for k, v in row.items()} for i in range(steps)]
        now = torch.empty((steps, rows), dtype=torch.uint8, device="cuda")
        turn = torch.zeros((steps, rows, 40), dtype=torch.uint8, device="cuda")
        s.now, s.turn = list(now), list(turn)
        s.result = {"rows": row, "stopped_now": now, "turns": _stats_views(turn.view(steps * rows, 40), steps * rows),
                    "state": _state_views(s.state, case["rollouts"])}
        s.graph = None
        if case["graph"]:
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                _step_calls(s)  # first use outside the capture, as a program does
            torch.cuda.current_stream().wait_stream(side)
            s.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s.graph):
                _step_calls(s)
            stride.stride_state_init(s.state, case["rollouts"])
        return s
    traj, turn, first = _layout(case, seed)
    s.off = [torch.from_numpy(a).cuda() for a in (traj, turn, first)]
    n_traj, n_turns, rows = case["traj"], case["traj"] * case["turns"], case["rows"]
    s.state = stride.new_state(n_traj)
    s.stats = stride.new_turn_stats(n_turns)
    s.status = torch.zeros(1, dtype=torch.int32, device="cuda")
    s.profile = stride.new_profile() if case["profile"] else None
    s.lam = _lam(case)
    s.result = {"state": _state_views(s.state, n_traj), "stats": _stats_views(s.stats, n_turns), "status": s.status}
    if s.profile is not None:
        s.result["profile"] = s.profile
    if kind == "scan":
        s.ls, s.lt = _logprob_inputs(case, seed)
        s.opd = torch.empty(rows, device="cuda")
        s.result["rows"] = {"opd": s.opd}
    else:
        sig = _sigma_t(case, seed, traj, turn, first)
        if kind == "shards":
            n, w = case["shards"], case["V"] // case["shards"]
            S, T, s.tok = _logits(rows, case["V"], case["V"], case["dtype"], case["sigma"], sig, _gen(seed))
            s.parts_S, s.parts_T = [], []
            for k in range(n):
                for src, dst in ((S, s.parts_S), (T, s.parts_T)):
                    x = torch.zeros((rows, case["ld"]), dtype=S.dtype, device="cuda")
                    x[:, :w] = src[:, k * w:(k + 1) * w]
                    dst.append(x)
            del S, T
            s.partials = torch.empty((n, rows, 6), device="cuda")
            s.ls, s.lt, s.opd, s.zs, s.zt = (torch.empty(rows, device="cuda") for _ in range(5))
            s.result["rows"] = {"logp_s": s.ls, "logp_t": s.lt, "opd": s.opd, "lse_s": s.zs, "lse_t": s.zt}
        else:
            s.S, s.T, s.tok = _logits(rows, case["V"], case["ld"], case["dtype"], case["sigma"], sig, _gen(seed))
            keys = ROW_KEYS[:case["outputs"]]
            s.out = {k: torch.empty(rows, device="cuda") for k in keys}
            s.result["rows"] = dict(s.out)
            if kind == "domains":
                dom = np.random.default_rng([seed, 10]).integers(0, case["domains"], n_traj)
                at, row0, parts = [0] * case["domains"], np.zeros(n_traj, np.int64), [[] for _ in range(case["domains"])]
                for i, d in enumerate(dom):
                    row0[i] = at[d]
                    at[d] += int(traj[i + 1] - traj[i])
                    parts[d].append(s.T[int(traj[i]):int(traj[i + 1])])
                s.T_dom = [torch.cat(p) if p else torch.zeros((1, case["ld"]), dtype=s.T.dtype, device="cuda") for p in parts]
                s.T = None
                s.dom = torch.from_numpy(dom.astype(np.uint8)).cuda()
                s.row0 = torch.from_numpy(row0).cuda()
    size = case.get("window", 0) or rows
    s.windows = [(a, min(rows, a + size)) for a in range(0, rows, size)]
    need = (stride.multi_teacher_workspace_size if kind == "domains" else stride.stride_score_batch_workspace_size)(
        min(size, rows))
    s.ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    if case.get("tasks"):
        s.mean, s.n_rec, s.task, s.ok = _buffer_inputs(case, seed)
        s.k_star, s.k_max = (torch.empty(case["tasks"], dtype=torch.int32, device="cuda") for _ in range(2))
        s.result["buffer"] = {"mean": s.mean, "n": s.n_rec, "k_star": s.k_star, "k_max": s.k_max}
    if case.get("entry") == "noalloc":
        s.cuts = [(s.S[a:b], s.T[a:b], s.tok[a:b], {k: v[a:b] for k, v in s.out.items()}, a, b) for a, b in s.windows]
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind in ("steps", "live"):
        if s.graph is not None:
            s.graph.replay()
        else:
            _step_calls(s)
        return s.result
    rows = case["rows"]
    stride.stride_state_init(s.state, case["traj"])
    if s.profile is not None:
        s.profile.zero_()
    if kind == "batch" and case["entry"] == "noalloc":
        for S, T, tok, out, a, b in s.cuts:
            stride.stride_score_batch_noalloc(S, T, tok, *s.off, a, b, case["mode"], s.lam, s.state, out=out,
                                              turn_stats=s.stats, dev_status=s.status, V=case["V"], profile=s.profile)
    elif kind == "batch":
        for a, b in s.windows:
            stride.stride_score_batch(s.S[a:b], s.T[a:b], s.tok[a:b], *s.off, a, b, case["mode"], s.lam, s.state,
                                      out={k: v[a:b] for k, v in s.out.items()}, turn_stats=s.stats,
                                      dev_status=s.status, workspace=s.ws, V=case["V"], profile=s.profile)
    elif kind == "domains":
        stride.stride_score_batch_multi_teacher(s.S, s.T_dom, s.dom, s.row0, s.tok, *s.off, 0, rows, case["mode"], s.lam,
                                                s.state, out=s.out, turn_stats=s.stats, dev_status=s.status,
                                                workspace=s.ws, V=case["V"], profile=s.profile)
    else:
        if kind == "shards":
            w = case["V"] // case["shards"]
            for k, (S, T) in enumerate(zip(s.parts_S, s.parts_T)):
                stride.stride_partial_lse(S, T, s.tok, k * w, s.partials[k], dev_status=s.status, V_shard=w)
            stride.stride_combine_partials(s.partials, s.ls, s.lt, s.zs, s.zt, dev_status=s.status)
        stride.stride_scan_logprobs(s.ls, s.lt, *s.off, 0, rows, case["mode"], s.lam, s.state, opd=s.opd,
                                    turn_stats=s.stats, dev_status=s.status, workspace=s.ws, profile=s.profile)
    if case.get("tasks"):
        stride.stride_buffer_record(s.mean, s.n_rec, s.task, None, s.stats, s.off[2], dev_status=s.status)
        stride.stride_select_restart(s.mean, s.n_rec, s.ok, -4.5, s.k_star, s.k_max)
    return s.result


# ---------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without, how exact it is, and the same in 64 bits
# ---------------------------------------------------------------------------------------------------------------------
def work(case):
    kind, rows = case["kind"], case["rows"]
    if kind == "scan":
        n = case["traj"] * case["turns"]
        b = rows * 12 + n * 48 + case["traj"] * 176 + case["tasks"] * max(12, case["turns"]) * 5 + case["tasks"] * 12
        return {"bytes": b, "flops": 12 * rows}
    elt = 4 if case["dtype"] == "f32" else 2
    if kind in ("steps", "live"):
        per_row = 2 * case["V"] * elt + 4 + 1 + 12 + 1 + 40 + 160
        if kind == "steps":
            # a stopped rollout's logits need not be read: about how many are read over the steps
            live = 0.85 if case["mode"] == stride.TOKEN_SUM else 0.95
        else:
            live = 1.0
        return {"bytes": live * per_row * rows * case["steps"], "flops": live * 8 * case["V"] * rows * case["steps"]}
    out = {"shards": 5}.get(kind, case.get("outputs", 0))
    b = rows * (2 * case["V"] * elt + 4 + 4 * out) + case["traj"] * (176 + case["turns"] * 48)
    return {"bytes": b, "flops": 8 * case["V"] * rows}


def tolerance(case):
    # Log-probs are differences of 32-bit numbers near 20 (rounding 1e-6), sums are 64-bit.  Measured against exact():
    # at most 1.6e-6 (the OPD signal and its sums, which cancel), 1e-7 and less everywhere else; whole values equal.
    return {"rel": 7e-6, "max": 1e-4}


def _row_exact(S, T, tok, V):
    """Log-probs and log-sum-exps of rows in 64 bits."""
    got = [torch.empty(S.shape[0], dtype=torch.float64, device="cuda") for _ in range(4)]
    for a in range(0, S.shape[0], 256):
        b = min(S.shape[0], a + 256)
        y = tok[a:b].long()[:, None]
        for x, x_y, z in ((S, got[0], got[2]), (T, got[1], got[3])):
            v = x[a:b, :V].double()
            z[a:b] = torch.logsumexp(v, 1)
            x_y[a:b] = v.gather(1, y)[:, 0]
    xs, xt, zs, zt = (v.cpu().numpy() for v in got)
    return {"logp_s": xs - zs, "logp_t": xt - zt, "opd": (xs - zs) - (xt - zt), "lse_s": zs, "lse_t": zt, "x_s": xs, "x_t": xt}


def _scan_exact(case, seed, ls, lt):
    traj, turn, first = _layout(case, seed)
    d, mode, lam = ls - lt, case["mode"], float(np.float32(_lam(case)))
    n = turn[1:] - turn[:-1]
    per = [np.add.reduceat(v, turn[:-1]) for v in (lt, d, ls * d)]
    cum, end, loss = np.zeros(len(n)), np.zeros(case["traj"]), np.zeros(case["traj"])
    for i in range(case["traj"]):
        k0, k1, r0, r1 = first[i], first[i + 1], traj[i], traj[i + 1]
        if mode == stride.TURN_MEAN:
            c = np.cumsum(per[0][k0:k1] / n[k0:k1])
            cum[k0:k1] = c
            hit = np.nonzero(c < lam)[0]
            last = turn[k0 + hit[0] + 1] if len(hit) else r1
        else:
            c = np.cumsum(lt[r0:r1])
            cum[k0:k1] = c[turn[k0 + 1:k1 + 1] - 1 - r0]
            hit = np.nonzero(c < lam)[0]
            last = r0 + hit[0] + 1 if len(hit) else r1
        end[i] = c[-1]
        loss[i] = np.sum((ls * d)[r0:last])
    prof = np.zeros((10, 3))
    pos = np.arange(len(lt)) - np.repeat(turn[:-1], n)
    bin_ = 10 * pos // np.repeat(n, n)
    for j, v in enumerate((d, lt, np.ones(len(lt)))):
        prof[:, j] = np.bincount(bin_, v, 10)
    return {"state": {"cum": end, "open_sums": np.zeros((case["traj"], 3)), "loss": loss, "counts": None, "turns": None},
            "stats": {"sum_t": per[0], "sum_d": per[1], "sum_l": per[2], "cum": cum, "mean_t": per[0] / n, "n": None},
            "status": None, **({"profile": prof} if case["profile"] else {})}


def _steps_exact(case, seed):
    S, T, tok, end, idx, lam = _step_inputs(case, seed)
    R, n, steps = case["rows"], case["rollouts"], case["steps"]
    row = _row_exact(S, T, tok, case["V"])
    end, lam = end.cpu().numpy(), lam.cpu().numpy().astype(np.float64)
    who = idx.cpu().numpy() if case["kind"] == "live" else np.arange(R)
    cum, loss, sums, cnt, stopped = np.zeros(n), np.zeros(n), np.zeros((n, 3)), np.zeros(n), np.zeros(n, bool)
    out = {k: np.full((steps, R), np.nan) for k in ROW_KEYS[:3]}
    ts = {k: np.zeros((steps, R)) for k in ("sum_t", "sum_d", "sum_l", "cum", "mean_t")}
    for k in range(steps):
        a = (k % case["ring"]) * R
        for b, r in enumerate(who):
            if stopped[r]:
                continue
            ls, lt, d = (row[key][a + b] for key in ROW_KEYS[:3])
            for key, v in zip(ROW_KEYS[:3], (ls, lt, d)):
                out[key][k, b] = v
            sums[r] += (lt, d, ls * d)
            cnt[r] += 1
            loss[r] += ls * d
            if case["mode"] == stride.TOKEN_SUM:
                cum[r] += lt
                stopped[r] |= cum[r] < lam[r]
            if end[k, b]:
                if case["mode"] == stride.TURN_MEAN:
                    cum[r] += sums[r, 0] / cnt[r]
                    stopped[r] |= cum[r] < lam[r]
                for key, v in zip(ts, (*sums[r], cum[r], sums[r, 0] / cnt[r])):
                    ts[key][k, b] = v
                sums[r], cnt[r] = 0.0, 0
    return {"rows": out, "stopped_now": None, "turns": {**{k: v.reshape(-1) for k, v in ts.items()}, "n": None},
            "state": {"cum": cum, "open_sums": sums, "loss": loss, "counts": None, "turns": None}}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("steps", "live"):
        return _steps_exact(case, seed)
    if kind == "scan":
        ls, lt = (v.double().cpu().numpy() for v in _logprob_inputs(case, seed))
        rows = {"opd": ls - lt}
    else:
        traj, turn, first = _layout(case, seed)
        ld = case["V"] if kind == "shards" else case["ld"]
        S, T, tok = _logits(case["rows"], case["V"], ld, case["dtype"], case["sigma"],
                            _sigma_t(case, seed, traj, turn, first), _gen(seed))
        rows = _row_exact(S, T, tok, case["V"])
        del S, T
        ls, lt = rows["logp_s"], rows["logp_t"]
        keys = ROW_KEYS[:5] if kind == "shards" else ROW_KEYS[:case["outputs"]]
        rows = {k: rows[k] for k in keys}
    r = {**_scan_exact(case, seed, ls, lt), "rows": rows}
    if case.get("tasks"):
        mean, _, task, _ = _buffer_inputs(case, seed)
        mean = mean.double().cpu().numpy()
        mean[task.cpu().numpy(), :case["turns"]] = r["stats"]["mean_t"].reshape(case["traj"], case["turns"])
        r["buffer"] = {"mean": mean, "n": None, "k_star": None, "k_max": None}
    return r
