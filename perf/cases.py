"""What a trainer has this library do, as cases that can be timed and compared.

Every case goes through the public binding (``paper_2605_28396_b200.api``) the way a training loop
does: the logits or hidden states come from the policies' forward pass, the gradient buffer is the
trainer's own, everything else is left to the call's defaults.

Paths (``case["path"]``):
  step          synchronous update on the prefix windows: divergence, gradient, windowed loss sums
  weighted      gamma > 0 update: read-only pass, return-to-go scan, gradient with its weights
  probe         delayed full-rollout probe: read-only pass over whole rollouts, alignment audit
  audit_step    the update and the audit on one batch: gradient inside the window, scalars beyond it
  drift         teacher drift along rollouts: entropy, rank, survival curves
  lmhead        the update from hidden states and LM heads, logits never materialised
  lmhead_audit  the audit in the space of the student's LM-head weight

Sizes are those of the repository's own workloads (``synth.CONFIGS``, ``synth.LMHEAD``, the tests and
the benchmark) and generic ones; value distributions are those of ``synth``.
"""
from __future__ import annotations

import math

import torch

from paper_2605_28396_b200 import api, synth

# Value recipes: standard deviation of the student logits, teacher = mix * student + noise, share of
# +10 spikes (the recipes of the configs with 4 096, 32 000 and 151 936 entries).
_RECIPES = {
    "plain": dict(s_std=2.0, mix=1.0, t_std=1.0, spike_p=0.0, tokens="uniform"),
    "mixed": dict(s_std=3.0, mix=0.8, t_std=1.5, spike_p=0.0, tokens="student"),
    "spiky": dict(s_std=4.0, mix=1.0, t_std=2.0, spike_p=0.05, tokens="student"),
}
_DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
_MODES = {"full": api.GRAD_FULL_KL, "sampled": api.GRAD_SAMPLED}


def _logits(name, path, B, T, V, *, ld=0, dtype="bf16", mode="full", recipe="spiky", lo=1 / 8,
            hi=1.0, rollout=1.0, gamma=0.0):
    """Windows are spread evenly over [lo, hi] of T, rollouts over [rollout, 1] of T (a rollout
    shorter than its window ends it early)."""
    return dict(name=name, path=path, B=B, T=T, V=V, ld=ld or V, dtype=dtype, mode=mode,
                recipe=recipe, lo=lo, hi=hi, rollout=rollout, gamma=gamma)


def _hidden(name, path, B, T, V, d_s, d_t, *, mode="full", grads="both", grad_dtype="bf16",
            w_std=0.02, lo=1 / 16, hi=1.0, rollout=1.0):
    return dict(name=name, path=path, B=B, T=T, V=V, d_s=d_s, d_t=d_t, mode=mode, grads=grads,
                grad_dtype=grad_dtype, w_std=w_std, lo=lo, hi=hi, rollout=rollout)


def listed():
    return [
        # a unit-test-sized update in fp32: launches and host work decide
        _logits("step_small_fp32", "step", 2, 64, 4096, dtype="f32", recipe="plain", lo=0.5),
        # an ordinary update of a 32 000-entry vocabulary
        _logits("step_32k", "step", 8, 1024, 32000, recipe="mixed"),
        # the headline update: reasoning-length rollouts, the largest vocabulary in use
        _logits("step_152k", "step", 16, 2048, 151936),
        # a vocabulary that is no multiple of anything, rows packed one after another
        _logits("step_odd_vocab", "step", 8, 512, 50257, recipe="mixed", lo=0.25, rollout=0.5),
        # fp32 logits and gradient, the sampled-token estimator
        _logits("step_fp32_sampled", "step", 8, 512, 32000, dtype="f32", mode="sampled",
                recipe="mixed", lo=0.25),
        # discounted return-to-go weights: two passes over the logits with a scan between them
        _logits("weighted_152k", "weighted", 8, 1024, 151936, mode="sampled", lo=0.25,
                rollout=0.5, gamma=0.99),
        # the delayed probe over whole rollouts that ended at different lengths
        _logits("probe_152k", "probe", 4, 8192, 151936, lo=1 / 16, hi=0.5, rollout=0.5),
        # update and audit from one batch
        _logits("audit_step_152k", "audit_step", 8, 1024, 151936, hi=0.75, rollout=0.75),
        # teacher drift diagnostics of a batch of rollouts
        _logits("drift_152k", "drift", 8, 2048, 151936, rollout=0.5),
        # the fused LM-head update at full size
        _hidden("lmhead_152k", "lmhead", 16, 4096, 151936, 2048, 2560),
        # the same for a small model and a few short rollouts
        _hidden("lmhead_small", "lmhead", 2, 300, 32000, 1024, 1536, lo=0.25, rollout=0.5),
        # the audit in weight space; rollouts outlast the longest candidate (2048 positions)
        _hidden("lmhead_audit", "lmhead_audit", 2, 4096, 151936, 2048, 2560, rollout=0.6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    path = rng.choice(["step"] * 6 + ["weighted", "probe", "probe", "audit_step", "drift"] +
                      ["lmhead"] * 3 + ["lmhead_audit"])
    if path.startswith("lmhead"):
        d_s = 8 * _log_int(rng, 512 // 8, 2560 // 8)
        d_t = 8 * _log_int(rng, d_s // 8, 3072 // 8)
        V = 8 * _log_int(rng, 8192 // 8, 151936 // 8)
        rows = _log_int(rng, 256, 16384)
        B = min(rng.randint(1, 16), max(1, rows // 32))
        T, rollout = max(1, rows // B), rng.choice([1.0, 0.5])
        if path == "lmhead_audit":       # rollouts outlast the longest candidate
            B, T, rollout = rng.randint(1, 4), _log_int(rng, 2304, 4608), 0.9
        case = _hidden("", path, B, T, V, d_s, d_t,
                       mode=rng.choice(["full", "full", "sampled"]),
                       grads=rng.choice(["both", "both", "both", "weight", "none"]),
                       grad_dtype=rng.choice(["bf16", "f32"]),
                       lo=rng.choice([1 / 16, 0.25]), rollout=rollout)
    else:
        V = _log_int(rng, 4096, 151936)
        kind = rng.choice(["round", "round", "padded", "odd"])
        if kind == "round":
            V = max(64, V // 64 * 64)
        ld = (V + 63) // 64 * 64 if kind == "padded" else V
        dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
        most = min(32768, 24e8 / V / (2 if dtype == "f32" else 1))
        rows = _log_int(rng, 64, most)
        B = min(rng.randint(1, 16), max(1, rows // 16))
        case = _logits("", path, B, max(1, rows // B), V, ld=ld, dtype=dtype,
                       mode="sampled" if path == "weighted" else rng.choice(["full", "full", "sampled"]),
                       recipe=rng.choice(["plain", "mixed", "spiky"]),
                       lo=rng.choice([1 / 16, 0.25, 0.5]), hi=rng.choice([0.5, 1.0]),
                       rollout=rng.choice([1.0, 0.5]),
                       gamma=rng.choice([0.9, 0.99, 1.0]) if path == "weighted" else 0.0)
    del case["name"]
    return case


def _lengths(case):
    """Window and rollout lengths as host lists (the same for every seed, so that the work is)."""
    B, T = case["B"], case["T"]

    def spread(lo, hi, order):
        step = [(b * order + order // 2) % B / max(1, B - 1) for b in range(B)] if B > 1 else [1.0]
        return [min(T, max(1, int(round(T * (lo + (hi - lo) * f))))) for f in step]

    return spread(case["lo"], case["hi"], 1), spread(case["rollout"], 1.0, 3)


def _generator(seed, b):
    g = torch.Generator(device="cuda")
    g.manual_seed(1 + 104729 * int(seed) + 17 * b)
    return g


def _int32(values):
    return torch.tensor(values, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    window, rollout = _lengths(case)
    if case["path"].startswith("lmhead"):
        return _prepare_hidden(case, seed, window, rollout)
    B, T, V, ld = case["B"], case["T"], case["V"], case["ld"]
    dt = _DTYPES[case["dtype"]]
    # rows past a rollout hold nothing a call may read
    student = torch.zeros((B, T, ld), dtype=dt, device="cuda")[:, :, :V]
    teacher = torch.zeros((B, T, ld), dtype=dt, device="cuda")[:, :, :V]
    tokens = torch.zeros((B, T), dtype=torch.int32, device="cuda")
    for b in range(B):
        n = rollout[b]
        synth.fill_sequence(student[b, :n], teacher[b, :n], tokens[b, :n],
                            gen=_generator(seed, b), **_RECIPES[case["recipe"]])
    grad = None
    if case["path"] in ("step", "weighted", "audit_step"):
        grad = torch.zeros((B, T, ld), dtype=dt, device="cuda")[:, :, :V]
    if case["path"] == "drift":
        student = None
    return dict(case=case, student=student, teacher=teacher, tokens=tokens, grad=grad,
                window=_int32(window), rollout=_int32(rollout), ks=_int32([1, 5, 20]))


def _prepare_hidden(case, seed, window, rollout):
    B, T, V = case["B"], case["T"], case["V"]
    g = _generator(seed, 999)
    ws = torch.randn((V, case["d_s"]), generator=g, device="cuda").mul_(case["w_std"]).bfloat16()
    wt = torch.randn((V, case["d_t"]), generator=g, device="cuda").mul_(case["w_std"]).bfloat16()
    hs = torch.zeros((B, T, case["d_s"]), dtype=torch.bfloat16, device="cuda")
    ht = torch.zeros((B, T, case["d_t"]), dtype=torch.bfloat16, device="cuda")
    tokens = torch.zeros((B, T), dtype=torch.int32, device="cuda")
    for b in range(B):
        g, n = _generator(seed, b), rollout[b]
        hs[b, :n] = torch.randn((n, case["d_s"]), generator=g, device="cuda").bfloat16()
        ht[b, :n] = torch.randn((n, case["d_t"]), generator=g, device="cuda").bfloat16()
        for t0 in range(0, n, 512):      # tokens from the student softmax (Gumbel-max)
            z = (hs[b, t0:min(n, t0 + 512)] @ ws.T).float()
            e = torch.rand(z.shape, generator=g, device="cuda").clamp_(min=1e-20)
            z -= e.log_().neg_().log_()
            tokens[b, t0:t0 + z.shape[0]] = z.argmax(dim=1).int()
    state = dict(case=case, hs=hs, ws=ws, ht=ht, wt=wt, tokens=tokens, window=_int32(window),
                 rollout=_int32(rollout), grad_hidden=None, grad_w=None)
    # the scheduler chose the windows on the host, so the trainer knows how many rows there are
    state["max_rows"] = sum(map(min, window, rollout)) if case["path"] == "lmhead" else sum(rollout)
    if case["path"] == "lmhead":
        if case["grads"] == "both":
            state["grad_hidden"] = torch.zeros_like(hs, dtype=_DTYPES[case["grad_dtype"]])
        if case["grads"] in ("both", "weight"):
            state["grad_w"] = torch.zeros((V, case["d_s"]), dtype=torch.float32, device="cuda")
    return state


def _scalars(o):
    return dict(kl=o.kl, logratio=o.logratio, gsq=o.gsq, status=o.dev_status)


def run(state):
    """One pass through the public entry points."""
    return _RUN[state["case"]["path"]](state)


def _run_step(s):
    o = api.adwin_opd_kl_fwd_bwd(s["student"], s["teacher"], s["tokens"], s["window"], s["rollout"],
                                 grad_mode=_MODES[s["case"]["mode"]], grad=s["grad"])
    seq, batch = api.adwin_window_reduce(o.kl, o.logratio, o.gsq, s["window"], s["rollout"])
    return dict(_scalars(o), grad=o.grad, seq=seq, batch=batch)


def _run_weighted(s):
    first = api.adwin_opd_kl_fwd_bwd(s["student"], s["teacher"], s["tokens"], s["window"],
                                     s["rollout"], want_gsq=False)
    rtg = api.adwin_return_to_go(first.logratio, s["window"], s["rollout"], s["case"]["gamma"])
    o = api.adwin_opd_kl_fwd_bwd_weighted(s["student"], s["teacher"], s["tokens"], s["window"],
                                          s["rollout"], rtg, grad=s["grad"])
    seq, batch = api.adwin_window_reduce(o.kl, o.logratio, o.gsq, s["window"], s["rollout"])
    return dict(_scalars(o), rtg=rtg, grad=o.grad, seq=seq, batch=batch)


def _audit(s, o):
    a = api.adwin_probe_align(o.kl, o.logratio, o.gsq, s["window"], s["rollout"])
    return dict(seq_stats=a.seq_stats, seq_full=a.seq_full, batch_stats=a.batch_stats,
                L_next=a.L_next, flags=a.flags)


def _run_probe(s):
    o = api.adwin_opd_kl_fwd_bwd(s["student"], s["teacher"], s["tokens"], s["window"], s["rollout"],
                                 grad_mode=_MODES[s["case"]["mode"]], flags=api.RANGE_FULL)
    return dict(_scalars(o), **_audit(s, o))


def _run_audit_step(s):
    o = api.adwin_opd_kl_fwd_bwd(s["student"], s["teacher"], s["tokens"], s["window"], s["rollout"],
                                 grad_mode=_MODES[s["case"]["mode"]], flags=api.RANGE_FULL,
                                 grad=s["grad"])
    seq, batch = api.adwin_window_reduce(o.kl, o.logratio, o.gsq, s["window"], s["rollout"])
    return dict(_scalars(o), grad=o.grad, seq=seq, batch=batch, **_audit(s, o))


def _run_drift(s):
    d = api.adwin_teacher_drift(s["teacher"], s["tokens"], s["rollout"])
    c = api.adwin_drift_curves(d.entropy, d.rank, s["rollout"], s["ks"])
    return dict(entropy=d.entropy, rank=d.rank, status=d.dev_status, worst=c.worst_rank,
                survival=c.survival, bf_mean=c.bf_mean, n_active=c.n_active)


def _run_lmhead(s):
    o = api.adwin_opd_kl_lmhead_fwd_bwd(s["hs"], s["ws"], s["ht"], s["wt"], s["tokens"], s["window"],
                                        s["rollout"], grad_mode=_MODES[s["case"]["mode"]],
                                        grad_hidden=s["grad_hidden"], grad_w=s["grad_w"],
                                        max_rows=s["max_rows"])
    seq, batch = api.adwin_window_reduce(o.kl, o.logratio, o.gsq, s["window"], s["rollout"])
    return dict(_scalars(o), grad_hidden=s["grad_hidden"], grad_w=s["grad_w"], seq=seq, batch=batch)


def _run_lmhead_audit(s):
    o = api.adwin_lmhead_weight_align(s["hs"], s["ws"], s["ht"], s["wt"], s["tokens"], s["rollout"],
                                      grad_mode=_MODES[s["case"]["mode"]], max_rows=s["max_rows"])
    return dict(_scalars(o), batch_stats=o.batch_stats, L_next=o.L_next, flags=o.flags)


_RUN = dict(step=_run_step, weighted=_run_weighted, probe=_run_probe, audit_step=_run_audit_step,
            drift=_run_drift, lmhead=_run_lmhead, lmhead_audit=_run_lmhead_audit)


def work(case):
    """Bytes that have to be read and written once and, for the contractions, their operations."""
    window, rollout = _lengths(case)
    n_win, n_all, V = sum(map(min, window, rollout)), sum(rollout), case["V"]
    path = case["path"]
    if not path.startswith("lmhead"):
        es = 4 if case["dtype"] == "f32" else 2
        row = V * es
        if path == "step":
            n = 3 * n_win
        elif path == "weighted":       # the scan stands between the two reads
            n = 5 * n_win
        elif path == "probe":
            n = 2 * n_all
        elif path == "audit_step":
            n = 2 * n_all + n_win
        else:
            n = n_all
        return {"bytes": float(n * row + 24 * case["B"] * case["T"]), "flops": 0.0}
    d_s, d_t = case["d_s"], case["d_t"]
    rows = n_win if path == "lmhead" else n_all
    flops = 2.0 * rows * V * (d_s + d_t)
    bytes_ = 2.0 * (V + rows) * (d_s + d_t)
    if path == "lmhead_audit":
        flops += 2.0 * rows * V * d_s
    else:
        if case["grads"] == "both":
            flops += 2.0 * rows * V * d_s
            bytes_ += rows * d_s * (4 if case["grad_dtype"] == "f32" else 2)
        if case["grads"] != "none":
            flops += 2.0 * rows * V * d_s
            bytes_ += 4.0 * V * d_s
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """About four times the largest distance from a 64-bit evaluation seen over the listed cases and
    eighty drawn ones.  A bf16 gradient is off by its own rounding (2-norm 2e-3, one entry 2^-8);
    the weight gradient's largest single error (0.09 of its root mean square) is a token that was
    sampled far more often than the rest.  Scalars alone: squared norms 1.8e-6 and, one row, 4e-5."""
    path = case["path"]
    if path == "lmhead_audit":
        # cosines of a gradient that was rounded to bf16: seen 3e-5, sampled estimator 6e-4
        return {"rel": 1.2e-4, "max": 3e-4} if case["mode"] == "full" else {"rel": 2.5e-3, "max": 2.6e-3}
    if path == "lmhead":
        return {"rel": 4e-5, "max": 1e-4} if case["grads"] == "none" else {"rel": 1e-2, "max": 0.4}
    if case["dtype"] == "bf16" and path in ("step", "weighted", "audit_step"):
        return {"rel": 7e-3, "max": 1.6e-2}
    return {"rel": 8e-6, "max": 2e-4}
