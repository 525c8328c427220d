"""GPU parity: the CUDA path (through the C ABI) against the float64 oracle, element by element."""
import math
import threading

import numpy as np
import pytest
import torch

from oracle import adwin_oracle as O
from paper_2605_28396_b200 import api, synth
from tests import parity as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
PATHS = {"staged": api.FORCE_STAGED, "generic": api.FORCE_GENERIC, "default": 0}


def run_and_check(batch, *, grad_dtype, grad_mode=api.GRAD_FULL_KL, flags=0, grad_scale=1.0,
                  allow_status=0, sentinel=7.0, rtol_gsq_grad=None):
    B, T, V = batch.shape
    grad = None
    if grad_dtype is not None:
        grad = torch.full((B, T, V), sentinel, dtype=grad_dtype, device=batch.student.device)
    got = api.adwin_opd_kl_fwd_bwd(batch.student, batch.teacher, batch.tokens, batch.window,
                                   batch.rollout_len, grad_scale=grad_scale, grad_mode=grad_mode,
                                   flags=flags, grad=grad, want_lse=True)
    torch.cuda.synchronize()
    api.raise_on_dev_status(got.dev_status, allow=allow_status)
    oflags = flags & (api.ZERO_TAIL | api.RANGE_FULL)
    ref = P.oracle_batch(batch, grad_scale=grad_scale, grad_mode=grad_mode, flags=oflags,
                         want_grad=grad is not None,
                         grad_init=None if grad is None else np.full((B, T, V), sentinel))
    rtol = P.rtol_for(batch.student.dtype, grad_dtype)
    w, r = batch.window.cpu().numpy(), batch.rollout_len.cpu().numpy()
    mask = P.processed_mask(w, r, T, bool(flags & api.RANGE_FULL))
    gmask = P.processed_mask(w, r, T, False) if grad is not None else None
    P.check_scalars(got, ref, rtol, mask, grad_mask=gmask, rtol_gsq_grad=rtol_gsq_grad)
    if grad is not None:
        g = got.grad.double().cpu().numpy()
        wmask = P.processed_mask(w, r, T, False)
        guard = 1e-4 if (grad_dtype == torch.float32 and grad_mode == api.GRAD_FULL_KL) else None
        P.check_grad_rows(g[wmask], ref["grad"][wmask], rtol, store=P.STORE[grad_dtype],
                          guard=guard)
        # rows outside the window: untouched (sentinel) or exactly zero with ZERO_TAIL
        want = 0.0 if flags & api.ZERO_TAIL else sentinel
        assert (g[~wmask] == want).all()
    return got, ref


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("mode", [api.GRAD_FULL_KL, api.GRAD_SAMPLED])
def test_config1_fp32(path, mode):
    batch = synth.make_batch(1, device=DEV)
    run_and_check(batch, grad_dtype=torch.float32, grad_mode=mode, flags=PATHS[path])


@pytest.mark.parametrize("path", PATHS)
def test_config2_bf16_full_size(path):
    batch = synth.make_batch(2, device=DEV)
    run_and_check(batch, grad_dtype=torch.bfloat16, flags=PATHS[path])


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("mode", [api.GRAD_FULL_KL, api.GRAD_SAMPLED])
def test_config3_reduced_T_full_vocab(path, mode):
    batch = synth.make_batch(3, device=DEV, B=4, T=48)           # windows 6,12,24,48
    run_and_check(batch, grad_dtype=torch.bfloat16, grad_mode=mode, flags=PATHS[path])


@pytest.mark.parametrize("path", PATHS)
def test_config4_probe_reduced_with_ragged_rollouts(path):
    batch = synth.make_batch(4, device=DEV, B=4, T=64, ragged_rollout=True)
    got, ref = run_and_check(batch, grad_dtype=None, flags=api.RANGE_FULL | PATHS[path])
    cands = torch.tensor([4, 8, 16, 32, 64], dtype=torch.int32, device=DEV)
    al = api.adwin_probe_align(got.kl, got.logratio, got.gsq, batch.window, batch.rollout_len,
                               cands, 0.0)
    torch.cuda.synchronize()
    w, r = batch.window.cpu().numpy(), batch.rollout_len.cpu().numpy()
    # (i) same per-token inputs through the oracle's audit: sums agree to float64 rounding
    same = O.probe_align(got.kl.cpu().numpy(), got.logratio.cpu().numpy(), got.gsq.cpu().numpy(),
                         w, r, cands.cpu().numpy(), math.sqrt(2) / 2)
    np.testing.assert_allclose(al.seq_stats.cpu().numpy(), same["seq_stats"], rtol=1e-12, atol=1e-12)
    np.testing.assert_allclose(al.seq_full.cpu().numpy(), same["seq_full"], rtol=1e-12, atol=1e-12)
    np.testing.assert_allclose(al.batch_stats.cpu().numpy(), same["batch_stats"], rtol=1e-12)
    assert int(al.L_next.item()) == same["L_next"] and int(al.flags.item()) == same["flags"]
    # (ii) end to end against the oracle run from the logits
    e2e = O.probe_align(ref["kl"], ref["logratio"], ref["gsq"], w, r, cands.cpu().numpy(),
                        math.sqrt(2) / 2)
    np.testing.assert_allclose(al.batch_stats.cpu().numpy()[:, :2], e2e["batch_stats"][:, :2],
                               rtol=P.RTOL_SUM)
    near = np.abs(e2e["batch_stats"][:-1, 0] - math.sqrt(2) / 2).min() <= 1e-6
    assert int(al.L_next.item()) == e2e["L_next"] or near


@pytest.mark.parametrize("path", PATHS)
def test_range_full_with_gradient_inside_window_only(path):
    batch = synth.make_batch(2, device=DEV, B=3, T=40, V=4096, ragged_rollout=True)
    batch.window = torch.tensor([5, 17, 0], dtype=torch.int32, device=DEV)
    batch.rollout_len = torch.tensor([40, 17, 9], dtype=torch.int32, device=DEV)
    run_and_check(batch, grad_dtype=torch.bfloat16, flags=api.RANGE_FULL | PATHS[path])
    run_and_check(batch, grad_dtype=torch.float32,
                  flags=api.RANGE_FULL | api.ZERO_TAIL | PATHS[path])


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("in_dt,g_dt", [(1, torch.bfloat16), (1, torch.float32),
                                        (2, torch.float32), (2, torch.bfloat16)])
def test_dtype_combinations_and_grad_scale(path, in_dt, g_dt):
    batch = synth.make_batch(in_dt, device=DEV, B=2, T=12, V=8192)
    batch.window = torch.tensor([12, 5], dtype=torch.int32, device=DEV)
    for mode in (api.GRAD_FULL_KL, api.GRAD_SAMPLED):
        run_and_check(batch, grad_dtype=g_dt, grad_mode=mode, grad_scale=-0.125,
                      flags=PATHS[path] | api.ZERO_TAIL)


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("in_dt,g_dt", [(2, torch.bfloat16), (1, torch.float32), (2, None)])
def test_sampled_token_far_below_the_row_maximum(path, in_dt, g_dt):
    """Rows whose sampled token has a vanishing probability (the staged kernel's shared reference
    overflows there and the row is redone with a running maximum), next to ordinary rows."""
    batch = synth.make_batch(in_dt, device=DEV, B=2, T=6, V=8192)
    batch.window = torch.tensor([6, 4], dtype=torch.int32, device=DEV)
    for (b, t, gap_s, gap_t) in [(0, 1, 90.0, 0.0), (0, 3, 0.0, 120.0), (1, 2, 60.0, 70.0),
                                 (1, 5, 200.0, 200.0)]:
        y = int(batch.tokens[b, t])
        batch.student[b, t, y] = batch.student[b, t].float().max() - gap_s
        batch.teacher[b, t, y] = batch.teacher[b, t].float().max() - gap_t
    flags = PATHS[path] | (api.RANGE_FULL if g_dt is None else 0)
    run_and_check(batch, grad_dtype=g_dt, flags=flags)
    run_and_check(batch, grad_dtype=g_dt, grad_mode=api.GRAD_SAMPLED, flags=flags)


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("in_dt,g_dt,shift", [(1, torch.float32, 8.0), (2, torch.bfloat16, 50.0),
                                              (2, torch.bfloat16, 1000.0), (2, None, 1000.0)])
def test_teacher_rows_shifted_by_a_constant(path, in_dt, g_dt, shift):
    """The divergence does not depend on a constant added to a logit row.  The kernels work with
    z - u in fp32, whose rounding grows with such an offset (offset * 2^-24 against differences of
    order one): an offset of 8 must stay inside the fp32 tolerance of 1e-5 (an offset of 50
    already costs 1.3e-5 on a gradient row in any fp32 evaluation of z - u), one of 1000 inside
    the bf16 tolerance."""
    batch = synth.make_batch(in_dt, device=DEV, B=2, T=10, V=8192)
    batch.window = torch.tensor([10, 6], dtype=torch.int32, device=DEV)
    batch.teacher = (batch.teacher.float() + shift).to(batch.teacher.dtype)
    # With the offset of 1000 the squared norm of a written gradient row is held to the arithmetic
    # tolerance of the dtype instead of 1e-4: the staged kernel forms coef*(z-u) - coef*E_p[z-u]
    # uncentred, which costs offset * 2^-24 = 6e-5 relative on every entry there.
    for mode in (api.GRAD_FULL_KL, api.GRAD_SAMPLED):
        run_and_check(batch, grad_dtype=g_dt, grad_mode=mode, flags=PATHS[path],
                      rtol_gsq_grad=2e-3 if shift >= 1000.0 else None)


@pytest.mark.parametrize("g_dt", [torch.bfloat16, None])
def test_teacher_logits_outside_the_range_of_the_polynomial_exponential(g_dt):
    """The staged kernel takes the exponential of the first teacher pair of every 16-byte piece
    from a polynomial that is only valid on a clamped range: entries far below the reference must
    still count as nil, and one far above it must still send the row to the safe path."""
    batch = synth.make_batch(2, device=DEV, B=2, T=5, V=8192)
    batch.window = torch.tensor([5, 3], dtype=torch.int32, device=DEV)
    first_pair = torch.arange(0, 8192, 8, device=DEV)
    batch.teacher[0, 1, first_pair[5:400]] = -3.0e4            # far below: 2^x underflows
    batch.teacher[0, 1, first_pair[5:400] + 1] = -250.0
    batch.teacher[1, 0, first_pair[::7]] = -1.0e3
    uy = float(batch.teacher[0, 3, int(batch.tokens[0, 3])])
    batch.teacher[0, 3, first_pair[17]] = uy + 96.0              # far above, polynomial position
    uy = float(batch.teacher[1, 2, int(batch.tokens[1, 2])])
    batch.teacher[1, 2, first_pair[900] + 1] = uy + 71.0         # just inside the clamp
    flags = api.RANGE_FULL if g_dt is None else 0
    run_and_check(batch, grad_dtype=g_dt, flags=flags)
    run_and_check(batch, grad_dtype=g_dt, grad_mode=api.GRAD_SAMPLED, flags=flags)


@pytest.mark.parametrize("V", [1, 2, 7, 8, 9, 1001, 4100, 65537])
def test_odd_vocab_sizes(V):
    batch = synth.make_batch(2, device=DEV, B=2, T=6, V=V)
    batch.window = torch.tensor([6, 3], dtype=torch.int32, device=DEV)
    run_and_check(batch, grad_dtype=torch.bfloat16)
    run_and_check(batch, grad_dtype=None)


@pytest.mark.parametrize("V", [409600, 1048576])
def test_vocabulary_beyond_what_tensor_memory_holds(V):
    """The staged kernel parks the streamed chunks of a row slice in tensor memory between its
    sweeps when they fit (up to 5 chunks + the resident slots per CTA, with clusters of up to 4);
    larger rows go back to fetching those chunks a second time through the shared-memory ring.
    Both sizes here are beyond the limit (the paper-scale vocabulary is inside it)."""
    batch = synth.make_batch(3, device=DEV, B=1, T=5, V=V)
    batch.window = torch.tensor([4], dtype=torch.int32, device=DEV)
    for mode in (api.GRAD_FULL_KL, api.GRAD_SAMPLED):
        run_and_check(batch, grad_dtype=torch.bfloat16, grad_mode=mode, flags=api.FORCE_STAGED)


@pytest.mark.parametrize("path", PATHS)
def test_padded_row_stride(path):
    B, T, V, ld = 2, 5, 4096, 4096 + 64
    base = synth.make_batch(2, device=DEV, B=B, T=T, V=ld)
    batch = synth.Batch(base.student[..., :V], base.teacher[..., :V],
                        torch.randint(0, V, (B, T), dtype=torch.int32, device=DEV),
                        torch.tensor([5, 2], dtype=torch.int32, device=DEV), base.rollout_len, 2)
    grad = torch.full((B, T, ld), 3.0, dtype=torch.bfloat16, device=DEV)
    got = api.adwin_opd_kl_fwd_bwd(batch.student, batch.teacher, batch.tokens, batch.window,
                                   batch.rollout_len, grad=grad[..., :V], flags=PATHS[path])
    torch.cuda.synchronize()
    ref = O.opd_kl_fwd_bwd(synth.bits_for_oracle(batch.student.contiguous()),
                           synth.bits_for_oracle(batch.teacher.contiguous()),
                           batch.tokens.cpu().numpy(), batch.window.cpu().numpy(), None)
    mask = P.processed_mask(batch.window.cpu().numpy(), np.array([T, T]), T)
    P.check_scalars(got, ref, 2e-3, mask)
    g = grad.double().cpu().numpy()
    P.check_grad_rows(g[..., :V][mask], ref["grad"][mask], 2e-3, store=2.0 ** -8)
    assert (g[..., V:] == 3.0).all()                     # padding columns never written


def test_unaligned_row_stride_runs_through_the_generic_kernel():
    B, T, V, ld = 2, 4, 1000, 1003                       # rows not 16-byte aligned
    base = synth.make_batch(2, device=DEV, B=B, T=T, V=ld)
    s, t = base.student[..., :V], base.teacher[..., :V]
    tok = torch.randint(0, V, (B, T), dtype=torch.int32, device=DEV)
    win = torch.tensor([4, 4], dtype=torch.int32, device=DEV)
    gbuf = torch.zeros((B, T, ld), dtype=torch.float32, device=DEV)
    got = api.adwin_opd_kl_fwd_bwd(s, t, tok, win, None, grad=gbuf[..., :V])
    torch.cuda.synchronize()
    ref = O.opd_kl_fwd_bwd(synth.bits_for_oracle(s.contiguous()),
                           synth.bits_for_oracle(t.contiguous()), tok.cpu().numpy(),
                           win.cpu().numpy(), None)
    mask = np.ones((B, T), dtype=bool)
    P.check_scalars(got, ref, 2e-3, mask)
    P.check_grad_rows(gbuf[..., :V].double().cpu().numpy()[mask], ref["grad"][mask], 2e-3)


@pytest.mark.parametrize("path", PATHS)
def test_degenerate_windows(path):
    batch = synth.make_batch(2, device=DEV, B=4, T=8, V=4096)
    batch.window = torch.tensor([0, 8, 100, 3], dtype=torch.int32, device=DEV)     # W=0, W>T
    batch.rollout_len = torch.tensor([8, 0, 5, 8], dtype=torch.int32, device=DEV)  # R=0, W>R
    got, _ = run_and_check(batch, grad_dtype=torch.bfloat16, flags=PATHS[path])
    seq, tot = api.adwin_window_reduce(got.kl, got.logratio, got.gsq, batch.window,
                                       batch.rollout_len)
    torch.cuda.synchronize()
    assert seq[:, 3].tolist() == [0.0, 0.0, 5.0, 3.0] and tot[3].item() == 8.0
    batch.window[:] = 0                                                            # nothing at all
    got, _ = run_and_check(batch, grad_dtype=torch.bfloat16, flags=PATHS[path])
    assert (got.kl == 0).all()


@pytest.mark.parametrize("path", PATHS)
def test_device_detected_conditions_set_status_bits(path):
    batch = synth.make_batch(2, device=DEV, B=2, T=6, V=4096)
    batch.tokens[0, 1] = 4096
    batch.tokens[1, 0] = -3
    got, ref = run_and_check(batch, grad_dtype=torch.bfloat16, flags=PATHS[path],
                             allow_status=api.DEV_TOKEN_RANGE)
    assert int(got.dev_status.item()) & api.DEV_TOKEN_RANGE
    assert torch.isnan(got.logratio[0, 1]) and torch.isnan(got.logratio[1, 0])
    assert torch.isfinite(got.kl).all()
    # invalid lengths are clamped and reported, never dereferenced out of range
    batch = synth.make_batch(2, device=DEV, B=3, T=6, V=4096)
    batch.window = torch.tensor([-2, 4, 6], dtype=torch.int32, device=DEV)
    batch.rollout_len = torch.tensor([6, -1, 9], dtype=torch.int32, device=DEV)
    got = api.adwin_opd_kl_fwd_bwd(batch.student, batch.teacher, batch.tokens, batch.window,
                                   batch.rollout_len, flags=PATHS[path])
    torch.cuda.synchronize()
    assert int(got.dev_status.item()) & api.DEV_WINDOW
    assert (got.kl[0] == 0).all() and (got.kl[1] == 0).all() and (got.kl[2] != 0).all()


@pytest.mark.parametrize("path", PATHS)
def test_bitwise_reproducible(path):
    batch = synth.make_batch(3, device=DEV, B=2, T=16, V=151936)
    outs = []
    for _ in range(3):
        g = torch.zeros(batch.shape, dtype=torch.bfloat16, device=DEV)
        got = api.adwin_opd_kl_fwd_bwd(batch.student, batch.teacher, batch.tokens, batch.window,
                                       batch.rollout_len, grad=g, flags=PATHS[path])
        torch.cuda.synchronize()
        outs.append((got.kl.clone(), got.logratio.clone(), got.gsq.clone(), g))
    for o in outs[1:]:
        for a, b in zip(outs[0], o):
            assert torch.equal(a, b)


def test_window_reduce_against_oracle():
    batch = synth.make_batch(2, device=DEV, B=6, T=64, V=4096, ragged_rollout=True)
    got, ref = run_and_check(batch, grad_dtype=torch.bfloat16)
    seq, tot = api.adwin_window_reduce(got.kl, got.logratio, got.gsq, batch.window,
                                       batch.rollout_len)
    torch.cuda.synchronize()
    w, r = batch.window.cpu().numpy(), batch.rollout_len.cpu().numpy()
    s_same, t_same = O.window_reduce(got.kl.cpu().numpy(), got.logratio.cpu().numpy(),
                                     got.gsq.cpu().numpy(), w, r)
    np.testing.assert_allclose(seq.cpu().numpy(), s_same, rtol=1e-13, atol=1e-13)
    np.testing.assert_allclose(tot.cpu().numpy(), t_same, rtol=1e-13, atol=1e-13)
    s_ref, t_ref = O.window_reduce(ref["kl"], ref["logratio"], ref["gsq"], w, r)
    mask = P.processed_mask(w, r, 64)
    terms = [np.abs(ref[k] * mask).sum() for k in ("kl", "logratio", "gsq")] + [0.0]
    P.check_sums(tot.cpu().numpy(), t_ref, terms)
    seq2, tot2 = api.adwin_window_reduce(got.kl, got.logratio, None, batch.window, None)
    torch.cuda.synchronize()
    assert (seq2[:, 2] == 0).all() and tot2[2].item() == 0


def test_probe_align_default_candidates_and_flags():
    B, T = 5, 4096
    g = torch.Generator(device=DEV).manual_seed(5)
    gsq = torch.rand((B, T), device=DEV, generator=g)
    kl = torch.rand((B, T), device=DEV, generator=g)
    c = torch.randn((B, T), device=DEV, generator=g)
    win = torch.full((B,), 256, dtype=torch.int32, device=DEV)
    rl = torch.tensor([4096, 3000, 100, 2048, 64], dtype=torch.int32, device=DEV)
    al = api.adwin_probe_align(kl, c, gsq, win, rl)
    torch.cuda.synchronize()
    ref = O.probe_align(kl.cpu().numpy(), c.cpu().numpy(), gsq.cpu().numpy(), win.cpu().numpy(),
                        rl.cpu().numpy(), np.array(api.DEFAULT_CANDIDATES, np.int32), api.RHO_STAR)
    np.testing.assert_allclose(al.batch_stats.cpu().numpy(), ref["batch_stats"], rtol=1e-12)
    np.testing.assert_allclose(al.seq_stats.cpu().numpy(), ref["seq_stats"], rtol=1e-12)
    assert int(al.L_next.item()) == ref["L_next"] and int(al.flags.item()) == ref["flags"]
    # nothing admissible / degenerate norms
    gsq0 = torch.zeros((B, T), device=DEV)
    al = api.adwin_probe_align(kl, c, gsq0, win, rl)
    torch.cuda.synchronize()
    assert int(al.flags.item()) & api.ALIGN_DEGENERATE and int(al.L_next.item()) == 64
    gsq1 = torch.zeros((B, T), device=DEV)
    gsq1[:, 60] = 1.0
    gsq1[:, 3000:] = 100.0
    al = api.adwin_probe_align(kl, c, gsq1, win, None, rho_star=0.9)
    torch.cuda.synchronize()
    assert int(al.flags.item()) & api.ALIGN_NONE_ADMISSIBLE and int(al.L_next.item()) == 2048


@pytest.mark.parametrize("flags", [0, api.RANGE_FULL | api.ZERO_TAIL])
def test_host_buffer_entry_point_matches_device_entry_point(flags):
    batch = synth.make_batch(2, device="cpu", B=3, T=70, V=8192, ragged_rollout=True)
    batch.window = torch.tensor([70, 9, 33], dtype=torch.int32)
    batch.rollout_len = torch.tensor([70, 40, 20], dtype=torch.int32)
    pin = lambda x: x.contiguous().pin_memory()
    s_h, t_h, tok_h = pin(batch.student), pin(batch.teacher), pin(batch.tokens)
    g_h = torch.full(batch.shape, 5.0, dtype=torch.bfloat16).pin_memory()
    got = api.adwin_opd_kl_fwd_bwd_host(s_h, t_h, tok_h, batch.window, batch.rollout_len,
                                        device=DEV, grad=g_h, flags=flags, rows_per_stage=16,
                                        grad_scale=0.5)
    torch.cuda.synchronize()
    assert int(got.dev_status.item()) == 0
    dgrad = torch.full(batch.shape, 5.0, dtype=torch.bfloat16, device=DEV)
    ref = api.adwin_opd_kl_fwd_bwd(batch.student.to(DEV), batch.teacher.to(DEV),
                                   batch.tokens.to(DEV), batch.window.to(DEV),
                                   batch.rollout_len.to(DEV), grad=dgrad, flags=flags,
                                   grad_scale=0.5)
    torch.cuda.synchronize()
    # same kernels on the same values: only the staging layout differs
    assert torch.allclose(got.kl, ref.kl.cpu(), rtol=1e-6, atol=1e-7)
    assert torch.allclose(got.logratio, ref.logratio.cpu(), rtol=1e-6, atol=1e-7)
    assert torch.allclose(got.gsq, ref.gsq.cpu(), rtol=1e-5, atol=1e-12)
    assert torch.equal(g_h, dgrad.cpu())
    with pytest.raises(api.AdwinError):
        api.adwin_opd_kl_fwd_bwd_host(s_h, t_h, tok_h, torch.tensor([-1, 2, 3], dtype=torch.int32),
                                      None, device=DEV)


def _oracle_on_rows(batch, rows, **kw):
    """Oracle on selected (b, t) rows only: each row becomes a one-token sequence inside its window."""
    bs = torch.tensor([b for b, _ in rows], device=batch.student.device)
    ts = torch.tensor([t for _, t in rows], device=batch.student.device)
    s = synth.bits_for_oracle(batch.student[bs, ts].unsqueeze(1))
    t = synth.bits_for_oracle(batch.teacher[bs, ts].unsqueeze(1))
    tok = batch.tokens[bs, ts].unsqueeze(1).cpu().numpy()
    return O.opd_kl_fwd_bwd(s, t, tok, np.ones(len(rows), np.int32), None, **kw)


def _sample_rows(limits, per_seq, rng):
    """First, last and a few random processed rows of every sequence."""
    rows = []
    for b, n in enumerate(limits):
        if n <= 0:
            continue
        ts = {0, int(n) - 1} | {int(x) for x in rng.integers(0, int(n), size=per_seq)}
        rows += [(b, t) for t in sorted(ts)]
    return rows


def test_config3_full_size_in_the_bench_launch_configuration_on_sampled_rows():
    """The workload bench.py times, at full size, with the oracle on sampled rows plus the
    properties that hold at any size (untouched tail, zeroed scalars, reproducible sums)."""
    batch = synth.make_batch(3, device=DEV)
    B, T, V = batch.shape
    sentinel = 7.0
    grad = torch.full((B, T, V), sentinel, dtype=torch.bfloat16, device=DEV)
    got = api.adwin_opd_kl_fwd_bwd(batch.student, batch.teacher, batch.tokens, batch.window,
                                   batch.rollout_len, grad=grad)
    torch.cuda.synchronize()
    api.raise_on_dev_status(got.dev_status)
    w = batch.window.cpu().numpy()
    rows = _sample_rows(w, 2, np.random.default_rng(3))
    ref = _oracle_on_rows(batch, rows)
    bs = torch.tensor([b for b, _ in rows], device=DEV)
    ts = torch.tensor([t for _, t in rows], device=DEV)
    sub = type("S", (), {})()
    sub.kl, sub.logratio, sub.gsq = (x[bs, ts].unsqueeze(1) for x in (got.kl, got.logratio, got.gsq))
    ones = np.ones((len(rows), 1), dtype=bool)
    P.check_scalars(sub, ref, 2e-3, ones, grad_mask=ones)
    P.check_grad_rows(grad[bs, ts].double().cpu().numpy(), ref["grad"][:, 0], 2e-3, store=2.0 ** -8)
    for b in range(B):                                   # rows past the window: never touched
        assert (grad[b, int(w[b]):] == sentinel).all()
        assert (got.kl[b, int(w[b]):] == 0).all() and (got.gsq[b, int(w[b]):] == 0).all()
    seq, tot = api.adwin_window_reduce(got.kl, got.logratio, got.gsq, batch.window, batch.rollout_len)
    torch.cuda.synchronize()
    mask = torch.arange(T, device=DEV)[None, :] < batch.window[:, None]
    want = (got.kl.double() * mask).sum()
    assert abs(tot[0].item() - want.item()) <= 1e-9 * abs(want.item())
    assert tot[3].item() == float(w.sum()) and torch.isfinite(got.kl).all() and (got.kl[mask] > -1e-4).all()


def test_config4_full_size_probe_pass_on_sampled_rows():
    """Delayed full-rollout probe at full size (B=8, T=8192, V=151936, ragged rollouts): one pass
    without a gradient, then the alignment audit; oracle on sampled rows, audit against the oracle's
    audit of the same per-token scalars."""
    batch = synth.make_batch(4, device=DEV, ragged_rollout=True, fill_all_rows=False)
    B, T, V = batch.shape
    got = api.adwin_opd_kl_fwd_bwd(batch.student, batch.teacher, batch.tokens, batch.window,
                                   batch.rollout_len, flags=api.RANGE_FULL)
    torch.cuda.synchronize()
    api.raise_on_dev_status(got.dev_status)
    w, r = batch.window.cpu().numpy(), batch.rollout_len.cpu().numpy()
    rows = _sample_rows(r, 3, np.random.default_rng(4))
    ref = _oracle_on_rows(batch, rows, want_grad=False)
    bs = torch.tensor([b for b, _ in rows], device=DEV)
    ts = torch.tensor([t for _, t in rows], device=DEV)
    sub = type("S", (), {})()
    sub.kl, sub.logratio, sub.gsq = (x[bs, ts].unsqueeze(1) for x in (got.kl, got.logratio, got.gsq))
    P.check_scalars(sub, ref, 2e-3, np.ones((len(rows), 1), dtype=bool))
    for b in range(B):
        assert (got.kl[b, int(r[b]):] == 0).all()
    al = api.adwin_probe_align(got.kl, got.logratio, got.gsq, batch.window, batch.rollout_len)
    torch.cuda.synchronize()
    same = O.probe_align(got.kl.cpu().numpy(), got.logratio.cpu().numpy(), got.gsq.cpu().numpy(),
                         w, r, np.array(api.DEFAULT_CANDIDATES, np.int32), api.RHO_STAR)
    np.testing.assert_allclose(al.batch_stats.cpu().numpy(), same["batch_stats"], rtol=1e-12)
    np.testing.assert_allclose(al.seq_stats.cpu().numpy(), same["seq_stats"], rtol=1e-12, atol=1e-12)
    assert int(al.L_next.item()) == same["L_next"] and int(al.flags.item()) == same["flags"]
    rho = al.batch_stats[:, 0].cpu().numpy()
    assert (np.diff(rho[:-1]) >= -1e-12).all() and (rho <= 1 + 1e-12).all()


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("in_dt,g_dt", [(1, torch.float32), (1, torch.bfloat16), (2, torch.bfloat16),
                                        (2, torch.float32), (2, None)])
@pytest.mark.parametrize("V", [33, 1001, 11523, 23046, 50257])
def test_rows_that_start_and_end_off_16_byte_boundaries(path, in_dt, g_dt, V):
    """Packed rows of an odd length: every row has another offset from a 16-byte boundary, its first
    and last pieces are shared with its neighbours (rows past the window must keep their sentinel),
    and the pieces end just before, on and after a chunk or a cluster slice (11 520 and 23 040
    bf16 entries are one and two full chunks).  Tokens in the partial pieces, and a row whose sampled
    token is far below the maximum (redone with a running maximum)."""
    batch = synth.make_batch(in_dt, device=DEV, B=2, T=7, V=V)
    batch.window = torch.tensor([7, 4], dtype=torch.int32, device=DEV)
    batch.tokens[0, 1], batch.tokens[0, 2], batch.tokens[1, 3] = 0, V - 1, V - 2
    # (both policies: z - u is centred on the sampled token's difference, whose magnitude times 2^-24
    # is the fp32 error of every centred difference -- 7e-6 for 120, most of the fp32 tolerance)
    y = int(batch.tokens[0, 4])
    batch.student[0, 4, y] = batch.student[0, 4].float().max() - 120.0
    batch.teacher[0, 4, y] = batch.teacher[0, 4].float().max() - 120.0
    flags = PATHS[path] | (api.RANGE_FULL if V == 1001 else 0)
    for mode in (api.GRAD_FULL_KL, api.GRAD_SAMPLED):
        run_and_check(batch, grad_dtype=g_dt, grad_mode=mode, flags=flags)


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("V,ld,ld_grad", [(1001, 1008, 1008), (1001, 1008, 1024), (1001, 1003, 1003),
                                          (1001, 1003, 1005), (12000, 12004, 12004)])
def test_odd_rows_at_a_padded_stride(path, V, ld, ld_grad):
    """Odd vocabularies in padded rows, whole and off the boundaries, the gradient at the same
    stride and at another one; the padding is never written."""
    B, T = 2, 5
    base = synth.make_batch(2, device=DEV, B=B, T=T, V=ld)
    s, t = base.student[..., :V], base.teacher[..., :V]
    tok = torch.randint(0, V, (B, T), dtype=torch.int32, device=DEV)
    win = torch.tensor([5, 3], dtype=torch.int32, device=DEV)
    grad = torch.full((B, T, ld_grad), 3.0, dtype=torch.bfloat16, device=DEV)
    got = api.adwin_opd_kl_fwd_bwd(s, t, tok, win, None, grad=grad[..., :V], flags=PATHS[path])
    torch.cuda.synchronize()
    api.raise_on_dev_status(got.dev_status)
    ref = O.opd_kl_fwd_bwd(synth.bits_for_oracle(s.contiguous()), synth.bits_for_oracle(t.contiguous()),
                           tok.cpu().numpy(), win.cpu().numpy(), None)
    mask = P.processed_mask(win.cpu().numpy(), np.array([T, T]), T)
    P.check_scalars(got, ref, 2e-3, mask)
    g = grad.double().cpu().numpy()
    P.check_grad_rows(g[..., :V][mask], ref["grad"][mask], 2e-3, store=2.0 ** -8)
    assert (g[..., V:] == 3.0).all() and (g[~mask] == 3.0).all()


def test_arrays_that_start_off_a_16_byte_boundary():
    """Student, teacher and gradient as views that begin two bytes into a piece, and the teacher at
    another offset than the student."""
    B, T, V = 2, 3, 1000
    base = synth.make_batch(2, device=DEV, B=B, T=T, V=V)
    n = B * T * V
    for off_s, off_t, off_g in ((1, 1, 1), (0, 1, 0), (3, 3, 0)):
        def view(x, off):
            buf = torch.zeros(n + 8, dtype=torch.bfloat16, device=DEV)
            v = buf[off:off + n].view(B, T, V)
            v.copy_(x)
            return v
        s, t = view(base.student, off_s), view(base.teacher, off_t)
        batch = synth.Batch(s, t, base.tokens, torch.tensor([3, 2], dtype=torch.int32, device=DEV),
                            base.rollout_len, 2)
        run_and_check(batch, grad_dtype=None)
        grad = view(torch.zeros_like(base.student), off_g)
        got = api.adwin_opd_kl_fwd_bwd(s, t, batch.tokens, batch.window, batch.rollout_len, grad=grad)
        torch.cuda.synchronize()
        api.raise_on_dev_status(got.dev_status)
        ref = P.oracle_batch(batch)
        mask = P.processed_mask([3, 2], batch.rollout_len.cpu().numpy(), T)
        P.check_grad_rows(grad.double().cpu().numpy()[mask], ref["grad"][mask], 2e-3, store=2.0 ** -8)


@pytest.mark.parametrize("B", [1, 3, 8, 9, 64, 65])
@pytest.mark.parametrize("K", [1, 6, 7, 8, 20])
def test_reductions_over_batch_and_candidate_counts(B, K):
    """One cluster up to 64 sequences, two launches beyond; eight prefix lengths per pass over a
    sequence (the rollout, the candidates, the window): counts on both sides of each line."""
    T = 700
    rng = np.random.default_rng(100 * B + K)
    kl, c, q = (rng.random((B, T), dtype=np.float32) for _ in range(3))
    r = rng.integers(0, T + 1, B).astype(np.int32)
    w = rng.integers(0, T + 1, B).astype(np.int32)
    cand = rng.permutation(np.arange(1, K + 1) * (T // K)).astype(np.int32)
    dev = [torch.from_numpy(x).to(DEV) for x in (kl, c, q, w, r, cand)]
    seq, tot = api.adwin_window_reduce(*dev[:5])
    al = api.adwin_probe_align(*dev)
    torch.cuda.synchronize()
    e = np.minimum(w, r)
    ref = np.array([[x[b, :e[b]].astype(np.float64).sum() for x in (kl, c, q)] + [e[b]] for b in range(B)])
    np.testing.assert_allclose(seq.cpu().numpy(), ref, rtol=1e-12)
    np.testing.assert_allclose(tot.cpu().numpy(), ref.sum(axis=0), rtol=1e-12)
    want = O.probe_align(kl, c, q, w, r, cand, math.sqrt(2) / 2)
    np.testing.assert_allclose(al.seq_stats.cpu().numpy(), want["seq_stats"], rtol=1e-12, atol=1e-12)
    np.testing.assert_allclose(al.seq_full.cpu().numpy(), want["seq_full"], rtol=1e-12, atol=1e-12)
    np.testing.assert_allclose(al.batch_stats.cpu().numpy(), want["batch_stats"], rtol=1e-12)
    assert int(al.L_next.item()) == want["L_next"] and int(al.flags.item()) == want["flags"]


def test_status_word_collects_or_starts_fresh():
    batch = synth.make_batch(2, device=DEV, B=2, T=6, V=4096)
    batch.tokens[0, 1] = -1
    args = (batch.student, batch.teacher, batch.tokens, batch.window, batch.rollout_len)
    for flags, start, want in ((0, 1 << 20, (1 << 20) | api.DEV_TOKEN_RANGE),
                               (api.STATUS_INIT, 1 << 20, api.DEV_TOKEN_RANGE)):
        status = torch.full((1,), start, dtype=torch.int32, device=DEV)
        api.adwin_opd_kl_fwd_bwd(*args, flags=flags | api.RANGE_FULL, dev_status=status)
        assert int(status.item()) == want
    batch.rollout_len[1] = 7                                     # longer than T
    o = api.adwin_opd_kl_fwd_bwd(*args, flags=api.RANGE_FULL)
    assert int(o.dev_status.item()) == api.DEV_TOKEN_RANGE | api.DEV_WINDOW


# The longest bf16 rows that the row kernel's shapes take (64, 128, 256 threads; 512 threads with one, two and four CTAs
# per row; half as many entries of fp32), and how many rows of them a call has to be for so that the shape goes by the
# length alone.  The sampled-token estimator keeps the student alone: twice as much on 512 threads.  Rows off the lines
# may lie in as much as 63 entries more (31 of fp32) than they have; bf16 rows of whole pieces up to 14 336 do not.
SHAPE_ENDS = ((6144, 298), (28672, 298), (57344, 150), (114688, 76), (229376, 38), (458752, 2), (237568, 76), (475136, 38),
              (950272, 2))


@pytest.mark.parametrize("in_dt,V,rows", [(2, v, 12) for v in (3584, 3592, 10240, 17920, 25600, 36000, 50688, 58880, 70001,
                                                               101376, 117760, 202752)] +
                         [(1, v, 12) for v in (1792, 5119, 33003, 50689, 58900, 101373, 118001)] +
                         [(2, v + more, rows) for v, rows in SHAPE_ENDS for more in (-63, -61, 0, 8, 64)] +
                         [(1, v // 2 + more, rows) for v, rows in SHAPE_ENDS for more in (-31, -29, 0, 4)])
def test_rows_held_by_one_cta_and_by_clusters(in_dt, V, rows):
    """The row kernel's shapes: rows of a few hundred pieces, rows that fill a CTA's shared memory and
    run over into tensor memory, rows split over two and four CTAs; at the end of every shape rows that
    fill it and rows of one more piece, on and off the lines (the last of each estimator go to the staged kernel); a
    sampled token in every slice, and rows whose token is far below the maximum (summed again from the
    copy on chip).  Few rows of a call have a gradient, whatever it is for."""
    T = max(6, rows // 2)
    batch = synth.make_batch(in_dt, device=DEV, B=2, T=T, V=V)
    batch.window = torch.tensor([6, 3], dtype=torch.int32, device=DEV)
    batch.rollout_len = torch.tensor([6, 6], dtype=torch.int32, device=DEV)
    for t, y in enumerate((0, V // 4 + 1, V // 2 + 1, 3 * V // 4 + 1, V - 1)):
        batch.tokens[0, t] = y
    for b, t in ((0, 1), (0, 4), (1, 2)):     # (both policies, see the test of odd rows)
        y = int(batch.tokens[b, t])
        batch.student[b, t, y] = batch.student[b, t].float().max() - 100.0
        batch.teacher[b, t, y] = batch.teacher[b, t].float().max() - 100.0
    # z - u of one at the token: the sampled gradient is proportional to c, whose error of about 3e-7 (a
    # difference of fp32 logits and logarithms) is within 1e-5 of it only for |c| > 0.03
    y = batch.tokens.long()[..., None]
    batch.teacher.scatter_(2, y, batch.student.gather(2, y) - 1.0)
    g_dt = torch.float32 if in_dt == 1 else torch.bfloat16
    for mode in (api.GRAD_FULL_KL, api.GRAD_SAMPLED):
        run_and_check(batch, grad_dtype=g_dt, grad_mode=mode)
    run_and_check(batch, grad_dtype=g_dt, flags=api.RANGE_FULL)


# Several rows for every CTA of a launch, so that a row's second sweep runs beside the next row's first and
# the ring of kept pieces turns over: the longest rows of each shape (bf16; half of that fp32), whose ring has no room
# beside a row, and rows that leave one and two groups; rows of whole lines, of whole pieces and rows that start anywhere
# in one; the first of a cluster of two and of four.
@pytest.mark.parametrize("in_dt,V,rows", [(2, 4099, 2500), (2, 4096, 2500), (2, 28665, 1250), (2, 57341, 620), (2, 57344, 620),
                                          (2, 5000, 2500), (2, 6081, 2500), (2, 6144, 2500), (2, 14328, 2500), (2, 14344, 2500),
                                          (2, 28609, 1250), (2, 28672, 1250), (2, 57281, 620), (2, 114625, 310), (2, 114688, 310),
                                          (2, 196609, 160), (2, 212992, 160), (2, 229376, 160), (2, 393217, 80), (2, 425984, 80),
                                          (2, 458752, 80), (2, 237568, 310), (2, 475136, 160), (2, 950272, 80), (1, 3072, 2500),
                                          (1, 28672, 620), (1, 57344, 310), (1, 114688, 160), (1, 229376, 80),
                                          (2, 114681, 310), (2, 114752, 170), (2, 262144, 80), (1, 2050, 2500),
                                          (1, 14331, 1250), (1, 57341, 310), (1, 57349, 170)])
def test_rows_one_after_another(in_dt, V, rows):
    batch = synth.make_batch(in_dt, device=DEV, B=2, T=rows // 2, V=V)
    batch.window = torch.tensor([rows // 2, rows // 2 - 3], dtype=torch.int32, device=DEV)
    check_rows_one_after_another(batch)


def check_rows_one_after_another(batch, second=False):
    # sampled tokens in the partial pieces of a row and between; every seventh far below the maximum, which
    # sums the row again.  z - u of eight there: c is a difference of fp32 logits and logarithms of up to 16, off by
    # 2e-6, and twice that over |c| has to stay below 1e-4 (the norm of the sampled gradient)
    V = batch.shape[2]
    for k, y in enumerate((0, 3, V - 1, V - 4, V // 2)):
        batch.tokens[:, k::6] = y
    y = batch.tokens.long()[..., None]
    z = batch.student.gather(2, y)
    z[:, ::7] = batch.student[:, ::7].float().amax(2, keepdim=True).to(z.dtype) - 100.0
    batch.student.scatter_(2, y, z)
    batch.teacher.scatter_(2, y, z - 8.0)
    if second:
        # In a short row the peak may have nearly all of the mass, and a gradient that is the rounding of z - u less its mean.
        # So an entry beside the peak gets 1/21 of its mass, at z - u = -16, eight and more from the peak's: 2^-24 * 16 a
        # rounding against 8 / 21 and more, 5e-6 of the norm, of which its tolerance of 1e-4 bears twenty.
        z, at = batch.student.max(2, keepdim=True)
        at = torch.where((at + 1) % V == y, at + 2, at + 1) % V
        z = (z.float() - 3.0).to(z.dtype)
        batch.student.scatter_(2, at, z)
        batch.teacher.scatter_(2, at, z + 16.0)
    g_dt = batch.student.dtype
    run_and_check(batch, grad_dtype=g_dt, grad_mode=api.GRAD_FULL_KL)
    run_and_check(batch, grad_dtype=g_dt, grad_mode=api.GRAD_SAMPLED)


# Rows of one and two groups of loads, several for every CTA of the 64-thread shape (1184 CTAs on 148 SMs): the
# loads run two rows ahead of the row whose sums are out, and so do its metadata.  Two long sequences, and
# many so short that a CTA's next row is several sequences on.
@pytest.mark.parametrize("in_dt,V", [(2, 33), (2, 64), (2, 961), (2, 1024), (2, 1032), (1, 33), (1, 481), (1, 512)])
@pytest.mark.parametrize("B,T", [(2, 3500), (900, 16)])
def test_short_rows_one_after_another(in_dt, V, B, T):
    batch = synth.make_batch(in_dt, device=DEV, B=B, T=T, V=V)
    rng = np.random.default_rng(V + B)
    batch.window = torch.from_numpy(rng.integers(T - 3 if B == 2 else 1, T + 1, B).astype(np.int32)).to(DEV)
    batch.rollout_len[:] = T
    check_rows_one_after_another(batch, second=True)


# Calls with a CTA or cluster for every row take wider shapes than the row's length alone asks for: at the piece
# counts where each is first taken (512, 1024 and 3584 pieces) and one piece below, on and off the lines, with as many
# rows as clusters of four and of two and one or two CTAs per SM hold at a time, and a few more than that.
@pytest.mark.parametrize("in_dt,V", [(2, 4088), (2, 4096), (2, 8184), (2, 8192), (2, 8131), (2, 28664), (2, 28672), (2, 50257),
                                     (1, 2048), (1, 4095), (1, 14332), (1, 14336), (1, 20001)])
@pytest.mark.parametrize("rows", [33, 37, 70, 78, 148, 150, 296, 298])
def test_calls_of_few_rows(in_dt, V, rows):
    batch = synth.make_batch(in_dt, device=DEV, B=1, T=rows, V=V)
    batch.window[:] = rows
    batch.rollout_len[:] = rows
    check_rows_one_after_another(batch)


@pytest.mark.parametrize("in_dt,V", [(2, 4095), (2, 4096), (2, 4104), (2, 20001), (1, 2047), (1, 2052), (1, 9001)])
@pytest.mark.parametrize("mode", [api.GRAD_FULL_KL, api.GRAD_SAMPLED])
def test_read_only_rows_that_outgrow_their_first_entries(in_dt, V, mode):
    """Rows without gradient are summed against the maximum of each thread's first entries: rows that
    rise after them by less than the sums bear, and by more (summed once more against running
    maxima), in the student, the teacher and both; row lengths around one whole group of loads."""
    batch = synth.make_batch(in_dt, device=DEV, B=2, T=5, V=V)
    batch.window = torch.tensor([5, 4], dtype=torch.int32, device=DEV)
    part = 4 * 128 * (4 if in_dt == 1 else 8)       # entries of the first group of a row
    for t, (rise_s, rise_t) in enumerate(((20.0, 20.0), (60.0, 0.0), (0.0, 60.0), (90.0, 80.0))):
        batch.student[0, t, :part] -= rise_s
        batch.teacher[0, t, :part] -= rise_t
        for x in (batch.student, batch.teacher):    # keep the sampled token near the maximum
            x[0, t, int(batch.tokens[0, t])] = x[0, t].float().max() - 1.0
    run_and_check(batch, grad_dtype=None, grad_mode=mode)
    run_and_check(batch, grad_dtype=None, grad_mode=mode, flags=api.RANGE_FULL)


@pytest.mark.parametrize("in_dt,V,rows", [(2, 120000, 20), (2, 120001, 20), (2, 32003, 300), (1, 33, 6), (1, 93534, 20),
                                          (1, 150001, 160)])
def test_read_only_rows_split_over_a_cluster(in_dt, V, rows):
    """Calls of few rows, read only: four, two and one CTAs per row (the lengths leave some clusters
    without a row), rows off 16-byte boundaries, the last CTA's share shorter than the others'."""
    batch = synth.make_batch(in_dt, device=DEV, B=2, T=rows // 2 + 1, V=V)
    batch.window = torch.tensor([min(rows // 2, 8), 3], dtype=torch.int32, device=DEV)
    for t, y in enumerate((0, V // 4 + 1, V - 1)):
        batch.tokens[1, t] = y
    for mode in (api.GRAD_FULL_KL, api.GRAD_SAMPLED):
        run_and_check(batch, grad_dtype=None, grad_mode=mode)


# (clusters of four for few rows; 151 936 entries also clusters of two, several rows each, more of them than the GPU
# holds at a time)
@pytest.mark.parametrize("V,rows", [(4096, 40), (40000, 24), (151936, 20), (151936, 180)])
def test_launches_that_overlap_their_predecessor(V, rows):
    """Kernels of a call are set up while the one before drains: calls in a row over the same buffers and
    workspace, on two streams and replayed from a graph, leave the bits that separate calls leave."""
    batches = [synth.make_batch(2, device=DEV, seed=s, B=2, T=rows // 2, V=V) for s in (1, 2)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]

    def call(batch, o=None, ws=None):
        grad = o.grad if o else torch.zeros_like(batch.student)
        o = api.adwin_opd_kl_fwd_bwd(batch.student, batch.teacher, batch.tokens, batch.window,
                                     batch.rollout_len, grad=grad, out=o, workspace=ws)
        return o, api.adwin_window_reduce(o.kl, o.logratio, o.gsq, batch.window, batch.rollout_len)

    def bits(o, red):
        return [x.clone() for x in (o.kl, o.logratio, o.gsq, o.grad, *red)]

    want = []
    for b in batches:
        want.append(bits(*call(b)))
        torch.cuda.synchronize()
    got = [[], []]
    for i, s in enumerate(streams):
        ws = torch.empty(1 << 16, dtype=torch.uint8, device=DEV)
        with torch.cuda.stream(s):
            s.wait_stream(torch.cuda.default_stream())
            o = None
            for n in range(12):           # the other batch first: its results are overwritten
                o, red = call(batches[(n + i + 1) % 2], o, ws)
            got[i] = bits(o, red)
    torch.cuda.synchronize()
    for i in (0, 1):
        assert all(torch.equal(a, b) for a, b in zip(got[i], want[i]))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        o, red = call(batches[0])
        o, red = call(batches[1], o)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(bits(o, red), want[1]))


def test_two_threads_with_vocabularies_of_their_own():
    """Two host threads that call with different row lengths (the same kernel, different shared memory
    per launch), each on its own stream: no launch may fail for what the other thread set up.  (Calls
    of the library itself, back to back: it runs without the interpreter's lock.)"""
    calls = {}
    for V in (30000, 50000):
        batch = synth.make_batch(2, device=DEV, seed=V, B=1, T=2, V=V)
        batch.window = torch.tensor([2], dtype=torch.int32, device=DEV)
        out = api.adwin_opd_kl_fwd_bwd(batch.student, batch.teacher, batch.tokens, batch.window,
                                       batch.rollout_len, grad=torch.zeros_like(batch.student))
        stream = torch.cuda.Stream()
        args = (batch.student.data_ptr(), batch.teacher.data_ptr(), api.BF16, 1, 2, V, V,
                batch.tokens.data_ptr(), batch.window.data_ptr(), batch.rollout_len.data_ptr(), 1.0,
                api.GRAD_FULL_KL, 0, out.grad.data_ptr(), api.BF16, V, out.kl.data_ptr(),
                out.logratio.data_ptr(), out.gsq.data_ptr(), None, None, out.workspace.data_ptr(),
                out.workspace.numel(), out.dev_status.data_ptr(), stream.cuda_stream)
        calls[V] = (batch, out, stream, args, out.grad.clone())
    torch.cuda.synchronize()
    failed = {}

    def work(V):
        torch.cuda.set_device(0)
        call, args = api.lib().adwin_opd_kl_fwd_bwd, calls[V][3]
        failed[V] = sum(call(*args) != api.OK for _ in range(20000))

    threads = [threading.Thread(target=work, args=(V,)) for V in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert failed == {30000: 0, 50000: 0}
    for batch, out, _, _, want in calls.values():
        api.raise_on_dev_status(out.dev_status)
        assert torch.equal(out.grad, want)


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("in_dt", [1, 2])
@pytest.mark.parametrize("V,masked,at", [(150, 3, "end"), (1001, 64, "end"), (1003, 293, "end"), (4099, 7, "start"),
                                         (4096, 293, "start"), (50257, 300, "end")])
@pytest.mark.parametrize("value", ["lowest", -1e30, -1e9])
def test_masked_vocabulary_entries(path, in_dt, V, masked, at, value):
    """Entries masked out in both policies, at either end of the vocabulary, so that some threads see
    nothing else (or nothing else first): they count for nothing, as in the oracle.  One row whose token
    is far below the maximum (summed against running maxima)."""
    batch = synth.make_batch(in_dt, device=DEV, B=2, T=4, V=V)
    batch.window = torch.tensor([4, 2], dtype=torch.int32, device=DEV)
    where = slice(V - masked, V) if at == "end" else slice(0, masked)
    value = torch.finfo(batch.student.dtype).min if value == "lowest" else value
    for x in (batch.student, batch.teacher):
        x[..., where] = value
    # (the token with the largest log-ratio: the sampled gradient's norm is c^2 times a constant, and c, a
    # difference of logits, is good to 1e-5, so that 1e-4 on the norm takes |c| > 0.2)
    batch.tokens[:] = (batch.student.float() - batch.teacher.float()).argmax(dim=2)
    y = int(batch.tokens[0, 2])
    batch.student[0, 2, y] = batch.student[0, 2].float().max() - 98.0
    batch.teacher[0, 2, y] = batch.teacher[0, 2].float().max() - 100.0
    g_dt = batch.student.dtype
    for mode in (api.GRAD_FULL_KL, api.GRAD_SAMPLED):
        for grad in (g_dt, None):
            run_and_check(batch, grad_dtype=grad, grad_mode=mode, flags=PATHS[path])


@pytest.mark.parametrize("in_dt,V", [(2, 4096), (2, 32000), (2, 50257), (2, 151936), (1, 20001)])
@pytest.mark.parametrize("rows", [6, 310])
def test_entries_that_only_the_teacher_masks(in_dt, V, rows):
    """Entries at -infinity in the teacher alone, where the student has mass: the divergence is infinite and so
    is the gradient (towards minus infinity, -p_k times it), with no entry of it undefined but the masked ones."""
    batch = synth.make_batch(in_dt, device=DEV, B=1, T=rows, V=V)
    batch.window[:] = batch.rollout_len[:] = rows
    batch.teacher[..., 100:140] = batch.student[..., 100:140] = float("-inf")
    batch.tokens[:] = batch.student.argmax(dim=2)
    batch.student[..., 100:140] = batch.student.float().amax(dim=2, keepdim=True) - 2.0
    grad = torch.zeros_like(batch.student)
    got = api.adwin_opd_kl_fwd_bwd(batch.student, batch.teacher, batch.tokens, batch.window, batch.rollout_len, grad=grad)
    torch.cuda.synchronize()
    assert (got.kl == float("inf")).all() and torch.isfinite(got.logratio).all()
    grad[..., 100:140] = float("-inf")
    assert (grad == float("-inf")).all()


@pytest.mark.parametrize("in_dt,V", [(2, 4096), (2, 4104), (2, 20001), (2, 120000), (1, 2052), (1, 9001)])
@pytest.mark.parametrize("mode", [api.GRAD_FULL_KL, api.GRAD_SAMPLED])
def test_read_only_rows_that_outgrow_first_entries_and_token(in_dt, V, mode):
    """Read-only sums refer to the maximum of a thread's first entries and the sampled token: rows in which
    both lie below the rest by less than the sums bear, and by more (summed once more against running
    maxima).  Both policies alike, so that z - u at the token stays small (its magnitude times 2^-24 is the
    error of every centred difference)."""
    batch = synth.make_batch(in_dt, device=DEV, B=2, T=4, V=V)
    batch.window = torch.tensor([4, 3], dtype=torch.int32, device=DEV)
    part = 4 * 128 * (4 if in_dt == 1 else 8)       # entries of the first group of a row
    for t, rise in enumerate((20.0, 60.0, 90.0)):
        for x in (batch.student, batch.teacher):
            x[0, t, :part] -= rise
    # inside the lowered part, z - u near one: the sampled norm is c^2 times a constant, so c must not be
    # near zero, and the one-sweep norm is centred on the token's z - u, whose distance from the others'
    # (3 standard deviations for the largest one) enters its error squared
    batch.tokens[:] = ((batch.student.float() - batch.teacher.float())[..., :part] - 1.0).abs().argmin(dim=2)
    run_and_check(batch, grad_dtype=None, grad_mode=mode)
    run_and_check(batch, grad_dtype=None, grad_mode=mode, flags=api.RANGE_FULL)


def test_read_only_precision_of_references_and_running_maxima():
    """kl and the log-ratio of a read-only row do not depend on the gradient mode, but the full-KL mode sums
    against references fixed early and the sampled mode against running maxima: the first may not be
    further from a 64-bit evaluation (10 % for the spread between two sets of 1100 rounding errors)."""
    batch = synth.make_batch(3, device=DEV, B=2, T=550)
    batch.rollout_len[:] = 550
    args = (batch.student, batch.teacher, batch.tokens, batch.window, batch.rollout_len)
    z, u = batch.student.flatten(0, 1), batch.teacher.flatten(0, 1)
    y = batch.tokens.flatten().long()[:, None]
    err = {}
    for mode in (api.GRAD_FULL_KL, api.GRAD_SAMPLED):
        got = api.adwin_opd_kl_fwd_bwd(*args, grad_mode=mode, flags=api.RANGE_FULL)
        kl, c = got.kl.double().flatten(), got.logratio.double().flatten()
        sums = torch.zeros(2, dtype=torch.float64, device=DEV)
        for r in range(0, len(y), 50):
            d = torch.log_softmax(z[r:r + 50].double(), 1)
            p = d.exp()
            d -= torch.log_softmax(u[r:r + 50].double(), 1)
            sums[0] += ((p * d).sum(1) - kl[r:r + 50]).square().sum()
            sums[1] += (d.gather(1, y[r:r + 50])[:, 0] - c[r:r + 50]).square().sum()
        err[mode] = sums.sqrt()
    assert (err[api.GRAD_FULL_KL] <= 1.1 * err[api.GRAD_SAMPLED]).all(), err


def test_precision_of_rows_with_gradient():
    """The row kernel adds a row up over more entries per thread than the staged kernel, and about the sampled token's
    z - u: its scalars may not be further from a 64-bit evaluation for it, with tokens drawn uniformly, which are
    poor centres (10 % for the spread between two sets of 2048 rounding errors)."""
    T, V = 2048, 50248
    z, u = (torch.zeros((1, T, V), dtype=torch.bfloat16, device=DEV) for _ in range(2))
    tokens = torch.zeros((1, T), dtype=torch.int32, device=DEV)
    gen = torch.Generator(device=DEV).manual_seed(7)
    synth.fill_sequence(z[0], u[0], tokens[0], s_std=2.0, mix=1.0, t_std=1.0, spike_p=0.0, tokens="uniform", gen=gen)
    window = torch.tensor([T], dtype=torch.int32, device=DEV)
    grad = torch.zeros_like(z)
    got = {flags: api.adwin_opd_kl_fwd_bwd(z, u, tokens, window, window, flags=flags, grad=grad)
           for flags in (0, api.FORCE_STAGED)}
    sums = {flags: torch.zeros(3, dtype=torch.float64, device=DEV) for flags in got}
    for r in range(0, T, 64):
        rows = slice(r, r + 64)
        d = torch.log_softmax(z[0, rows].double(), 1)
        p = d.exp()
        d -= torch.log_softmax(u[0, rows].double(), 1)
        kl = (p * d).sum(1)
        gsq = (p * (d - kl[:, None])).square().sum(1)
        c = d.gather(1, tokens[0, rows].long()[:, None])[:, 0]
        for flags, o in got.items():
            sums[flags] += torch.stack([((o.kl[0, rows].double() - kl) / kl).square().sum(),
                                        (o.logratio[0, rows].double() - c).square().sum(),
                                        ((o.gsq[0, rows].double() - gsq) / gsq).square().sum()])
    assert (sums[0].sqrt() <= 1.1 * sums[api.FORCE_STAGED].sqrt()).all(), sums
