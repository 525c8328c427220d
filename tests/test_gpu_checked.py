"""The bounds-checked build flavour (-DADWIN_CHECKED) on the small and odd-shaped parity cases.

A memory checker is not available where these tests run, so the library has a flavour in which
every index the kernels form by hand is tested before the access and a violation raises
ADWIN_DEV_BOUNDS instead of touching memory.  Here the cases with ragged tails, degenerate
windows, padded strides and the overflow fallback run through that flavour: the status word must
stay clear (the helpers raise on any bit) and the results must equal the ordinary build's bit for
bit.
"""
import pytest
import torch

from paper_2605_28396_b200 import api, build, synth
from tests import test_gpu_lmhead as L
from tests import test_gpu_parity as G

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture()
def checked_library():
    path = build.build(checked=True)
    api.use_library(path)
    try:
        yield path
    finally:
        api.use_library(None)


@pytest.mark.parametrize("V", [1, 7, 9, 1001, 4100, 65537])
def test_odd_vocabularies(checked_library, V):
    G.test_odd_vocab_sizes(V)


@pytest.mark.parametrize("path", G.PATHS)
def test_degenerate_windows_padded_strides_and_overflow_fallback(checked_library, path):
    G.test_degenerate_windows(path)
    G.test_padded_row_stride(path)
    G.test_range_full_with_gradient_inside_window_only(path)
    G.test_sampled_token_far_below_the_row_maximum(path, 2, torch.bfloat16)
    G.test_config3_reduced_T_full_vocab(path, api.GRAD_FULL_KL)


def test_status_word_collects_or_starts_fresh(checked_library):
    G.test_status_word_collects_or_starts_fresh()


def test_teacher_drift_and_return_to_go(checked_library):
    from tests import test_gpu_drift as D
    from tests import test_gpu_rtg as R
    for name in dir(D):
        if name.startswith("test_") and "full_size" not in name:
            fn = getattr(D, name)
            if fn.__code__.co_argcount == 0:
                fn()
    for name in dir(R):
        if name.startswith("test_") and "full_size" not in name:
            fn = getattr(R, name)
            if fn.__code__.co_argcount == 0:
                fn()


@pytest.mark.parametrize("path", G.PATHS)
def test_rows_off_16_byte_boundaries(checked_library, path):
    for V in (33, 1001, 50257):
        for in_dt, g_dt in ((1, torch.float32), (2, torch.bfloat16), (2, None)):
            G.test_rows_that_start_and_end_off_16_byte_boundaries(path, in_dt, g_dt, V)
    for V, ld, ld_grad in ((1001, 1008, 1024), (1001, 1003, 1005), (12000, 12004, 12004)):
        G.test_odd_rows_at_a_padded_stride(path, V, ld, ld_grad)
    G.test_arrays_that_start_off_a_16_byte_boundary()


@pytest.mark.parametrize("v,rows", G.SHAPE_ENDS)
def test_ends_of_the_row_kernels_shapes(checked_library, v, rows):
    for V in (v - 63, v - 61, v, v + 8):
        G.test_rows_held_by_one_cta_and_by_clusters(2, V, rows)
    for V in (v // 2 - 31, v // 2, v // 2 + 4):
        G.test_rows_held_by_one_cta_and_by_clusters(1, V, rows)


@pytest.mark.parametrize("in_dt,V,rows", [(2, 4099, 2500), (2, 6144, 2500), (2, 28609, 1250), (2, 57281, 620), (2, 114625, 310),
                                          (2, 151936, 160), (2, 229376, 160), (2, 262144, 80), (2, 458752, 80), (1, 2050, 2500),
                                          (1, 57341, 310)])
def test_rows_one_after_another(checked_library, in_dt, V, rows):
    G.test_rows_one_after_another(in_dt, V, rows)


@pytest.mark.parametrize("in_dt,V,rows", [(2, 8192, 33), (2, 28672, 70), (2, 50257, 37), (2, 50257, 148), (1, 4095, 296)])
def test_calls_of_few_rows(checked_library, in_dt, V, rows):
    G.test_calls_of_few_rows(in_dt, V, rows)


@pytest.mark.parametrize("in_dt,V", [(2, 33), (2, 961), (2, 1024), (2, 1032), (1, 481)])
def test_short_rows_one_after_another(checked_library, in_dt, V):
    G.test_short_rows_one_after_another(in_dt, V, 2, 3500)
    G.test_short_rows_one_after_another(in_dt, V, 900, 16)


def test_read_only_rows(checked_library):
    for in_dt, V, rows in ((2, 120001, 20), (2, 32003, 300), (1, 93534, 20)):
        G.test_read_only_rows_split_over_a_cluster(in_dt, V, rows)
    for in_dt, V in ((2, 4104), (2, 20001), (1, 2052)):
        for mode in (api.GRAD_FULL_KL, api.GRAD_SAMPLED):
            G.test_read_only_rows_that_outgrow_their_first_entries(in_dt, V, mode)


def test_fused_lm_head_small_and_ragged(checked_library):
    L.test_small_case_modes_and_flags(api.GRAD_FULL_KL, api.RANGE_FULL)
    for windows in ([127], [60, 69, 0, 128], [257, 3]):
        L.test_rows_packed_across_sequences_at_tile_edges(windows)
    L.test_ragged_vocabulary_and_hidden_sizes(1000, 72, 200)
    L.test_all_windows_empty_gives_zero_gradients()


def test_results_equal_the_ordinary_build_bit_for_bit():
    batch = synth.make_batch(3, device=DEV, B=4, T=48)
    lm = synth.make_lmhead_batch(DEV, B=2, T=150, V=1000, d_s=72, d_t=200, w_std=0.15)
    outs = []
    for checked in (False, True):
        api.use_library(build.build(checked=True) if checked else None)
        try:
            grad = torch.zeros(batch.shape, dtype=torch.bfloat16, device=DEV)
            a = api.adwin_opd_kl_fwd_bwd(batch.student, batch.teacher, batch.tokens, batch.window,
                                         batch.rollout_len, grad=grad)
            b = api.adwin_opd_kl_fwd_bwd(batch.student, batch.teacher, batch.tokens, batch.window,
                                         batch.rollout_len, flags=api.RANGE_FULL)
            dW = torch.zeros((1000, 72), dtype=torch.float32, device=DEV)
            c = api.adwin_opd_kl_lmhead_fwd_bwd(lm.hidden_student, lm.w_student, lm.hidden_teacher,
                                                lm.w_teacher, lm.tokens, lm.window, lm.rollout_len,
                                                grad_w=dW)
            torch.cuda.synchronize()
            for o in (a, b, c):
                api.raise_on_dev_status(o.dev_status)
            outs.append((grad, a.kl, a.gsq, b.kl, b.gsq, dW, c.kl, c.gsq))
        finally:
            api.use_library(None)
    for x, y in zip(*outs):
        assert torch.equal(x, y)
