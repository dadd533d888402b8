"""GPU parity of the CUDA eviction pass against the float64 oracle.

Every test calls the library through the C ABI (via the ctypes binding) and
compares with ``oracle.oracle_unit`` on the same bytes (the oracle reads the
device tensors back exactly). Small cases compare every unit and every
intermediate; the five evaluation configurations run at full size, in the
launch configuration bench.py times, with sampled units checked against the
oracle and size-independent properties checked on every unit.
"""

from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import JacapParams, oracle_unit
from paper_2609_08131_gb300 import jacap_params
from paper_2609_08131_gb300.api import Cache, Evictor, evict
from paper_2609_08131_gb300.workloads import Workload, config, generate, unit_arrays

from oracle_pool import run_units
from parity import assert_rows_bitwise, assert_scores_close, assert_selection, gpu_selection_properties

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def make_cache(t, wl):
    return Cache(t.q_win, t.k, t.v, t.cu_seqlens, t.seqlens, wl.num_q_heads)


def check_unit(ev, t, wl, params, s, layer, g, check_w=True):
    q, K, V = unit_arrays(t, wl.num_q_heads, s, layer, g)
    ora = oracle_unit(q, K, V, ev.budget, JacapParams(tau=params.tau, weight_div_dk=bool(params.weight_div_dk),
                                                       cov_unbiased=bool(params.cov_unbiased),
                                                       linear_weighting=bool(params.linear_weighting),
                                                       full_covariance=bool(params.full_covariance)))
    cu = t.cu_seqlens.cpu().tolist()
    a, b = cu[s], cu[s + 1]
    n = b - a
    gs = ev.scores[layer, g, a:b].double().cpu().numpy()
    if check_w:
        gw = ev.intermediates()["weights"][layer, g, a:b].double().cpu().numpy()
        assert_scores_close(gw, ora["w"], "weights")
    assert_scores_close(gs, ora["scores"])
    gidx = ev.idx[layer, g, s].cpu().numpy()
    assert_selection(gidx, n, ev.budget, ora["scores"], ora["idx"])
    kept = min(n, ev.budget)
    sel = torch.as_tensor(gidx[:kept], dtype=torch.long, device=t.k.device)
    assert_rows_bitwise(t.k[layer, g, a:b][sel], ev.k_out[layer, g, s, :kept])
    assert_rows_bitwise(t.v[layer, g, a:b][sel], ev.v_out[layer, g, s, :kept])
    if kept < ev.budget:
        assert bool((ev.k_out[layer, g, s, kept:] == 0).all()) and bool((ev.v_out[layer, g, s, kept:] == 0).all())
    return ora


SMALL = {
    # name: (workload, params)
    "bf16_gqa4_ragged_tails": (Workload("t", 2, 8, 2, (1000, 300, 129), 16, 64, seed=11), jacap_params()),
    "bf16_mha_tau1": (Workload("t", 1, 4, 4, (777,), 8, 100, seed=12), jacap_params(tau=1.0)),
    "bf16_gqa2_peaky_tiny_seq": (Workload("t", 1, 4, 2, (500, 1, 2), 16, 32, seed=13), jacap_params(tau=0.3)),
    "bf16_gqa8_one_past_tile": (Workload("t", 1, 8, 1, (4101,), 32, 256, seed=14), jacap_params()),
    "bf16_sinks_unbiased_nodiv": (Workload("t", 1, 8, 2, (2048, 1500), 64, 200, seed=15, sink_tokens=4,
                                           sink_scale=4.0), jacap_params(tau=2.0, weight_div_dk=0, cov_unbiased=1)),
    "f32_outlier_mha": (Workload("t", 1, 4, 4, (1500, 2049), 32, 128, dtype="f32", dist="outlier", seed=16,
                                 outlier_channels=4, outlier_scale=8.0), jacap_params()),
    "f32_gqa4_peaky": (Workload("t", 2, 8, 2, (600, 130), 8, 50, dtype="f32", seed=17), jacap_params(tau=0.5)),
    "bf16_budget_exceeds_all": (Workload("t", 1, 4, 2, (100, 257), 8, 300, seed=18), jacap_params()),
    "bf16_gqa4_linear_weighting": (Workload("t", 2, 8, 2, (1500, 700), 16, 128, seed=19),
                                   jacap_params(linear_weighting=1)),
    # full-covariance kappa (App. B.2) on the tensor-core kernel
    "bf16_gqa4_full_cov_w32": (Workload("t", 2, 8, 2, (1300, 300), 32, 96, seed=22), jacap_params(full_covariance=1)),
    "bf16_gqa2_full_cov_w64_unbiased": (Workload("t", 1, 4, 2, (900, 129), 64, 64, seed=23),
                                        jacap_params(full_covariance=1, cov_unbiased=1, tau=2.0)),
    "bf16_gqa8_full_cov_w8": (Workload("t", 1, 8, 1, (700,), 8, 64, seed=24), jacap_params(full_covariance=1)),
    "bf16_gqa8_full_cov_w16": (Workload("t", 1, 16, 2, (1100, 40), 16, 64, seed=27), jacap_params(full_covariance=1)),
    # 8 centred queries per group: the image's zero padding rows
    "bf16_mha_full_cov_w8_tau1": (Workload("t", 2, 4, 4, (650, 3), 8, 32, seed=28),
                                  jacap_params(full_covariance=1, tau=1.0)),
    # ... and the CUDA-core kernel (w = 24; float32)
    "bf16_gqa4_full_cov_w24": (Workload("t", 1, 8, 2, (600, 200), 24, 64, seed=25), jacap_params(full_covariance=1)),
    "f32_gqa2_full_cov": (Workload("t", 1, 4, 2, (500,), 16, 32, dtype="f32", seed=26),
                          jacap_params(full_covariance=1)),
    "f32_mha_linear_weighting": (Workload("t", 1, 4, 4, (900,), 8, 64, dtype="f32", seed=20),
                                 jacap_params(linear_weighting=1, cov_unbiased=1)),
    # GQA ratios of the paper's other models: Qwen3-14B (40 q / 8 kv heads,
    # G = 5) and Nemotron-7B (28 q / 4 kv heads, G = 7), plus G = 3 and 6.
    # Odd G gives 8-byte aligned logits/kappa rows and 4-byte aligned kappa halves.
    "bf16_gqa5_qwen3_14b_heads": (Workload("t", 2, 40, 8, (1200, 333), 32, 128, seed=41), jacap_params()),
    "bf16_gqa7_nemotron_heads": (Workload("t", 2, 28, 4, (1500, 129), 32, 128, seed=42), jacap_params()),
    "bf16_gqa3_tau1": (Workload("t", 1, 6, 2, (800, 257), 16, 64, seed=43), jacap_params(tau=1.0)),
    "bf16_gqa6_unbiased": (Workload("t", 1, 12, 2, (700, 130), 16, 64, seed=44), jacap_params(cov_unbiased=1)),
    "bf16_gqa7_peaky_linear": (Workload("t", 1, 14, 2, (650, 3), 8, 40, seed=45), jacap_params(linear_weighting=1)),
    "f32_gqa5": (Workload("t", 1, 10, 2, (600, 77), 16, 64, dtype="f32", seed=46), jacap_params(tau=0.7)),
    "f32_gqa7": (Workload("t", 1, 14, 2, (500, 70), 8, 32, dtype="f32", seed=47), jacap_params()),
    # full covariance: tensor-core kernel with G w = 96, 80, 112 centred queries
    # (the last with a 32-row mu' image), CUDA-core kernel with G w = 192
    "bf16_gqa3_full_cov_w32": (Workload("t", 1, 6, 2, (900, 100), 32, 64, seed=48), jacap_params(full_covariance=1)),
    "bf16_gqa5_full_cov_w16": (Workload("t", 1, 10, 2, (700,), 16, 64, seed=49), jacap_params(full_covariance=1)),
    "bf16_gqa7_full_cov_w16": (Workload("t", 1, 14, 2, (640, 33), 16, 64, seed=50),
                               jacap_params(full_covariance=1, tau=2.0)),
    "bf16_gqa6_full_cov_w32_simt": (Workload("t", 1, 12, 2, (500,), 32, 64, seed=51),
                                    jacap_params(full_covariance=1)),
}


def with_schedule(p, schedule):
    return jacap_params(p.tau, p.weight_div_dk, p.ridge, p.cov_unbiased, p.linear_weighting, p.full_covariance,
                        schedule)


# every bf16 case under both schedules (separate kernels; the fused persistent
# launch); float32 caches always take the separate kernels
SMALL_RUNS = [(n, sch) for n in SMALL for sch in ((1, 2) if SMALL[n][0].dtype == "bf16" else (0,))]


@pytest.mark.parametrize("name,schedule", SMALL_RUNS, ids=[f"{n}-s{s}" for n, s in SMALL_RUNS])
def test_small_caches_every_unit(name, schedule):
    wl, params = SMALL[name]
    params = with_schedule(params, schedule)
    t = generate(wl, DEV)
    ev = evict(make_cache(t, wl), wl.budget, params)
    for s in range(len(wl.seqlens)):
        for layer in range(wl.num_layers):
            for g in range(wl.num_kv_heads):
                check_unit(ev, t, wl, params, s, layer, g)
    gpu_selection_properties(ev.scores, ev.idx, ev.kept, wl.seqlens, wl.budget)


@pytest.mark.parametrize("schedule", [1, 2])
def test_intermediates_match_the_oracle(schedule):
    wl = Workload("t", 2, 8, 2, (900, 333), 16, 64, seed=21)
    params = jacap_params(tau=1.5, schedule=schedule)
    t = generate(wl, DEV)
    ev = evict(make_cache(t, wl), wl.budget, params)
    inter = ev.intermediates()
    G = wl.num_q_heads // wl.num_kv_heads
    import oracle.jacap_oracle as O
    for s in range(2):
        for layer in range(2):
            for g in range(2):
                q, K, V = unit_arrays(t, wl.num_q_heads, s, layer, g)
                for j in range(G):
                    mu, lam = O.window_stats(q[j])
                    h = g * G + j
                    np.testing.assert_allclose(inter["mu_scaled"][s, layer, h].double().cpu().numpy(),
                                               mu / (params.tau * np.sqrt(128)), rtol=1e-5, atol=1e-7)
                    np.testing.assert_allclose(inter["lambda"][s, layer, h].double().cpu().numpy(), lam,
                                               rtol=1e-5, atol=1e-7)
                w = O.unit_weights(K, q, JacapParams(tau=params.tau))
                A = O.capacity_matrix(V, w)
                G_ora = A - np.eye(128)
                G_gpu = inter["gram"][layer, g, s].double().cpu().numpy()
                np.testing.assert_allclose(G_gpu, G_ora, rtol=1e-4, atol=1e-5 * np.abs(G_ora).max())
                Lc = np.linalg.cholesky(A)
                Minv = np.linalg.inv(Lc)
                np.testing.assert_allclose(inter["chol_inv"][layer, g, s].double().cpu().numpy(), Minv,
                                           rtol=1e-4, atol=1e-6)


def test_layer_groups_bound_the_workspace_and_match_the_oracle():
    # the pass over groups of 2 of 5 layers with a workspace sized for a group
    wl = Workload("t", 5, 12, 2, (900, 333), 16, 64, seed=31)
    t = generate(wl, DEV)
    whole = Evictor(make_cache(t, wl), wl.budget)
    ev = Evictor(make_cache(t, wl), wl.budget, layer_group=2)
    assert ev.ws.numel() < whole.ws.numel() and [n for _, n in ev.groups] == [2, 2, 1]
    ev.run()
    ev.check()
    for s in range(len(wl.seqlens)):
        for layer in range(wl.num_layers):
            for g in range(wl.num_kv_heads):
                check_unit(ev, t, wl, jacap_params(), s, layer, g, check_w=False)
    gpu_selection_properties(ev.scores, ev.idx, ev.kept, wl.seqlens, wl.budget)


@pytest.mark.parametrize("schedule", [1, 2])
def test_repeat_calls_are_bitwise_deterministic(schedule):
    wl = Workload("t", 2, 8, 2, (1500, 700), 16, 64, seed=22)
    t = generate(wl, DEV)
    ev = Evictor(make_cache(t, wl), wl.budget, jacap_params(schedule=schedule))
    ev.run()
    ev.check()
    s1, i1 = ev.scores.clone(), ev.idx.clone()
    ev.run()
    ev.check()
    assert torch.equal(ev.scores, s1) and torch.equal(ev.idx, i1)


def test_strided_cache_views():
    # K/V as views into a padded buffer (token stride 136) and a head-major
    # buffer; the TMA maps and the gather must follow the strides.
    wl = Workload("t", 2, 8, 2, (700, 260), 16, 64, seed=23)
    t = generate(wl, DEV)
    L, Hkv, N, d = t.k.shape
    kb = torch.zeros((Hkv, L, N, 136), dtype=t.k.dtype, device=DEV)
    vb = torch.zeros_like(kb)
    kb[..., :d] = t.k.transpose(0, 1)
    vb[..., :d] = t.v.transpose(0, 1)
    k2 = kb.transpose(0, 1)[..., :d]
    v2 = vb.transpose(0, 1)[..., :d]
    ev_ref = evict(make_cache(t, wl), wl.budget)
    t2 = replace(t, k=k2, v=v2)
    ev = evict(Cache(t.q_win, k2, v2, t.cu_seqlens, t.seqlens, wl.num_q_heads), wl.budget)
    assert torch.equal(ev.scores, ev_ref.scores)
    assert torch.equal(ev.idx, ev_ref.idx)
    assert torch.equal(ev.k_out, ev_ref.k_out) and torch.equal(ev.v_out, ev_ref.v_out)
    check_unit(ev, t2, wl, jacap_params(), 1, 1, 1)


@pytest.mark.parametrize("name", ["bf16_gqa4_ragged_tails", "bf16_gqa2_peaky_tiny_seq", "f32_gqa4_peaky",
                                  "bf16_budget_exceeds_all"])
def test_fused_select_compact_equals_the_two_calls(name):
    # jacap_select_compact (one launch) against jacap_select + jacap_compact on
    # the same scores: positions, kept counts and rows bit for bit
    wl, params = SMALL[name]
    t = generate(wl, DEV)
    ev = evict(make_cache(t, wl), wl.budget, params)  # the fused call
    sep = Evictor(make_cache(t, wl), wl.budget, params)
    sep.scores.copy_(ev.scores)
    sep.ws[:64].zero_()
    sep.k_out.fill_(7)  # the zero rows must be written, not left over
    sep.v_out.fill_(7)
    sep.select()
    sep.compact()
    sep.check()
    assert torch.equal(ev.idx, sep.idx) and torch.equal(ev.kept, sep.kept)
    assert_rows_bitwise(sep.k_out, ev.k_out)
    assert_rows_bitwise(sep.v_out, ev.v_out)


def test_fused_select_compact_zero_fills_a_malformed_request():
    # request 1 claims tokens 300 .. 599 of a 500-token cache: it is refused
    # (positions -1, zero rows, status invalid argument) and request 0 is served
    wl = Workload("t", 1, 4, 2, (300, 200), 8, 32, seed=25)
    t = generate(wl, DEV)
    bad = torch.tensor([0, 300, 600], dtype=torch.int32, device=DEV)
    ev = Evictor(Cache(t.q_win, t.k, t.v, bad, [300, 300], wl.num_q_heads), wl.budget)
    ev.scores.fill_(1.0)  # all equal: the first B positions are kept
    ev.k_out.fill_(7)
    ev.v_out.fill_(7)
    ev.ws[:64].zero_()
    ev.select_compact()
    assert ev.device_status() == 1  # JACAP_ERR_INVALID_ARG
    assert ev.kept.cpu().tolist() == [wl.budget, 0]
    assert bool((ev.idx[:, :, 1] == -1).all())
    assert bool((ev.k_out[:, :, 1] == 0).all()) and bool((ev.v_out[:, :, 1] == 0).all())
    assert ev.idx[0, 0, 0].cpu().tolist() == list(range(wl.budget))
    for g in range(wl.num_kv_heads):
        assert_rows_bitwise(t.k[0, g, :wl.budget], ev.k_out[0, g, 0])
        assert_rows_bitwise(t.v[0, g, :wl.budget], ev.v_out[0, g, 0])


def test_window_of_one_gives_zero_scores_and_first_positions():
    wl = Workload("t", 1, 4, 2, (600,), 1, 40, seed=24)
    t = generate(wl, DEV)
    ev = evict(make_cache(t, wl), wl.budget)
    assert bool((ev.scores == 0).all())
    assert ev.idx[0, 0, 0].cpu().tolist() == list(range(40))


def test_malformed_cu_seqlens_is_reported_on_the_device():
    wl = Workload("t", 1, 4, 2, (300, 200), 8, 32, seed=25)
    t = generate(wl, DEV)
    bad = torch.tensor([0, 300, 400], dtype=torch.int32, device=DEV)  # does not end at N_tot
    ev = Evictor(Cache(t.q_win, t.k, t.v, bad, [300, 100], wl.num_q_heads), wl.budget)
    ev.run()
    assert ev.device_status() == 1  # JACAP_ERR_INVALID_ARG


def test_nonfinite_input_is_reported_on_the_device():
    wl = Workload("t", 1, 4, 2, (300,), 8, 32, seed=26)
    t = generate(wl, DEV)
    t.k[0, 1, 17, 5] = float("nan")
    ev = Evictor(make_cache(t, wl), wl.budget)
    ev.run()
    assert ev.device_status() == 5  # JACAP_ERR_NONFINITE


@pytest.mark.parametrize("dtype", ("bf16", "f32"))
def test_windows_that_are_not_finite_among_many_are_reported(dtype):
    """The statistics of 4096 heads, some of whose windows hold a NaN: their blocks set the status word
    while others read it, and each block skips or finishes as a whole. The next pass, over finite
    windows, starts clean."""
    wl = Workload("t", 32, 32, 8, (300, 200, 129, 77), 8, 32, dtype=dtype, seed=29)
    t = generate(wl, DEV)
    ref = evict(make_cache(t, wl), wl.budget)
    q = t.q_win.clone()
    t.q_win[:, ::3, ::5, 3, 17] = float("nan")
    ev = Evictor(make_cache(t, wl), wl.budget)
    for _ in range(5):
        ev.run()
        assert ev.device_status() == 5  # JACAP_ERR_NONFINITE
    t.q_win.copy_(q)
    ev.run()
    ev.check()
    assert torch.equal(ev.scores, ref.scores) and torch.equal(ev.idx, ref.idx)


def test_config1_every_unit():
    wl = config(1)
    t = generate(wl, DEV)
    ev = evict(make_cache(t, wl), wl.budget)
    for g in range(wl.num_kv_heads):
        check_unit(ev, t, wl, jacap_params(), 0, 0, g)
    gpu_selection_properties(ev.scores, ev.idx, ev.kept, wl.seqlens, wl.budget)


def _spread_units(wl, count):
    """`count` units (request, layer, KV head): the first and the last layer and
    KV head, the shortest and the longest request, the rest drawn with a fixed
    seed."""
    S, L, H = len(wl.seqlens), wl.num_layers, wl.num_kv_heads
    out = []

    def add(u):
        if u not in out:
            out.append(u)

    for s in dict.fromkeys([int(np.argmin(wl.seqlens)), int(np.argmax(wl.seqlens)), 0, S - 1]):
        add((s, 0, 0))
        add((s, L - 1, H - 1))
    add((0, 0, H - 1))
    add((0, L - 1, 0))
    r = np.random.default_rng(1000 + S * 100 + L)
    while len(out) < count:
        add((int(r.integers(S)), int(r.integers(L)), int(r.integers(H))))
    return out[:count]


def _check_sampled_units(t, wl, evs, units):
    """Scores, TOP-B sets (for every evictor's budget) and kept rows of `units`
    against the oracle, run on a pool of processes."""
    budgets = sorted({e.budget for e in evs})
    arrays = [tuple(x.astype(np.float32) for x in unit_arrays(t, wl.num_q_heads, s, layer, g))
              for (s, layer, g) in units]
    results = run_units(arrays, budgets)
    cu = t.cu_seqlens.cpu().tolist()
    for (s, layer, g), (ora_scores, ora_idx) in zip(units, results):
        a, b = cu[s], cu[s + 1]
        gs = evs[0].scores[layer, g, a:b].double().cpu().numpy()
        assert_scores_close(gs, ora_scores, f"scores of unit {(s, layer, g)}")
        for ev in evs:
            gidx = ev.idx[layer, g, s].cpu().numpy()
            assert_selection(gidx, b - a, ev.budget, ora_scores, ora_idx[ev.budget])
            kept = min(b - a, ev.budget)
            sel = torch.as_tensor(gidx[:kept], dtype=torch.long, device=t.k.device)
            assert_rows_bitwise(t.k[layer, g, a:b][sel], ev.k_out[layer, g, s, :kept])
            assert_rows_bitwise(t.v[layer, g, a:b][sel], ev.v_out[layer, g, s, :kept])


@pytest.mark.parametrize("index,samples", [(2, 8), (3, 8), (4, 16), (5, 16)])
def test_full_size_config(index, samples):
    wl = config(index)
    t = generate(wl, DEV)
    ev = evict(make_cache(t, wl), wl.budget)
    gpu_selection_properties(ev.scores, ev.idx, ev.kept, wl.seqlens, wl.budget)
    evs = [ev]
    if index == 2:
        # the other two budgets of the configuration: selection (and compaction)
        # on the same scores, as separate calls and as the fused call
        for b in (128, 2048):
            ev2 = Evictor(make_cache(t, wl), b)
            ev2.scores.copy_(ev.scores)
            ev2.ws[:64].zero_()  # status word: select honours the one jacap_score leaves
            ev2.select()
            ev2.compact()
            gpu_selection_properties(ev2.scores, ev2.idx, ev2.kept, wl.seqlens, b)
            k2, v2 = ev2.k_out.clone(), ev2.v_out.clone()
            ev2.select_compact()
            assert_rows_bitwise(k2, ev2.k_out)
            assert_rows_bitwise(v2, ev2.v_out)
            del k2, v2
            evs.append(ev2)
    _check_sampled_units(t, wl, evs, _spread_units(wl, samples))
    del ev, evs, t
    torch.cuda.empty_cache()


def _output_factors(wl, d_o, seed, device):
    """Synthetic output maps W (d_o x 128) per plane and their 128 x 128 factors
    F = R of W = Q R (float32 on the device); W stays on the host for the oracle."""
    r = np.random.default_rng(seed)
    L, Hkv = wl.num_layers, wl.num_kv_heads
    W = r.normal(size=(L, Hkv, d_o, 128)) / np.sqrt(128)
    F = np.stack([[np.linalg.qr(W[l, g])[1] for g in range(Hkv)] for l in range(L)])
    return W, torch.as_tensor(F, dtype=torch.float32, device=device).contiguous()


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_output_directions_every_unit(dtype):
    # u_i = W v_i (Sec. 3.1) through the reduced d x d form on the GPU vs the
    # oracle's explicit d_o-dimensional capacity matrix
    wl = Workload("t", 2, 8, 2, (1300, 400), 16, 96, dtype=dtype, seed=21)
    t = generate(wl, DEV)
    W, F = _output_factors(wl, 192, 5, DEV)
    params = jacap_params()
    ev = Evictor(make_cache(t, wl), wl.budget, params, out_factor=F)
    ev.run()
    ev.check()
    # the factors the GPU used, in float64, define the same W^T W as W up to rounding
    cu = t.cu_seqlens.cpu().tolist()
    for s in range(len(wl.seqlens)):
        for layer in range(wl.num_layers):
            for g in range(wl.num_kv_heads):
                q, K, V = unit_arrays(t, wl.num_q_heads, s, layer, g)
                Ff = F[layer, g].double().cpu().numpy()  # a d x d output map with the GPU's exact factor
                ora = oracle_unit(q, K, V, wl.budget, JacapParams(), out_proj=Ff)
                a, b = cu[s], cu[s + 1]
                assert_scores_close(ev.scores[layer, g, a:b].double().cpu().numpy(), ora["scores"])
                assert_selection(ev.idx[layer, g, s].cpu().numpy(), b - a, wl.budget, ora["scores"], ora["idx"])
                # and the explicit d_o-dimensional output map gives the same scores (push-through)
                ora_w = oracle_unit(q, K, V, wl.budget, JacapParams(), out_proj=W[layer, g])
                assert_scores_close(ev.scores[layer, g, a:b].double().cpu().numpy(), ora_w["scores"])


def test_pass_replays_from_a_cuda_graph():
    # the whole pass (scores, selection, compaction) captured once into a CUDA
    # graph and replayed gives the eager pass's results bit for bit
    wl, params = SMALL["bf16_gqa4_ragged_tails"]
    t = generate(wl, DEV)
    ev = evict(make_cache(t, wl), wl.budget, params)  # eager, also warms every kernel up
    ref = [x.clone() for x in (ev.scores, ev.idx, ev.kept, ev.k_out, ev.v_out)]
    for x in (ev.scores, ev.k_out, ev.v_out):
        x.zero_()
    ev.idx.fill_(-7)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(g, stream=side, capture_error_mode="thread_local"):
            ev.run(side)
    torch.cuda.current_stream().wait_stream(side)
    for _ in range(2):
        g.replay()
        torch.cuda.synchronize()
        ev.check()
        got = (ev.scores, ev.idx, ev.kept, ev.k_out, ev.v_out)
        assert all(torch.equal(a, b) for a, b in zip(ref, got))


def test_a_wait_that_nothing_ends_expires_and_the_context_stays_usable():
    # failure detection without a fault: a bounded wait on an mbarrier that
    # nothing arrives on gives up after its limit, the status word says
    # timeout, and the next pass on the same workspace runs clean
    import time

    from paper_2609_08131_gb300 import JACAP_ERR_TIMEOUT, jacap_selftest_wait
    from paper_2609_08131_gb300.api import _ptr, _stream

    wl = Workload("t", 1, 4, 2, (700, 129), 8, 64, seed=29)
    t = generate(wl, DEV)
    ev = Evictor(make_cache(t, wl), wl.budget)
    t0 = time.time()
    assert jacap_selftest_wait(_ptr(ev.ws), ev.ws.numel(), 20_000_000, _stream()) == 0
    assert ev.device_status() == JACAP_ERR_TIMEOUT
    assert time.time() - t0 < 5.0
    ev.run()
    ev.check()
    for g in range(wl.num_kv_heads):
        check_unit(ev, t, wl, jacap_params(), 1, 0, g)


def test_host_cache_pass_with_output_directions_matches_the_device_pass():
    # HostEvictor hands each layer group its slice of the output factors: the
    # kept positions and rows equal those of the device-resident pass (both run
    # the same kernels on the same bytes; only the chunking of a group's
    # layout may differ, so positions may differ only at near ties)
    from paper_2609_08131_gb300.api import HostEvictor

    wl = Workload("t", 3, 8, 2, (900, 300), 16, 64, seed=44)
    t = generate(wl, DEV)
    _, F = _output_factors(wl, 160, 9, DEV)
    dev = Evictor(make_cache(t, wl), wl.budget, jacap_params(), out_factor=F)
    dev.run()
    dev.check()
    he = HostEvictor(t.q_win.cpu().pin_memory(), t.k.cpu().pin_memory(), t.v.cpu().pin_memory(), t.cu_seqlens,
                     list(wl.seqlens), wl.num_q_heads, wl.budget, jacap_params(), group_layers=2, device=DEV,
                     out_factor=F)
    he.run()
    a, b = he.idx_h.reshape(-1, wl.budget).numpy(), dev.idx.cpu().reshape(-1, wl.budget).numpy()
    differ = sum(len(np.setdiff1d(x, y)) for x, y in zip(a, b))
    assert differ <= 2, differ
    if differ == 0:
        assert_rows_bitwise(dev.k_out, he.k_out_h)
        assert_rows_bitwise(dev.v_out, he.v_out_h)


def test_many_short_units_take_the_small_selection_ctas():
    # more units than SMs and requests of at most 4096 tokens: the selection
    # runs 256-thread CTAs (four or more per SM); sampled units against the
    # oracle, every unit's selection properties, and the fused selection +
    # compaction against the two separate calls
    wl = Workload("t", 24, 16, 8, (1500, 700, 129), 16, 96, seed=46)  # 24 x 8 x 3 = 576 units
    assert wl.num_layers * wl.num_kv_heads * len(wl.seqlens) > torch.cuda.get_device_properties(0).multi_processor_count
    t = generate(wl, DEV)
    ev = evict(make_cache(t, wl), wl.budget)
    gpu_selection_properties(ev.scores, ev.idx, ev.kept, wl.seqlens, wl.budget)
    for (s, layer, g) in ((0, 0, 0), (1, 11, 5), (2, 23, 7), (0, 17, 3)):
        check_unit(ev, t, wl, jacap_params(), s, layer, g, check_w=False)
    sep = Evictor(make_cache(t, wl), wl.budget)
    sep.scores.copy_(ev.scores)
    sep.ws[:64].zero_()
    sep.select()
    sep.compact()
    sep.check()
    assert torch.equal(ev.idx, sep.idx) and torch.equal(ev.kept, sep.kept)
    assert_rows_bitwise(sep.k_out, ev.k_out)
    assert_rows_bitwise(sep.v_out, ev.v_out)


def test_full_size_full_covariance():
    # the K pass with the full-covariance kappa on the 32-layer 32K-token
    # cache (every CTA runs several units, one image per run): sampled units
    # against the oracle, every unit's selection properties
    wl = config(2)
    t = generate(wl, DEV)
    params = jacap_params(full_covariance=1)
    ev = evict(make_cache(t, wl), wl.budget, params)
    gpu_selection_properties(ev.scores, ev.idx, ev.kept, wl.seqlens, wl.budget)
    for (layer, g) in ((0, 0), (31, 7), (13, 4)):
        check_unit(ev, t, wl, params, 0, layer, g, check_w=False)
    del ev, t
    torch.cuda.empty_cache()


@pytest.mark.parametrize("G", range(1, 9))
@pytest.mark.parametrize("scale", (1.0, 1e-12, 64.0))
def test_kappa_of_every_group_size_at_tile_edges(G, scale):
    """kappa through the linear surrogate's weights, w = (1/d) sum_h kappa_h, for requests that end
    before, on and after a tile's edge and keys far from 1. All terms are positive, squares and
    products are exact, so the error is that of lambda in float32 ((w + 3) 2^-24 relative: two sums
    over the window) and of at most 16 truncated and 8 rounded additions (2^-23 each at most). The
    factor of I + G, of rank 1 beside I for the request of one token, may lose its pivots in float32
    at the largest scale and report it after the weights are written: the status is not asked."""
    wl = Workload("t", 1, 2 * G, 2, (129, 1, 128, 127, 385), 16, 8, seed=300 + G)
    t = generate(wl, "cuda")
    t.k.mul_(scale)
    ev = evict(make_cache(t, wl), wl.budget, jacap_params(linear_weighting=1), check=False)
    w = ev.intermediates()["weights"].double()
    cu = t.cu_seqlens.tolist()
    bound = (16 + 3) * 2.0 ** -24 + (16 + 8) * 2.0 ** -23
    for s in range(len(wl.seqlens)):
        q = t.q_win[s, 0].double().view(2, G, 16, 128)
        lam = (q - q.mean(2, keepdim=True)).square().mean(2).sum(1)  # [2, 128], summed over the heads
        k2 = t.k[0, :, cu[s]:cu[s + 1]].double().square()
        ref = torch.einsum("gnc,gc->gn", k2, lam) / 128
        assert bool(((w[0, :, cu[s]:cu[s + 1]] - ref).abs() <= bound * ref).all())


@pytest.mark.parametrize("layers, lens", [
    (1, (1, 0, 700, 128, 129)),                                       # one run per CTA
    (2, tuple((37 * i * i) % 1700 for i in range(40))),               # more requests than a warp, one empty
    (8, (9000, 1, 0, 15000, 127, 128, 129, 6000, 0, 22001)),          # long runs, then short ones
])
def test_packed_requests_score_as_each_request_alone(layers, lens):
    """Every token of a packed cache is scored once, whichever runs its request is cut into: the
    scores are those of each request on its own, up to the order of float32 sums (the two partitions
    add the same non-negative terms; the pass is within 1e-5 of float64 either way)."""
    wl = Workload("t", layers, 8, 2, lens, 16, 32, seed=77)
    t = generate(wl, "cuda")
    ev = Evictor(make_cache(t, wl), wl.budget)
    ev.scores.fill_(-1.0)
    ev.run()
    ev.check()
    cu = t.cu_seqlens.tolist()
    for s, n in enumerate(lens):
        if n == 0:
            continue
        k, v = t.k[:, :, cu[s]:cu[s + 1]].contiguous(), t.v[:, :, cu[s]:cu[s + 1]].contiguous()
        one = evict(Cache(t.q_win[s:s + 1], k, v, torch.tensor([0, n], dtype=torch.int32, device="cuda"), [n], 8),
                    wl.budget)
        got, ref = ev.scores[:, :, cu[s]:cu[s + 1]].double(), one.scores.double()
        assert bool(((got - ref).abs() <= 2e-5 * ref).all())


@pytest.mark.parametrize("layers, hkv, lens, tau", [
    (1, 2, (20000,), 10.0),          # a few units of many partial Grams, summed by the launch before
    (1, 2, (20000,), 0.2),           # ... with a Gram far from 0
    (1, 1, (1, 0, 3, 130), 0.2),     # units of few tokens, one without any
    (20, 8, (300, 129), 1.0),        # more units than two CTAs per SM hold at once
])
def test_factor_inverts_the_capacity_matrix(layers, hkv, lens, tau):
    """X = L^{-1} as the factor writes it against A = I + G (G as it summed it): X A X^T = I within
    the bound of a backward stable factor and triangular inverse, 4 n 2^-24 cond(A) with n = 128,
    and X is lower triangular with zeros above. (The factor reads G's lower triangle; within a
    diagonal tile the products v_a (w v_b) of the other one are rounded on the other side.)"""
    wl = Workload("t", layers, 4 * hkv, hkv, lens, 16, 16, seed=91)
    t = generate(wl, "cuda")
    ev = evict(make_cache(t, wl), wl.budget, jacap_params(tau=tau))
    x = ev.intermediates()
    G, X = x["gram"].double(), x["chol_inv"].double()
    assert bool((X.triu(1) == 0).all())
    A = G.tril() + G.tril(-1).mT + torch.eye(128, dtype=torch.float64, device="cuda")
    cond = torch.linalg.cond(A)
    err = (X @ A @ X.mT - torch.eye(128, dtype=torch.float64, device="cuda")).abs().amax((-2, -1))
    assert bool((err <= 4 * 128 * 2.0 ** -24 * cond).all()), (err / cond).max()


@pytest.mark.parametrize("layers, hkv, lens, tau", [(1, 2, (20000,), 10.0), (1, 1, (1, 0, 130), 0.2), (20, 8, (300,), 1.0)])
def test_factor_with_output_directions_of_a_full_factor(layers, hkv, lens, tau):
    """T = L_M^{-1} F as the factor writes it, F a full matrix: T^T T = F^T M^{-1} F, M = I + F G F^T,
    within first-order bounds: forming M errs by 2 n 2^-24 |F|^2 |G| and M^{-1} is at most 1, the
    factor and the product T by 2 n 2^-24 cond(M), both taken between F^T and F (Frobenius norms)."""
    wl = Workload("t", layers, 4 * hkv, hkv, lens, 16, 16, seed=92)
    t = generate(wl, DEV)
    g = torch.Generator(device=DEV).manual_seed(5)
    F = torch.randn((layers, hkv, 128, 128), generator=g, device=DEV) / 128 ** 0.5
    ev = Evictor(make_cache(t, wl), wl.budget, jacap_params(tau=tau), out_factor=F)
    ev.run()
    ev.check()
    x = ev.intermediates()
    G, T, Fd = x["gram"].double(), x["chol_inv"].double(), F.double()[:, :, None]
    G = G.tril() + G.tril(-1).mT
    M = torch.eye(128, dtype=torch.float64, device=DEV) + Fd @ G @ Fd.mT
    err = (T.mT @ T - Fd.mT @ torch.linalg.solve(M, Fd.expand_as(M))).abs().amax((-2, -1))
    nf, ng = Fd.square().sum((-2, -1)), G.square().sum((-2, -1)).sqrt()
    bound = 2 * 128 * 2.0 ** -24 * (nf * ng + torch.linalg.cond(M)) * nf
    assert bool((err <= bound).all()), (err / bound).max()


SELECT_UNITS = ((1, 1), (20, 8), (40, 8))  # layers, KV heads: few units, more than SMs, more than twice


@pytest.mark.parametrize("layers, hkv", SELECT_UNITS)
@pytest.mark.parametrize("n", (1000, 4097, 8193, 20000, 40000))
@pytest.mark.parametrize("kind", ("spread", "ties", "equal", "wide", "zero_but_few"))
def test_selection_of_any_scores_is_the_stable_order(layers, hkv, n, kind):
    """jacap_select against a stable descending sort: scores of a few octaves, many equal scores at
    the boundary (by rank, and too many for that), all equal, spread over the whole exponent range
    (the B-th score far below the maximum), and fewer than B that are not 0. Selection compares bit
    patterns, so the positions are exactly those of the sort."""
    if layers * hkv > 8 and n > 20000:
        hkv, layers = 8, 20
    g = torch.Generator(device=DEV).manual_seed(n + layers)
    lens = (n, max(1, n // 3))
    N = sum(lens)
    B = max(1, n // 5)
    x = torch.rand((layers, hkv, N), generator=g, device=DEV)
    if kind == "spread":
        x = torch.exp(x * 4 - 9)
    elif kind == "ties":
        x = (x * 7).floor() / 8
    elif kind == "equal":
        x = torch.full_like(x, 0.25)
    elif kind == "wide":
        x = torch.exp2(x * 200 - 120) * (1 + x)
    else:
        x = torch.where(x < 0.03, x, torch.zeros_like(x))
    k = torch.zeros((layers, hkv, N, 128), dtype=torch.bfloat16, device=DEV)
    q = torch.zeros((2, layers, hkv, 1, 128), dtype=torch.bfloat16, device=DEV)
    cu = torch.tensor([0, lens[0], N], dtype=torch.int32, device=DEV)
    ev = Evictor(Cache(q, k, k, cu, list(lens), hkv), B)
    ev.ws[:64].zero_()
    ev.scores.copy_(x)
    ev.select()
    ev.check()
    for s, m in enumerate(lens):
        a = 0 if s == 0 else lens[0]
        order = torch.sort(x[:, :, a:a + m], dim=-1, descending=True, stable=True).indices[..., :B]
        want = torch.sort(order, dim=-1).values.int()
        kept = min(m, B)
        assert torch.equal(ev.idx[:, :, s, :kept], want[..., :kept])
        assert bool((ev.idx[:, :, s, kept:] == -1).all())


def test_f32_tiles_at_their_edges():
    """The float32 Gram and score kernels on requests that end before, on and after a tile's edge,
    every unit against the oracle (with weights and selection)."""
    wl = Workload("t", 2, 8, 2, (1, 127, 128, 129, 257, 640), 8, 48, dtype="f32", dist="outlier", seed=95,
                  outlier_channels=4, outlier_scale=8.0)
    t = generate(wl, DEV)
    params = jacap_params(tau=0.5)
    ev = evict(make_cache(t, wl), wl.budget, params)
    for s in range(len(wl.seqlens)):
        for layer in range(2):
            for g in range(2):
                check_unit(ev, t, wl, params, s, layer, g)


def _select(x, B):
    """jacap_select_compact of one request's scores x [L, Hkv, n]; K holds each token's position."""
    L, hkv, n = x.shape
    k = torch.zeros((L, hkv, n, 128), dtype=torch.float32, device=DEV)
    k[..., 0] = torch.arange(n, device=DEV)
    q = torch.zeros((1, L, hkv, 1, 128), dtype=torch.float32, device=DEV)
    ev = Evictor(Cache(q, k, k, torch.tensor([0, n], dtype=torch.int32, device=DEV), [n], hkv), B)
    ev.ws[:64].zero_()
    ev.scores.copy_(x)
    return ev


@pytest.mark.parametrize("layers, hkv", SELECT_UNITS)
@pytest.mark.parametrize("n", (2052, 4097, 20000, 40000))
@pytest.mark.parametrize("kind", ("far_below", "above_the_first_slab", "far_above", "half_ties", "subnormal", "equal_tail"))
def test_selection_outside_the_fine_bins_is_the_stable_order(layers, hkv, n, kind):
    """Boundaries that the selection's first histogram does not resolve: octaves far below the
    maximum, later slabs that exceed the first one's maximum (by an octave and by many), ties of which
    some are kept that straddle lanes, warps and slabs, subnormal scores and a tail of equal ones; at
    budgets whose bin holds a handful of keys and thousands. Bit patterns, so exactly the stable sort."""
    if layers * hkv > 8 and n > 20000:
        hkv, layers = 8, 20
    g = torch.Generator(device=DEV).manual_seed(n + layers)
    x = torch.rand((layers, hkv, n), generator=g, device=DEV)
    at = torch.arange(n, device=DEV)
    if kind == "far_below":
        x = torch.where(at % 97 == 0, x * 2.0 ** 40, x + 1e-3)
    elif kind == "above_the_first_slab":
        x = (x + 1e-2) * torch.where(at >= n - n // 4, 2.0 ** 6, 1.0)
    elif kind == "far_above":
        x = (x + 1e-2) * torch.exp2(at / n * 60 - 30)
    elif kind == "half_ties":
        x = torch.where(x < 0.6, torch.full_like(x, 0.3), x)
    elif kind == "subnormal":
        x = x * 2.0 ** -130
    else:
        x = torch.where(at < n // 3, x, torch.full_like(x, 2.0 ** -20))
    order = torch.sort(x, dim=-1, descending=True, stable=True).indices
    for B in (1, n // 97 + 200, n // 3, n - n // 5):
        ev = _select(x, B)
        ev.select_compact()
        ev.check()
        want = torch.sort(order[..., :B], dim=-1).values.int()
        assert torch.equal(ev.idx[:, :, 0], want)
        assert torch.equal(ev.k_out[:, :, 0, :, 0], want.float())


@pytest.mark.parametrize("kind", ("equal", "far_below", "far_above"))
def test_selection_takes_about_as_long_whatever_the_scores(kind):
    """256 units of 131072 scores, all equal (a window of one query), with the boundary 20 octaves below
    the maximum or growing along the request, against scores of a few octaves: a further digit is one
    more read of the keys beside at least four, so at most 1.6 times as long with the ranking saved or
    not (a read that waits for each key took 4 to 6 times as long)."""
    n, B = 131072, 8192
    g = torch.Generator(device=DEV).manual_seed(3)
    x = torch.rand((32, 8, n), generator=g, device=DEV)

    def us(scores):
        ev = _select(scores[:, :, :1024], 16)  # (a small cache; jacap_select reads no K or V)
        wide = torch.empty((32, 8, 1, B), dtype=torch.int32, device=DEV)
        lay = ev.lay
        cu = torch.tensor([0, n], dtype=torch.int32, device=DEV)
        lay.cu_seqlens, lay.max_seqlen, lay.total_tokens = cu.data_ptr(), n, n
        from paper_2609_08131_gb300 import jacap_select, jacap_workspace_size
        from paper_2609_08131_gb300.api import _ptr, _stream

        ws = torch.zeros(jacap_workspace_size(lay, B), dtype=torch.uint8, device=DEV)
        times = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            assert jacap_select(lay, _ptr(scores), B, _ptr(wide), _ptr(ev.kept), _ptr(ws), ws.numel(), _stream()) == 0
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return sorted(times)[3]

    plain = us(torch.exp(x * 4 - 9))
    if kind == "equal":
        y = torch.full_like(x, 0.25)
    elif kind == "far_below":
        y = torch.where(torch.arange(n, device=DEV) % 97 == 0, x * 2.0 ** 20, x + 1e-3)
    else:
        y = x * torch.linspace(0, 30, n, device=DEV).exp2()
    assert us(y.contiguous()) < 1.6 * plain


@pytest.mark.parametrize("G", range(1, 9))
def test_kappa_rounds_like_float32_multiply_adds(G):
    """kappa against 64 bits (through the linear surrogate's weights, lambda as the pass holds it), over
    131072 tokens: no bias and an rms error below half a unit in the last place, 2^-24, relative. Sums
    rounded to nearest show 4.5e-8 to 5.1e-8; sums that truncate, as the tensor cores', are too small
    by 6e-8 (two additions per group of channels) to 1.2e-7 (four). The mean over independent tokens is
    known to 5e-8 / sqrt(131072) < 2e-10; a quarter of 2^-24 is allowed for it."""
    wl = Workload("t", 2, 8 * G, 8, (8192,), 32, 64, seed=400 + G)
    t = generate(wl, DEV)
    ev = evict(make_cache(t, wl), wl.budget, jacap_params(linear_weighting=1))
    x = ev.intermediates()
    lam = x["lambda"][0].double().view(2, 8, G, 128).sum(2)
    ref = torch.einsum("lgnc,lgc->lgn", t.k.double().square(), lam) / 128
    err = x["weights"].double() / ref - 1
    assert abs(float(err.mean())) <= 0.25 * 2.0 ** -24
    assert float(err.square().mean().sqrt()) <= 2.0 ** -24


@pytest.mark.parametrize("dtype", ("bf16", "f32"))
@pytest.mark.parametrize("layers, hkv, lens", [
    (1, 1, (40000,)),               # one unit of 313 chunks: the reducing launch lists its partials twice
    (2, 1, (70000,)),
    (1, 1, (40000,) + (20,) * 60),  # the same in a pack whose mean has few partials: the factor lists them itself
    (36, 16, (1000,)),              # 576 units, four CTAs on an SM: in float32 eight partials each, reduced
    (40, 16, (1000,)),              # 640 units, three
])
def test_every_partial_gram_of_a_long_unit_is_summed(dtype, layers, hkv, lens):
    """G as the factor leaves it against sum_i w_i v_i v_i^T in 64 bits, with the pass's own weights, in
    units of more chunks than the lists of partials hold at once (256 and 288), and in each variant of
    the factor behind the reducing launch. w v is split within
    2^-17; sums over n tokens and their partials are float32, of random signs off the diagonal and each
    truncation at most 2^-23: 2^-15 of the sum of the terms' magnitudes covers them. One chunk of 313
    left out, or taken twice, is 3e-3 of it."""
    wl = Workload("t", layers, 4 * hkv, hkv, lens, 16, 16, dtype=dtype, dist="latent" if dtype == "bf16" else "outlier",
                  seed=93)
    t = generate(wl, DEV)
    ev = evict(make_cache(t, wl), wl.budget)
    x = ev.intermediates()
    at = 0
    for s, n in enumerate(lens):
        v, w = t.v[:, :, at:at + n].double(), x["weights"][:, :, at:at + n, None].double()
        at += n
        ref, size = v.mT @ (w * v), v.abs().mT @ (w * v.abs())
        assert bool(((x["gram"][:, :, s].double() - ref).abs() <= 2.0 ** -15 * size).all()), s
