"""GPU parity: the CUDA path, called through the C ABI, against the CPU oracle.

Bar: retained positions bit-exact outside a 1e-6 tie band on the attention
mass; K_out a bit-exact gather; V_out bit-exact where no injection happens,
within 1e-4 (fp32) / 2e-2 relative (bf16) otherwise; delta compared with an
eigen-gap-aware tolerance (the principal subspace is only determined up to the
gap between the last kept and first dropped eigenvalue).
"""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
import paper_2604_13349_b200 as P
from paper_2604_13349_b200 import synth
from tests import _parity as par

pytestmark = pytest.mark.gpu


def small(name, *, seed=7, layers=1, kv_heads=2, G=2, n_obs=5, d=64, dtype="f32", rank=2,
          caches=((100, 10),), heavy=3, n_outlier=0, n_sink=0):
    hs = synth.HeadSpec(head_dim=d, n_q=G * n_obs, n_outlier=n_outlier, heavy_count=heavy, n_sink=n_sink)
    return synth.Workload(name=name, seed=seed, layers=layers, kv_heads=kv_heads, q_heads=kv_heads * G,
                          n_obs=n_obs, rank=rank, dtype=dtype, head=hs,
                          caches=tuple(synth.CacheSpec(T=t, budget=b) for t, b in caches))


def all_heads(w):
    return [(l, h) for l in range(w.layers) for h in range(w.kv_heads)]


def run_and_check(w, rank=None, evict=False, heads=None, arrays=None, flags=0):
    arrays = arrays or [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    outs, _, st = par.run_gpu(w, arrays, rank=rank, evict=evict, flags=flags)
    assert st & 0xFF == 0, "device status %#x" % st
    eff_rank = 0 if evict else (w.rank if rank is None else rank)
    reps = []
    for ci in range(len(w.caches)):
        reps += par.check_cache(w, ci, arrays[ci], outs[ci], heads or all_heads(w), rank=eff_rank)
    print("\n[%s] %s" % (w.name, par.summarize(reps)))
    return outs, reps, arrays


# ---------------------------------------------------------------------------
# benchmark configurations that the oracle finishes whole
# ---------------------------------------------------------------------------
def test_c1_tiny_fp32_whole():
    outs, reps, _ = run_and_check(synth.workload("c1"))
    assert all(not r.oracle_skipped for r in reps)          # budget 32 < head_dim 64: OBF is active
    assert all(not r.band_mismatch for r in reps)


def test_c1_rank0_and_evict_only_agree():
    w = synth.workload("c1")
    a, _, arrays = run_and_check(w, rank=0)
    b, _, _ = run_and_check(w, evict=True, arrays=arrays)
    for x, y in zip(a, b):
        assert torch.equal(x["idx"], y["idx"]) and torch.equal(x["K_out"], y["K_out"])
        assert torch.equal(x["V_out"], y["V_out"])


def test_c2_bf16_whole():
    outs, reps, _ = run_and_check(synth.workload("c2"))
    assert all(r.oracle_skipped for r in reps)              # budget 205 > head_dim: span is full, delta = 0
    diags = P.parse_diag(outs[0]["diag"])
    assert all(dg["status"] & P.binding.OBF_DEV_SPAN_FULL for dg in diags)
    assert all(dg["span_rank"] == 128 for dg in diags)


# ---------------------------------------------------------------------------
# shapes: ragged tiles, tiny T, every dtype / head_dim, multi-layer, ragged batch
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("T,budget", [(1, 1), (2, 1), (63, 9), (65, 64), (129, 17), (1000, 31), (1025, 100)])
def test_ragged_shapes(dtype, d, T, budget):
    w = small("ragged", d=d, dtype=dtype, caches=((T, budget),), heavy=min(3, T), seed=T * 3 + d)
    run_and_check(w)


@pytest.mark.parametrize("G,n_obs", [(1, 1), (1, 5), (3, 7), (4, 16), (4, 40), (5, 32)])
def test_query_counts(G, n_obs):
    w = small("queries", G=G, n_obs=n_obs, d=128, dtype="bf16", caches=((300, 20),), n_outlier=3, seed=G * 10 + n_obs)
    run_and_check(w)


def test_multi_layer_ragged_batch_in_one_call():
    w = small("batch", layers=3, kv_heads=2, d=128, dtype="bf16", rank=2, n_sink=4,
              caches=((130, 13), (64, 64), (777, 100), (40, 3), (1, 1)))
    outs, reps, _ = run_and_check(w)
    assert len(reps) == 5 * 6


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_budget_at_least_T_is_the_identity(dtype):
    w = small("identity", d=64, dtype=dtype, caches=((50, 50), (50, 80)))
    outs, _, arrays = run_and_check(w)
    for ci in range(2):
        assert torch.equal(outs[ci]["idx"][0, 0].cpu(), torch.arange(50, dtype=torch.int32))
        assert np.array_equal(par.out_bits(outs[ci]["K_out"]), arrays[ci]["K"].view(
            np.int16 if dtype == "bf16" else np.int32))
        assert np.array_equal(par.out_bits(outs[ci]["V_out"]), arrays[ci]["V"].view(
            np.int16 if dtype == "bf16" else np.int32))


@pytest.mark.parametrize("rank", [1, 3, 64])
def test_rank_sweep_including_full_rank_cap(rank):
    w = small("ranks", d=64, dtype="f32", rank=rank, caches=((200, 12),))
    outs, reps, _ = run_and_check(w)
    assert all(not r.oracle_skipped for r in reps)


def test_codimension_one():
    w = small("codim1", d=64, dtype="f32", rank=2, caches=((150, 63),))
    outs, reps, _ = run_and_check(w)
    diags = P.parse_diag(outs[0]["diag"])
    assert all(dg["span_rank"] == 63 and dg["rho_eff"] == 1 for dg in diags)


@pytest.mark.parametrize("budget,rank", [(2, 8), (31, 1), (32, 2), (33, 4), (64, 8), (65, 2), (95, 3), (97, 9), (126, 2), (127, 2)])
def test_basis_sizes_around_the_batches_and_stages_of_the_dense_algebra(budget, rank):
    # retained rows come in batches of 32, reflectors in stages of 32, the tridiagonal form of what they leave ends at one
    # or two rows, more than eight eigenpairs take the Jacobi route
    w = small("basis", d=128, dtype="bf16", rank=rank, caches=((333, budget),), n_outlier=3, seed=budget)
    outs, reps, _ = run_and_check(w)
    assert all(dg["span_rank"] == budget for dg in P.parse_diag(outs[0]["diag"]))


@pytest.mark.parametrize("dtype,d,budgets", [("bf16", 128, (128, 129, 255, 257)), ("bf16", 64, (64, 65, 127, 129)),
                                             ("f32", 128, (128, 140)), ("f32", 64, (64, 65)), ("bf16", 128, (127, 128))])
def test_span_test_at_budgets_around_head_dim_and_its_row_limit(dtype, d, budgets):
    # full spans with few rows to spare, down to none (tiny pivots: the reflectors then decide): delta = 0 bit for bit;
    # one row short of head_dim: nothing to test
    w = small("span", d=d, dtype=dtype, rank=2, caches=tuple((700, b) for b in budgets), n_outlier=3, seed=d + len(budgets))
    outs, reps, _ = run_and_check(w)
    for o, b in zip(outs, budgets):
        assert all(dg["span_rank"] == min(b, d) for dg in P.parse_diag(o["diag"]))


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("bf16", 64), ("f32", 128), ("f32", 64)])
@pytest.mark.parametrize("channel", [1, 15, 16, 33, -1])
def test_span_test_finds_one_channel_that_depends_on_another(dtype, d, channel):
    # one channel repeats the first of its panel or of all (first and last pivots of a panel, first and last panel) on every row that can
    # be retained: the span lacks one dimension, which a few unselectable tokens carry
    channel %= d
    w = small("dep", d=d, dtype=dtype, rank=1, caches=((600, d + 40),), heavy=0, kv_heads=2, seed=60 + channel)
    arrays = [synth.gen_cache(w, 0)]
    a = arrays[0]
    K = par.f32_view(a["K"], dtype).copy(); V = par.f32_view(a["V"], dtype).copy()
    Qv = par.f32_view(a["Q"], dtype).reshape(1, 2, w.n_q, d)
    g = np.random.default_rng(channel)
    kept_apart = V[..., channel].copy()
    V[..., channel] = V[..., 0 if channel % 2 else 16 * (channel // 16) - 1]
    for h in range(2):
        qm = Qv[0, h].mean(axis=0)
        odd = g.choice(600, 15, replace=False)
        K[0, h, odd] = -1.5 * qm / np.linalg.norm(qm) * np.linalg.norm(K[0, h, odd], axis=1, keepdims=True)
        V[0, h, odd, channel] = kept_apart[0, h, odd]
    a["K"], a["V"] = (synth.to_bf16_bits(K), synth.to_bf16_bits(V)) if dtype == "bf16" else (K, V)
    outs, reps, _ = run_and_check(w, arrays=arrays)
    assert all(dg["span_rank"] == d - 1 for dg in P.parse_diag(outs[0]["diag"]))
    assert all(not r.oracle_skipped for r in reps)


def test_budget_above_head_dim_full_rank_is_bit_exact_eviction():
    w = small("full", d=64, dtype="bf16", rank=3, caches=((400, 90),))
    outs, reps, _ = run_and_check(w)
    assert all(r.oracle_skipped for r in reps)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_rank_deficient_values_with_budget_above_head_dim(dtype):
    # every value lives in the first 40 channels except a few tokens the keys make unselectable:
    # budget >= head_dim, span(V_keep) has dimension 40, the residual is not zero.
    w = small("rd", d=64, dtype=dtype, rank=2, caches=((300, 80),), heavy=0, kv_heads=2, seed=21)
    arrays = [synth.gen_cache(w, 0)]
    a = arrays[0]
    K = par.f32_view(a["K"], dtype).copy(); V = par.f32_view(a["V"], dtype).copy()
    Qv = par.f32_view(a["Q"], dtype).reshape(1, 2, w.n_q, 64)
    g = np.random.default_rng(5)
    V[..., 40:] = 0.0
    for h in range(2):
        qm = Qv[0, h].mean(axis=0)
        odd = g.choice(300, 15, replace=False)
        K[0, h, odd] = -1.5 * qm / np.linalg.norm(qm) * np.linalg.norm(K[0, h, odd], axis=1, keepdims=True)
        V[0, h, odd, 40:] = g.standard_normal((15, 24)).astype(np.float32)
    if dtype == "bf16":
        a["K"], a["V"] = synth.to_bf16_bits(K), synth.to_bf16_bits(V)
    else:
        a["K"], a["V"] = K, V
    outs, reps, _ = run_and_check(w, arrays=arrays)
    diags = P.parse_diag(outs[0]["diag"])
    assert all(dg["span_rank"] == 40 for dg in diags)
    assert all(not r.oracle_skipped for r in reps)
    assert torch.all(outs[0]["delta"][..., :40].abs() < 1e-5)
    assert torch.all(outs[0]["delta"].norm(dim=-1) > 1e-6)


# ---------------------------------------------------------------------------
# tuned bf16 / head_dim 128 path (tensor cores) against the oracle and against the shape-generic path
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("caches", [((128, 16),), ((300, 20), (130, 129), (777, 100)), ((1000, 200), (257, 31)),
                                    ((4096, 64),)])
def test_tuned_path_ragged_batches_match_oracle_and_generic_path(caches):
    w = small("tuned", layers=2, kv_heads=3, G=2, n_obs=9, d=128, dtype="bf16", rank=2, caches=caches,
              n_outlier=3, n_sink=2, seed=len(caches) * 31 + caches[0][0])
    a, reps, arrays = run_and_check(w)
    b, _, _ = run_and_check(w, arrays=arrays, flags=P.binding.OBF_FLAG_GENERIC_PATH)
    for x, y in zip(a, b):
        assert torch.equal(x["K_out"], y["K_out"])
        same = torch.equal(x["idx"], y["idx"])
        if same:
            assert torch.allclose(x["delta"], y["delta"], atol=2e-4, rtol=1e-3)
    assert any(not r.oracle_skipped for r in reps) or all(c[1] >= 128 for c in caches)


@pytest.mark.parametrize("G,n_obs,caches", [(2, 9, ((128, 16), (129, 64), (300, 63), (777, 100))),
                                            (2, 65, ((513, 30), (1025, 32))),       # two query tiles per head
                                            (4, 32, ((2048, 200),))])               # budget above head_dim: the span test's rows
def test_tuned_path_with_heads_of_64_channels(G, n_obs, caches):
    w = small("tuned64", layers=2, kv_heads=3, G=G, n_obs=n_obs, d=64, dtype="bf16", rank=2, caches=caches, n_outlier=3,
              n_sink=2, seed=40 + G)
    a, reps, arrays = run_and_check(w)
    names = [n for n, _ in P.obf_compress_profiled(par.params_for(w), a[0]["cache_structs"], a[0]["workspace"])]
    assert "k_score_tc" in names and "k_gram_tc" in names
    b, _, _ = run_and_check(w, arrays=arrays, flags=P.binding.OBF_FLAG_GENERIC_PATH)
    for x, y in zip(a, b):
        assert torch.equal(x["K_out"], y["K_out"])


def test_tuned_path_with_many_caches_of_different_lengths():
    # twelve caches in one call: every role of the score kernel walks the per-cache table
    Ts = [128, 131, 200, 256, 300, 511, 512, 513, 640, 777, 900, 1025]
    w = small("many", layers=1, kv_heads=2, G=2, n_obs=8, d=128, dtype="bf16", rank=2,
              caches=tuple((t, 16 + (t % 7)) for t in Ts), n_outlier=3, n_sink=2, seed=5)
    a, reps, arrays = run_and_check(w)
    assert all(not r.oracle_skipped for r in reps)
    b, _, _ = run_and_check(w, arrays=arrays, flags=P.binding.OBF_FLAG_GENERIC_PATH)
    for x, y in zip(a, b):
        assert torch.equal(x["K_out"], y["K_out"])


def test_tuned_path_rank_deficient_values_with_budget_above_head_dim():
    # head_dim 128, budget 160 >= head_dim, but every selectable value lives in the first 90 channels
    w = small("rd128", d=128, dtype="bf16", rank=3, caches=((700, 160),), heavy=0, kv_heads=2, seed=23)
    arrays = [synth.gen_cache(w, 0)]
    a = arrays[0]
    K = par.f32_view(a["K"], "bf16").copy(); V = par.f32_view(a["V"], "bf16").copy()
    Qv = par.f32_view(a["Q"], "bf16").reshape(1, 2, w.n_q, 128)
    g = np.random.default_rng(6)
    V[..., 90:] = 0.0
    for h in range(2):
        qm = Qv[0, h].mean(axis=0)
        odd = g.choice(700, 40, replace=False)
        K[0, h, odd] = -1.5 * qm / np.linalg.norm(qm) * np.linalg.norm(K[0, h, odd], axis=1, keepdims=True)
        V[0, h, odd, 90:] = g.standard_normal((40, 38)).astype(np.float32)
    a["K"], a["V"] = synth.to_bf16_bits(K), synth.to_bf16_bits(V)
    outs, reps, _ = run_and_check(w, arrays=arrays)
    diags = P.parse_diag(outs[0]["diag"])
    assert all(dg["span_rank"] == 90 for dg in diags)
    assert all(not r.oracle_skipped for r in reps)
    assert torch.all(outs[0]["delta"][..., :90].abs() < 1e-4)
    assert torch.all(outs[0]["delta"].norm(dim=-1) > 1e-6)


def _subspace_case(full_later: bool):
    """T = 2000, budget 400 >= head_dim.  Positions below 1500 hold values confined to the first 100 channels, so
    the first 256 retained rows (the subset the span test factorises) have rank 100.  full_later: the values at
    positions >= 1500 fill all 128 channels, else they are confined too and only a few unselectable tokens carry
    the other channels."""
    w = small("subspace", d=128, dtype="bf16", rank=3, caches=((2000, 400),), heavy=0, kv_heads=2, seed=29)
    arrays = [synth.gen_cache(w, 0)]
    a = arrays[0]
    K = par.f32_view(a["K"], "bf16").copy(); V = par.f32_view(a["V"], "bf16").copy()
    Qv = par.f32_view(a["Q"], "bf16").reshape(1, 2, w.n_q, 128)
    g = np.random.default_rng(8)
    V[:, :, :1500, 100:] = 0.0
    if not full_later:
        V[:, :, 1500:, 100:] = 0.0
        for h in range(2):
            qm = Qv[0, h].mean(axis=0)
            odd = g.choice(2000, 60, replace=False)
            K[0, h, odd] = -1.5 * qm / np.linalg.norm(qm) * np.linalg.norm(K[0, h, odd], axis=1, keepdims=True)
            V[0, h, odd, 100:] = g.standard_normal((60, 28)).astype(np.float32)
    a["K"], a["V"] = synth.to_bf16_bits(K), synth.to_bf16_bits(V)
    outs, reps, _ = run_and_check(w, arrays=arrays)
    idx = outs[0]["idx"].cpu().numpy()
    for h in range(2):
        assert (idx[0, h] < 1500).sum() >= 256 and (idx[0, h] >= 1500).sum() >= 40    # the construction holds
    return outs, reps


def test_span_subset_deficient_but_all_retained_rows_span_everything():
    # the Cholesky test on the first 256 retained rows fails; Gram-Schmidt over all 400 must reach rank 128: delta = 0
    outs, reps = _subspace_case(full_later=True)
    diags = P.parse_diag(outs[0]["diag"])
    assert all(dg["span_rank"] == 128 for dg in diags)
    assert all(r.oracle_skipped for r in reps)               # run_and_check has compared V_out bit for bit
    assert torch.all(outs[0]["delta"] == 0)


def test_span_subset_deficient_and_all_retained_rows_deficient_too():
    outs, reps = _subspace_case(full_later=False)
    diags = P.parse_diag(outs[0]["diag"])
    assert all(dg["span_rank"] == 100 for dg in diags)
    assert all(not r.oracle_skipped for r in reps)
    assert torch.all(outs[0]["delta"][..., :100].abs() < 1e-4)
    assert torch.all(outs[0]["delta"].norm(dim=-1) > 1e-6)


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("bf16", 64), ("f32", 64)])
@pytest.mark.parametrize("budget", [1, 2, 3, 4, 32, 33, 34, 35, 36, 61])
def test_retained_rows_two_apart_do_not_stand_in_for_one_another(dtype, d, budget):
    # Retained rows pass through two buffers in turn, in batches of 32.  Of every four the first two add a direction each, the third is a
    # multiple of the first and the fourth of the second: a row read in the place of the one two before or behind it changes the span.
    # 160 heads, so that two of 128 channels share a multiprocessor.
    w = small("turns", layers=20, kv_heads=8, d=d, dtype=dtype, rank=1, caches=((97, budget),), heavy=0, seed=150 + budget)
    arrays = [synth.gen_cache(w, 0)]
    a = arrays[0]
    V = par.f32_view(a["V"], dtype).copy()
    Qv = par.f32_view(a["Q"], dtype).reshape(w.layers, w.kv_heads, w.n_q, d)
    place = np.arange(budget)
    source = place - 2 * (place % 4 // 2)
    for l, h in all_heads(w):
        idx = oracle.topk(oracle.scores(par.f32_view(a["K"][l, h], dtype), Qv[l, h]), budget)[0]
        V[l, h, idx] = V[l, h, idx[source]] * np.where(place % 4 < 2, 1.0, -2.0).astype(np.float32)[:, None]
    a["V"] = synth.to_bf16_bits(V) if dtype == "bf16" else V
    outs, reps, _ = run_and_check(w, arrays=arrays, heads=[(0, 0), (7, 3), (19, 7)])
    assert all(dg["span_rank"] == len(set(source)) for dg in P.parse_diag(outs[0]["diag"]))
    assert all(not r.oracle_skipped for r in reps)


@pytest.mark.parametrize("dtype,d,flags", [("f32", 64, 0), ("f32", 128, 0), ("bf16", 64, 0), ("f32", 64, P.binding.OBF_FLAG_FAST_PATH)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_retained_row_that_is_not_finite_stays_out_of_the_others(dtype, d, flags, bad):
    # such a row adds no direction, like a row of zeros: the head's other rows get the delta that they would get beside that
    # (bf16 heads of 128 channels sum over all rows and skip the head)
    for row in (0, 1, 5, 33):
        w = small("notfinite", d=d, dtype=dtype, rank=1, kv_heads=1, caches=((300, 34),), seed=3)
        a = synth.gen_cache(w, 0)
        idx = oracle.topk(oracle.scores(par.f32_view(a["K"][0, 0], dtype), par.f32_view(a["Q"], dtype).reshape(w.n_q, d)), 34)[0]
        got = []
        for value in (0.0, bad):
            V = par.f32_view(a["V"], dtype).copy()
            V[0, 0, idx[row]] = 0.0
            V[0, 0, idx[row], 3] = value
            out, _, st = par.run_gpu(w, [dict(a, V=synth.to_bf16_bits(V) if dtype == "bf16" else V)], flags=flags)
            assert P.parse_diag(out[0]["diag"])[0]["span_rank"] == 33
            assert torch.all(out[0]["delta"].isfinite()) and torch.any(out[0]["delta"] != 0)
            got.append((out[0]["delta"][0, 0].cpu().numpy(), np.delete(out[0]["V_out"][0, 0].float().cpu().numpy(), row, axis=0)))
        assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1]), row


def test_retained_rows_with_a_dominant_common_component():
    # budget 24 < head_dim: every value is a common vector plus 3 % of noise, so after the first retained row every
    # further row loses nearly all of its norm to the basis in the first Gram-Schmidt pass and the kernel has to go
    # round a second time for it (a row that keeps more than half of its squared norm is orthogonalised once);
    # the basis, delta and V_out must still agree with the oracle, which always orthogonalises twice
    w = small("common", d=128, dtype="bf16", rank=2, caches=((900, 24),), heavy=4, kv_heads=2, seed=41)
    arrays = [synth.gen_cache(w, 0)]
    a = arrays[0]
    V = par.f32_view(a["V"], "bf16").copy()
    g = np.random.default_rng(5)
    common = g.standard_normal(128).astype(np.float32)
    V[:] = common + 0.03 * V
    a["V"] = synth.to_bf16_bits(V)
    outs, reps, _ = run_and_check(w, arrays=arrays)
    diags = P.parse_diag(outs[0]["diag"])
    assert all(dg["span_rank"] == 24 for dg in diags)
    assert all(not r.oracle_skipped for r in reps)
    assert torch.all(outs[0]["delta"].norm(dim=-1) > 0)


@pytest.mark.parametrize("T,budget", [(20000, 300), (70000, 250), (80000, 200)])
def test_long_prompts_take_the_fallback_kernels(T, budget):
    # 20000 keys: more than the select kernel keeps in shared memory; 70000 keys: one head is 274 chunks,
    # nearly all slots of the persistent score kernel, two a block; 80000 keys: more chunks than that kernel has slots,
    # so the shape-generic score kernels run (the Gram pass stays tuned)
    w = small("long", layers=1, kv_heads=1, G=4, n_obs=8, d=128, dtype="bf16", rank=1, caches=((T, budget),),
              n_outlier=3, n_sink=4, heavy=8, seed=T % 97)
    outs, reps, _ = run_and_check(w)
    assert all(r.oracle_skipped for r in reps)              # budget >= head_dim with generic values: delta = 0


@pytest.mark.parametrize("G,n_obs,caches", [(5, 32, ((640, 24),)),          # 160 rows: two query tiles per head
                                            (4, 40, ((1024, 32), (300, 20), (2048, 32))),   # the paper's 40 latent steps
                                            (8, 32, ((700, 40),)),          # 256 rows: two full tiles
                                            (2, 65, ((513, 30),))])         # 130 rows: second tile nearly empty
def test_between_129_and_256_query_rows_take_two_query_tiles_per_head(G, n_obs, caches):
    w = small("wideq", layers=2, kv_heads=3, G=G, n_obs=n_obs, d=128, dtype="bf16", rank=2, caches=caches,
              n_outlier=3, seed=77 + G)
    a, reps, arrays = run_and_check(w)
    assert all(not r.oracle_skipped for r in reps)
    names = [n for n, _ in P.obf_compress_profiled(par.params_for(w), a[0]["cache_structs"], a[0]["workspace"])]
    assert "k_score_tc" in names and "k_score_join" in names
    b, _, _ = run_and_check(w, arrays=arrays, flags=P.binding.OBF_FLAG_GENERIC_PATH)
    for x, y in zip(a, b):
        assert torch.equal(x["K_out"], y["K_out"])


def test_more_than_256_query_rows_use_the_generic_score_kernels_and_the_tuned_gram_pass():
    w = small("widerq", layers=1, kv_heads=2, G=9, n_obs=32, d=128, dtype="bf16", rank=2, caches=((640, 24),),
              n_outlier=3, seed=78)
    outs, reps, arrays = run_and_check(w)
    assert all(not r.oracle_skipped for r in reps)
    names = [n for n, _ in P.obf_compress_profiled(par.params_for(w), outs[0]["cache_structs"], outs[0]["workspace"])]
    assert "k_score_stats" in names and "k_gram_tc" in names


@pytest.mark.parametrize("d,G,n_obs,caches", [(64, 4, 16, ((64, 9), (65, 9), (129, 9), (2100, 30))), (128, 3, 22, ((700, 20), (150, 20)))])
def test_key_splits_of_the_shape_generic_statistics(d, G, n_obs, caches):
    # one cache of a batch fills all key splits, shorter ones leave some empty; n_q = 64, 66 rows
    w = small("splits", layers=1, kv_heads=2, G=G, n_obs=n_obs, d=d, dtype="f32", caches=caches, seed=d + G)
    run_and_check(w)


def test_exact_ties_go_to_the_lowest_position():
    # duplicated keys give bit-identical masses on the GPU as well; ties must resolve to lower positions
    w = small("ties", d=64, dtype="f32", rank=0, caches=((96, 20),), heavy=0, kv_heads=1)
    arrays = [synth.gen_cache(w, 0)]
    K = arrays[0]["K"]
    K[0, 0, 48:] = K[0, 0, :48]                          # position j+48 duplicates position j
    outs, _, st = par.run_gpu(w, arrays, rank=0)
    idx = outs[0]["idx"][0, 0].cpu().numpy()
    sc = outs[0]["scores"][0, 0].cpu().numpy()
    assert np.array_equal(sc[:48], sc[48:])
    ref = oracle.topk(sc.astype(np.float64), 20)[0]      # the oracle's rule applied to the GPU's own masses
    assert np.array_equal(idx, ref)
    assert all((j - 48) in idx for j in idx if j >= 48)     # a kept duplicate implies its lower twin is kept
    all_equal = small("alleq", d=64, dtype="bf16", rank=0, caches=((77, 11),), heavy=0, kv_heads=1)
    arr2 = [synth.gen_cache(all_equal, 0)]
    arr2[0]["K"][0, 0, :] = arr2[0]["K"][0, 0, 0]
    o2, _, _ = par.run_gpu(all_equal, arr2, rank=0)
    assert np.array_equal(o2[0]["idx"][0, 0].cpu().numpy(), np.arange(11))


def test_runs_are_deterministic():
    w = synth.workload("c1")
    arrays = [synth.gen_cache(w, 0)]
    a, _, _ = par.run_gpu(w, arrays)
    b, _, _ = par.run_gpu(w, arrays)
    for key in ("idx", "K_out", "V_out", "scores", "delta"):
        assert torch.equal(a[0][key], b[0][key]), key


def test_non_finite_inputs_set_the_status_word_and_stay_in_bounds():
    w = small("nan", d=64, dtype="f32", rank=1, caches=((120, 10),), kv_heads=1)
    arrays = [synth.gen_cache(w, 0)]
    arrays[0]["K"][0, 0, 5, 3] = np.nan
    outs, _, st = par.run_gpu(w, arrays)
    assert st & P.binding.OBF_DEV_NONFINITE
    idx = outs[0]["idx"][0, 0].cpu().numpy()
    assert len(set(idx.tolist())) == 10 and idx.min() >= 0 and idx.max() < 120


def test_a_device_side_wait_that_runs_out_reports_a_timeout_and_the_kernels_return():
    # nothing publishes the head's softmax normalisers and the wait limit is 20 ms: the score kernel's wait runs out
    w = small("expire", layers=1, kv_heads=2, G=2, n_obs=8, d=128, dtype="bf16", rank=2, caches=((700, 40),), seed=13)
    arrays = [synth.gen_cache(w, 0)]
    outs, dev, st = par.run_gpu(w, arrays, flags=P.binding.OBF_FLAG_TEST_WAIT_EXPIRES)
    assert st & P.binding.OBF_DEV_TIMEOUT
    idx = outs[0]["idx"].cpu().numpy()
    assert idx.min() >= 0 and idx.max() < 700               # whatever was selected lies inside the cache
    assert np.all(np.diff(idx, axis=-1) > 0)
    # the workspace, the streams and the device are as usable as before
    ws = outs[0]["workspace"]
    good = P.compress_caches(par.params_for(w), dev, want_scores=True, workspace=ws)
    torch.cuda.synchronize()
    assert P.obf_last_device_status(ws) & 0xFF == 0
    reps = par.check_cache(w, 0, arrays[0], good[0], all_heads(w))
    assert all(not r.oracle_skipped for r in reps)
    # the hook is refused outside its small shapes
    big = small("expire_big", layers=3, kv_heads=2, G=2, n_obs=8, d=128, dtype="bf16", caches=((700, 40),))
    with pytest.raises(Exception):
        par.run_gpu(big, [synth.gen_cache(big, 0)], flags=P.binding.OBF_FLAG_TEST_WAIT_EXPIRES)


def test_host_entry_point_matches_the_device_entry_point():
    w = synth.workload("c1")
    arrays = [synth.gen_cache(w, 0)]
    outs, _, _ = par.run_gpu(w, arrays)
    params = par.params_for(w)
    k = w.caches[0].budget
    hK = torch.from_numpy(arrays[0]["K"]).pin_memory(); hV = torch.from_numpy(arrays[0]["V"]).pin_memory()
    hQ = torch.from_numpy(arrays[0]["Q"]).pin_memory()
    oK = torch.empty((1, 2, k, 64)).pin_memory(); oV = torch.empty((1, 2, k, 64)).pin_memory()
    oI = torch.empty((1, 2, k), dtype=torch.int32).pin_memory()
    oD = torch.empty((1, 2, 64)).pin_memory()
    c = P.make_cache(hK, hV, hQ, 256, k, oK, oV, oI, None, None, oD)
    arena = torch.empty(P.obf_host_arena_bytes(params, [c]), dtype=torch.uint8, device="cuda")
    P.obf_compress_host(params, [c], arena)
    assert torch.equal(oI, outs[0]["idx"].cpu())
    assert torch.equal(oK, outs[0]["K_out"].cpu()) and torch.equal(oV, outs[0]["V_out"].cpu())
    assert torch.equal(oD, outs[0]["delta"].cpu())


@pytest.mark.parametrize("layers", [1, 5, 9])
def test_host_entry_point_pipelines_slabs_of_layers_for_ragged_batches(layers):
    # layer counts that the slabs do not divide evenly, two caches of different lengths, bf16 on the tuned path
    w = small("host", layers=layers, kv_heads=2, G=2, n_obs=8, d=128, dtype="bf16", rank=2,
              caches=((300, 20), (700, 140)), n_outlier=3, seed=19 + layers)
    arrays = [synth.gen_cache(w, ci) for ci in range(2)]
    outs, _, st = par.run_gpu(w, arrays)
    assert st & 0xFF == 0
    params = par.params_for(w)
    host, cs = [], []
    for ci, (T, b) in enumerate(((300, 20), (700, 140))):
        a = arrays[ci]
        h = {n: torch.from_numpy(a[n].view(np.int16)).view(torch.bfloat16).pin_memory() for n in ("K", "V", "Q")}
        h["oK"] = torch.empty((layers, 2, b, 128), dtype=torch.bfloat16).pin_memory()
        h["oV"] = torch.empty((layers, 2, b, 128), dtype=torch.bfloat16).pin_memory()
        h["oI"] = torch.empty((layers, 2, b), dtype=torch.int32).pin_memory()
        h["oS"] = torch.empty((layers, 2, T), dtype=torch.float32).pin_memory()
        h["oD"] = torch.empty((layers, 2, 128), dtype=torch.float32).pin_memory()
        host.append(h)
        cs.append(P.make_cache(h["K"], h["V"], h["Q"], T, b, h["oK"], h["oV"], h["oI"], None, h["oS"], h["oD"]))
    arena = torch.empty(P.obf_host_arena_bytes(params, cs), dtype=torch.uint8, device="cuda")
    for _ in range(2):                                      # twice: the second call reuses the arena and the streams
        P.obf_compress_host(params, cs, arena)
    for ci in range(2):
        h = host[ci]
        assert torch.equal(h["oI"], outs[ci]["idx"].cpu())
        assert torch.equal(h["oK"].view(torch.int16), outs[ci]["K_out"].cpu().view(torch.int16))
        assert torch.allclose(h["oV"].float(), outs[ci]["V_out"].cpu().float(), rtol=1e-2, atol=1e-5)
        assert torch.equal(h["oS"], outs[ci]["scores"].cpu())
        # the streaming pass cuts its tile sequence by the size of the call, so a slab adds its partial sums
        # up in another order than the whole call: delta agrees to fp32 rounding of the largest terms of those
        # sums (2^-22 of a value row's norm, about 15 here), not bit for bit
        assert torch.allclose(h["oD"], outs[ci]["delta"].cpu(), rtol=1e-4, atol=4e-6)


# ---------------------------------------------------------------------------
# benchmark configurations at full size: every head of every cache against one oracle run per cache, and the
# call shape the benchmark times (no optional outputs) bit for bit against the call with all outputs
# ---------------------------------------------------------------------------
@pytest.fixture(scope="module")
def c4_arrays():
    return [synth.gen_cache(synth.workload("c4"), 0)]


def run_whole(wname, arrays=None, evict=False, flags=0, layerwise=False):
    w = synth.workload(wname)
    arrays = arrays or [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    outs, dev, st = par.run_gpu(w, arrays, evict=evict, flags=flags)
    assert st & 0xFF == 0, "device status %#x" % st
    # what the benchmark times: the same call without diagnostics, masses and delta
    bare, _, st2 = par.run_gpu(w, arrays, evict=evict, flags=flags, want_scores=False, dev=dev,
                               want_delta=False, want_diag=False)
    assert st2 & 0xFF == 0
    for x, y in zip(outs, bare):
        assert torch.equal(x["idx"], y["idx"]), "retained positions depend on the optional outputs"
        assert torch.equal(x["K_out"].view(torch.int16), y["K_out"].view(torch.int16))
        assert torch.equal(x["V_out"].view(torch.int16), y["V_out"].view(torch.int16))
    del bare
    total = {}
    for ci in range(len(w.caches)):
        st_ci = par.check_cache_whole(w, ci, arrays[ci], outs[ci], rank=0 if evict else None, layerwise=layerwise)
        for k, v in st_ci.items():
            total[k] = total.get(k, 0) + v
    print("\n[%s whole] %s" % (wname, total))
    assert total["heads"] == len(w.caches) * w.layers * w.kv_heads
    return total


def test_c3_full_size_every_head():
    run_whole("c3")


def test_c4_full_size_rank4_every_head(c4_arrays):
    run_whole("c4", arrays=c4_arrays)


def test_c4_full_size_evict_only_every_head(c4_arrays):
    run_whole("c4_evict", arrays=c4_arrays, evict=True)


def test_c4_full_size_layerwise_every_layer(c4_arrays):
    run_whole("c4_layer", arrays=c4_arrays, flags=P.binding.OBF_FLAG_LAYERWISE, layerwise=True)


def test_c5_ragged_relay_batch_every_head_of_every_cache():
    run_whole("c5")


def test_paper_regime_budget_32_every_head():
    # kv_budget = 32 < head_dim with 40 latent steps: OBF's dense algebra runs for every head
    total = run_whole("pa")
    assert total["backfilled"] == total["heads"]


# ---------------------------------------------------------------------------
# layerwise selector: one retained set per layer, back-fill per head
# ---------------------------------------------------------------------------
def run_and_check_layerwise(w, arrays=None, flags=0, evict=False):
    arrays = arrays or [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    outs, _, st = par.run_gpu(w, arrays, evict=evict, flags=flags | P.binding.OBF_FLAG_LAYERWISE)
    assert st & 0xFF == 0, "device status %#x" % st
    reps = []
    for ci in range(len(w.caches)):
        reps += par.check_cache_layerwise(w, ci, arrays[ci], outs[ci], range(w.layers), rank=0 if evict else None)
    print("\n[%s layerwise] %s" % (w.name, par.summarize(reps)))
    return outs, reps, arrays


@pytest.mark.parametrize("dtype,d", [("f32", 64), ("bf16", 64), ("f32", 128)])
def test_layerwise_small_budgets_backfill_every_head(dtype, d):
    w = small("lw", layers=3, kv_heads=4, G=2, n_obs=5, d=d, dtype=dtype, rank=2, caches=((220, 14), (97, 9)), seed=33)
    outs, reps, _ = run_and_check_layerwise(w)
    assert all(not r.oracle_skipped for r in reps)              # budget < head_dim: OBF is active everywhere


def test_layerwise_c1_and_its_eviction_only_form():
    w = synth.workload("c1")
    a, reps, arrays = run_and_check_layerwise(w)
    assert all(not r.oracle_skipped for r in reps)
    b, _, _ = run_and_check_layerwise(w, arrays=arrays, evict=True)
    for x, y in zip(a, b):
        assert torch.equal(x["idx"], y["idx"]) and torch.equal(x["K_out"], y["K_out"])


@pytest.mark.parametrize("caches", [((300, 20), (130, 129), (777, 100)), ((2048, 205),)])
def test_layerwise_on_the_tensor_core_path(caches):
    w = small("lw_tuned", layers=2, kv_heads=3, G=2, n_obs=9, d=128, dtype="bf16", rank=4, caches=caches,
              n_outlier=3, n_sink=2, seed=51 + len(caches))
    a, reps, arrays = run_and_check_layerwise(w)
    b, _, _ = run_and_check_layerwise(w, arrays=arrays, flags=P.binding.OBF_FLAG_GENERIC_PATH)
    for x, y in zip(a, b):
        assert torch.equal(x["K_out"], y["K_out"])


def test_layerwise_with_one_kv_head_equals_headwise():
    w = small("lw1", layers=2, kv_heads=1, G=4, n_obs=4, d=64, dtype="f32", rank=1, caches=((150, 11),), seed=3)
    a, _, arrays = run_and_check_layerwise(w)
    b, _, _ = run_and_check(w, arrays=arrays)
    assert torch.equal(a[0]["idx"], b[0]["idx"]) and torch.equal(a[0]["V_out"], b[0]["V_out"])


def test_layerwise_rejects_prompts_that_do_not_fit_shared_memory():
    w = small("lw_long", layers=1, kv_heads=2, d=64, dtype="f32", rank=0, caches=((20000, 8),))
    arrays = [synth.gen_cache(w, 0)]
    with pytest.raises(Exception):
        par.run_gpu(w, arrays, flags=P.binding.OBF_FLAG_LAYERWISE)


# ---------------------------------------------------------------------------
# eigen-solve of the small-rank path: a residual spectrum with a tie at the top
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("rank", [1, 2, 3])
def test_residual_with_two_equal_leading_singular_values(rank):
    # The retained values live in the first 10 channels; every deleted value adds a component along channel 20
    # or channel 21, with the same energy on both and no correlation between them: the residual has two equal
    # leading singular values and nothing else.  Rank 2 and 3 have a unique answer (Delta = r_bar); rank 1 does
    # not (any direction of that plane is a leading singular vector), so only the invariants are checked for it.
    w = small("tie", d=64, dtype="f32", rank=rank, caches=((240, 12),), heavy=0, kv_heads=2, seed=77)
    arrays = [synth.gen_cache(w, 0)]
    a = arrays[0]
    Qv = a["Q"].reshape(1, 2, w.n_q, 64)
    g = np.random.default_rng(9)
    V = np.zeros_like(a["V"])
    for h in range(2):
        A = oracle.scores(a["K"][0, h], Qv[0, h])
        keep = np.zeros(240, bool); keep[oracle.topk(A, 12)[0]] = True
        V[0, h, :, :10] = g.standard_normal((240, 10)).astype(np.float32)
        dele = np.flatnonzero(~keep)
        half = len(dele) // 2
        V[0, h, dele[:half], 20] = 0.5                       # same count, same magnitude, disjoint supports
        V[0, h, dele[half:2 * half], 21] = 0.5
    a["V"] = V
    outs, reps, _ = run_and_check(w, arrays=arrays)
    assert all(not r.oracle_skipped for r in reps)
    d = outs[0]["delta"].cpu().numpy()
    assert np.all(np.abs(d[..., :10]) < 1e-5) and np.all(np.abs(d[..., 22:]) < 1e-5)
    if rank >= 2:
        assert all(r.gap_rel > 0.5 for r in reps)            # the plane itself is well separated from the rest
        assert np.all(np.linalg.norm(d, axis=-1) > 1e-4)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("rank", [2, 4])
@pytest.mark.parametrize("gap", [1e-2, 2e-3, 1.2e-3])
def test_close_eigenvalues_inside_the_principal_subspace(d, rank, gap):
    # The last two of the wanted eigenvalues lie a small gap apart and a fifth from the next one: the vectors of the two are
    # sensitive to the gap, the subspace (Eq. 5) is not, so delta must not be either.  No part of the deleted values lies in the
    # retained span, whose coordinates are separate.
    T, k, n = 600, 24, d - 24
    w = small("close", d=d, dtype="f32", rank=rank, kv_heads=1, caches=((T, k),), seed=103)
    for seed in range(4):
        a = synth.gen_cache(w, 0)
        rng = np.random.default_rng(seed)
        idx = oracle.topk(oracle.scores(a["K"][0, 0], a["Q"].reshape(1, 1, w.n_q, d)[0, 0]), k)[0]
        lam = 0.8 ** np.arange(n)
        lam[rank - 1] = lam[rank - 2] - gap * lam[0]
        lam[rank:] = lam[rank - 1] * 0.8 ** np.arange(1, n - rank + 1)
        U = np.linalg.qr(rng.standard_normal((T - k, n)))[0]
        W = np.linalg.qr(rng.standard_normal((n, n)))[0]
        V = np.zeros((T, d))
        dele = np.setdiff1d(np.arange(T), idx)
        V[idx, :k] = rng.standard_normal((k, k))
        V[dele, k:] = (U * np.sqrt(lam)) @ W * np.sqrt(T)
        a["V"] = (V @ np.linalg.qr(rng.standard_normal((d, d)))[0]).astype(np.float32)[None, None]
        out = par.run_gpu(w, [a])[0][0]
        g_idx = out["idx"][0, 0].cpu().numpy()
        ref = oracle.backfill(a["K"][0, 0], a["V"][0, 0], out["scores"][0, 0].cpu().numpy().astype(np.float64), g_idx, rank)["delta"]
        got = out["delta"][0, 0].cpu().numpy().astype(np.float64)
        # some 32 roundings of 2^-24 on the way to the subspace, over its distance of 0.2 (0.8^rank of it at most) from the rest
        assert np.linalg.norm(got - ref) <= 32 * par.U32 / (0.2 * 0.8 ** (rank - 2)) * np.linalg.norm(ref), (seed, np.linalg.norm(got - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("d,k", [(128, 24), (128, 70), (64, 20)])
@pytest.mark.parametrize("rank", [1, 2, 4, 8])
@pytest.mark.parametrize("spectrum", ["falls", "repeated", "outliers", "flat", "few"])
def test_tridiagonal_form_that_ends_early(d, k, rank, spectrum):
    # The reduction ends when its first rows hold the wanted eigenpairs and the next one.  Spectra that fall off end early, flat ones
    # late; a repeated eigenvalue must not be taken for one (the first rows hold one copy of it each), nor may a residual of
    # low rank end with fewer.
    T, n = 500, d - k
    w = small("early", d=d, dtype="f32", rank=rank, kv_heads=1, caches=((T, k),), seed=131)
    for seed in range(3):
        a = synth.gen_cache(w, 0)
        rng = np.random.default_rng(seed)
        idx = oracle.topk(oracle.scores(a["K"][0, 0], a["Q"].reshape(1, 1, w.n_q, d)[0, 0]), k)[0]
        lam = 0.75 ** np.arange(n)
        if spectrum == "repeated":
            lam = np.concatenate([np.full(rank, 0.5), 0.2 * 0.75 ** np.arange(n - rank)])
            lam[0] = 1.0 if rank > 2 else 0.5
        elif spectrum == "outliers":
            lam = np.concatenate([np.linspace(1.0, 0.9, rank), np.linspace(0.02, 0.01, n - rank)])
        elif spectrum == "flat":
            lam = np.linspace(1.0, 0.5, n)
            lam[:rank] += 0.2
        elif spectrum == "few":
            lam[rank + 1:] = 0.0
        U = np.linalg.qr(rng.standard_normal((T - k, n)))[0]
        W = np.linalg.qr(rng.standard_normal((n, n)))[0]
        V = np.zeros((T, d))
        dele = np.setdiff1d(np.arange(T), idx)
        V[idx, :k] = np.linalg.qr(rng.standard_normal((k, k)))[0] * np.sqrt(k)      # (nothing of their own that magnifies roundings)
        V[dele, k:] = (U * np.sqrt(lam)) @ W * np.sqrt(T)
        a["V"] = (V @ np.linalg.qr(rng.standard_normal((d, d)))[0]).astype(np.float32)[None, None]
        out = par.run_gpu(w, [a])[0][0]
        args = a["K"][0, 0], a["V"][0, 0], out["scores"][0, 0].cpu().numpy().astype(np.float64), out["idx"][0, 0].cpu().numpy()
        ref, whole = oracle.backfill(*args, rank), oracle.backfill(*args, n)["delta"]
        got = out["delta"][0, 0].cpu().numpy().astype(np.float64)
        gap = (lam[rank - 1] - lam[rank]) / lam[0]
        # some 32 roundings of 2^-24 on the way to the subspace, over its distance from the rest, of the vector that is projected on it
        err = np.linalg.norm(got - ref["delta"]) / np.linalg.norm(whole)
        assert err <= 32 * par.U32 / gap, (seed, err)
        dg, want = P.parse_diag(out["diag"])[0], ref["diag"]
        for key in ("lam_1", "lam_rho", "lam_next"):
            # the Gram matrix is a sum of T products, its eigenvalues are resolved to 6e-8 of a bound that is twice the largest at most
            assert abs(dg[key] - want[key]) <= 32 * par.U32 * want["lam_1"], (key, dg[key], want[key])


@pytest.mark.parametrize("rank", [1, 2, 4])
@pytest.mark.parametrize("first", [1, 6, 15])
@pytest.mark.parametrize("dead", [False, True])
def test_tridiagonal_form_that_falls_apart(rank, first, dead):
    # The retained values fill the first channels, the deleted ones two groups of channels on tokens of their own: the residual's Gram
    # matrix is block diagonal and so is the tridiagonal form, whose first rows hold a block of small eigenvalues (or, dead, of zeros)
    # and say nothing about how far the second block, with the wanted ones, has come.
    d, k, T = 128, 24, 500
    w = small("apart", d=d, dtype="f32", rank=rank, kv_heads=1, caches=((T, k),), seed=137)
    a = synth.gen_cache(w, 0)
    rng = np.random.default_rng(first)
    idx = oracle.topk(oracle.scores(a["K"][0, 0], a["Q"].reshape(1, 1, w.n_q, d)[0, 0]), k)[0]
    dele = np.setdiff1d(np.arange(T), idx)
    n = d - k - first
    lam = 0.9 ** np.arange(n)
    V = np.zeros((T, d))
    V[idx, :k] = np.linalg.qr(rng.standard_normal((k, k)))[0] * np.sqrt(k)
    if not dead:
        V[dele[:100], k:k + first] = 0.05 * rng.standard_normal((100, first))
    rows = len(dele) - 100
    V[dele[100:], k + first:] = (np.linalg.qr(rng.standard_normal((rows, n)))[0] * np.sqrt(lam)) @ np.linalg.qr(rng.standard_normal((n, n)))[0] * np.sqrt(T)
    a["V"] = V.astype(np.float32)[None, None]
    out = par.run_gpu(w, [a])[0][0]
    args = a["K"][0, 0], a["V"][0, 0], out["scores"][0, 0].cpu().numpy().astype(np.float64), out["idx"][0, 0].cpu().numpy()
    ref, whole = oracle.backfill(*args, rank), oracle.backfill(*args, d)["delta"]
    gap = (lam[rank - 1] - lam[rank]) / lam[0]
    # some 32 roundings of 2^-24 on the way to the subspace, over its distance from the rest, of the vector that is projected on it
    assert np.linalg.norm(out["delta"][0, 0].cpu().numpy().astype(np.float64) - ref["delta"]) <= 32 * par.U32 / gap * np.linalg.norm(whole)


def _backfill_of_a_form(a_diag, a_off, rank):
    """One fp32 head of 128 channels whose residual has the Gram matrix with this diagonal and these couplings: the retained rows fill the
    first channels, two neighbouring channels a deleted token (a row of the transposed Cholesky factor), so that the reduction
    leaves the matrix as it is.  (Without couplings a_diag is the whole matrix.)  Error of delta over the norm of what is projected, and
    the limit: some 32 roundings of 2^-24 over the distance of the wanted eigenvalues from the next."""
    n = len(a_diag)
    d, T = 128, 500
    k = d - n
    w = small("form", d=d, dtype="f32", rank=rank, kv_heads=1, caches=((T, k),), seed=139)
    a = synth.gen_cache(w, 0)
    rng = np.random.default_rng(n)
    idx = oracle.topk(oracle.scores(a["K"][0, 0], a["Q"].reshape(1, 1, w.n_q, d)[0, 0]), k)[0]
    dele = np.setdiff1d(np.arange(T), idx)
    M = a_diag if a_off is None else np.diag(a_diag) + np.diag(a_off, 1) + np.diag(a_off, -1)
    V = np.zeros((T, d))
    V[idx, :k] = np.linalg.qr(rng.standard_normal((k, k)))[0] * np.sqrt(k)
    V[rng.choice(dele, n, replace=False), k:] = np.linalg.cholesky(M).T * np.sqrt(T)
    a["V"] = V.astype(np.float32)[None, None]
    out = par.run_gpu(w, [a])[0][0]
    args = a["K"][0, 0], a["V"][0, 0], out["scores"][0, 0].cpu().numpy().astype(np.float64), out["idx"][0, 0].cpu().numpy()
    ref, whole = oracle.backfill(*args, rank), oracle.backfill(*args, d)["delta"]
    lam = np.linalg.eigvalsh(M)[::-1]
    # (the eigenvalues are resolved to 6e-8 of a bound that is twice the largest at most)
    dg, want = P.parse_diag(out["diag"])[0], ref["diag"]
    for key in ("lam_1", "lam_rho", "lam_next"):
        assert abs(dg[key] - want[key]) <= 32 * par.U32 * want["lam_1"], (key, dg[key], want[key])
    err = np.linalg.norm(out["delta"][0, 0].cpu().numpy().astype(np.float64) - ref["delta"]) / np.linalg.norm(whole)
    return err, 32 * par.U32 * lam[0] / (lam[rank - 1] - lam[rank])


@pytest.mark.parametrize("rank", [1, 2, 4, 8])
def test_tridiagonal_form_that_is_asked_about_several_times(rank):
    # a spectrum that falls off slowly: by how the rest comes down
    for seed in range(3):
        Q = np.linalg.qr(np.random.default_rng(seed).standard_normal((104, 104)))[0]
        err, limit = _backfill_of_a_form((Q * 0.95 ** np.arange(104)) @ Q.T, None, rank)
        assert err <= limit, (seed, err, limit)


@pytest.mark.parametrize("rank,first", [(2, 19), (2, 20), (2, 21), (2, 22), (2, 33), (3, 26), (3, 27), (4, 26), (4, 27), (8, 26), (8, 27)])
@pytest.mark.parametrize("coupling", [1e-8, 1e-5, 1e-3])
def test_largest_eigenvalue_that_enters_the_tridiagonal_form_late(rank, first, coupling):
    # Two groups of rows, hardly coupled.  The first holds all wanted eigenvalues but the largest, and the next one, and is complete (or has its
    # vectors settled) when the form's first rows are looked at; the second, with the largest eigenvalue, has only begun.
    for seed in range(3):
        rng = np.random.default_rng(seed)
        diag, off = np.zeros(104), np.full(103, coupling)
        small_ones = lambda n, by: 0.002 + 0.25 * by ** np.arange(n)
        for at, lam in ((0, np.concatenate([0.6 - 0.2 * np.arange(rank) / rank, small_ones(first - rank, 0.7)])),
                        (first, np.concatenate([[1.0], small_ones(103 - first, 0.8)]))):
            # the form of a dense matrix with these eigenvalues, by Lanczos' recurrence with all vectors kept orthogonal
            n = len(lam)
            q = [rng.standard_normal(n)]
            q[0] /= np.linalg.norm(q[0])
            for i in range(n):
                y = lam * q[i]
                diag[at + i] = q[i] @ y
                for _ in range(2):
                    y -= np.array(q).T @ (np.array(q) @ y)
                if i + 1 < n:
                    off[at + i] = np.linalg.norm(y)
                    q.append(y / off[at + i])
        err, limit = _backfill_of_a_form(diag, off, rank)
        assert err <= limit, (seed, err, limit)


@pytest.mark.parametrize("coupling", [0.05, 0.2])
def test_largest_eigenvalue_two_rows_before_the_end_of_the_leading_part(coupling):
    # no wanted eigenvalue's neighbourhood looks unsettled but the largest one's
    diag, off = np.full(104, 0.06), np.zeros(103)
    diag[[0, 1, 22]] = 0.6, 0.5, 1.0
    off[:30] = 0.02
    off[22], diag[23] = coupling, 0.06 + coupling ** 2
    err, limit = _backfill_of_a_form(diag, off, 2)
    assert err <= limit, (err, limit)


def test_next_eigenvalue_close_to_one_outside_the_leading_part():
    # The first row holds the wanted eigenvalue, rows 16 and 17 the next one, with a coupling of 2e-5 to a row behind them whose own
    # eigenvalue is 8e-5 smaller: as much as the leading part and the rest may share without the rest's bound showing it.
    diag, off = np.full(104, 1e-3), np.zeros(103)
    diag[0], diag[1:16], diag[17] = 1.0, 0.06, 0.06
    off[:15], off[15], off[16], off[17] = 0.02, 1e-3, 1e-3, 9e-3
    shift = 129 / 257 * 1.02                                  # the one just below the next eigenvalue
    diag[16], diag[18] = shift, shift - 2.5e-4
    for _ in range(5):
        T = np.diag(diag[:18]) + np.diag(off[:17], 1) + np.diag(off[:17], -1)
        diag[16] += shift + 1e-5 - np.linalg.eigvalsh(T)[-2]
    err, limit = _backfill_of_a_form(diag, off, 1)
    assert err <= limit, (err, limit)


@pytest.mark.parametrize("rank", [2, 8])
@pytest.mark.parametrize("leakage", [1e-9, 1e-7, 1e-6])
def test_two_groups_of_channels_that_hardly_mix(rank, leakage):
    for seed, first in enumerate((10, 18, 20, 25, 40)):
        rng = np.random.default_rng(seed)
        # (an eigenvalue of the second group, then one of the first, and so on, down to a floor)
        M = leakage * rng.standard_normal((104, 104))
        M += M.T
        for lo, hi, lead in ((0, first, 0.8), (first, 104, 1.0)):
            Q = np.linalg.qr(rng.standard_normal((hi - lo, hi - lo)))[0]
            M[lo:hi, lo:hi] = (Q * (1e-3 + lead * 0.7 ** np.arange(hi - lo))) @ Q.T
        err, limit = _backfill_of_a_form(M, None, rank)
        assert err <= limit, (seed, err, limit)


# ---------------------------------------------------------------------------
# protected sink prefix: the first s positions are retained besides the budget
# ---------------------------------------------------------------------------
def check_sink(w, n_sink, outs, arrays, layerwise=False, rank=None):
    rank = w.rank if rank is None else rank
    d, n_q, H = w.head.head_dim, w.n_q, w.kv_heads
    bits = np.int16 if w.dtype == "bf16" else np.int32
    reps = []
    for ci in range(len(w.caches)):
        a, out = arrays[ci], outs[ci]
        budget = w.caches[ci].budget
        Qv = a["Q"].reshape(w.layers, H, n_q, d)
        diags = P.parse_diag(out["diag"])
        for l in range(w.layers):
            K, V, Q = par.f32_view(a["K"][l], w.dtype), par.f32_view(a["V"][l], w.dtype), par.f32_view(Qv[l], w.dtype)
            lay = oracle.layer(K, V, Q, budget, rank, n_sink=n_sink) if layerwise else None
            for h in range(H):
                if layerwise:
                    ref = {"A": lay["A"][h], "idx": lay["idx"][h], "delta": lay["delta"][h], "V_out": lay["V_out"][h],
                           "diag": lay["diag"][h]}
                    sel, band = lay["S"].copy(), par.TIE_BAND * H
                else:
                    ref = oracle.head(K[h], V[h], Q[h], budget, rank, n_sink=n_sink)
                    sel, band = ref["A"].copy(), par.TIE_BAND
                sel[:n_sink] = np.inf                               # protected positions are never in the tie band
                g_idx = out["idx"][l, h].cpu().numpy()
                assert g_idx[:min(n_sink, K.shape[1])].tolist() == list(range(min(n_sink, K.shape[1])))
                reps.append(par.check_head(
                    w.dtype, K[h], V[h], Q[h], budget, rank, g_idx, par.out_bits(out["K_out"][l, h]),
                    par.out_bits(out["V_out"][l, h]), par.out_to_f32(out["V_out"][l, h]),
                    out["scores"][l, h].cpu().numpy(), out["delta"][l, h].cpu().numpy(), diags[l * H + h],
                    a["K"][l, h].view(bits), a["V"][l, h].view(bits), name="sink cache %d layer %d head %d" % (ci, l, h),
                    ref=ref, sel_scores=sel, tie_band=band, k_expected=oracle.k_eff(K.shape[1], budget, n_sink)))
    return reps


@pytest.mark.parametrize("dtype,d,caches,layerwise", [
    ("f32", 64, ((200, 12), (90, 9)), False), ("bf16", 128, ((300, 20), (777, 100), (130, 129)), False),
    ("f32", 64, ((200, 12),), True), ("bf16", 128, ((512, 28),), True)])
def test_sink_prefix_is_retained_besides_the_budget(dtype, d, caches, layerwise):
    w = small("sink", layers=2, kv_heads=3, G=2, n_obs=6, d=d, dtype=dtype, rank=2, caches=caches, seed=91, n_sink=0)
    arrays = [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    flags = P.binding.OBF_FLAG_SINK(4) | (P.binding.OBF_FLAG_LAYERWISE if layerwise else 0)
    outs, _, st = par.run_gpu(w, arrays, flags=flags)
    assert st & 0xFF == 0
    for ci, (T, b) in enumerate(caches):
        assert outs[ci]["idx"].shape[-1] == min(4, T) + min(b, T - min(4, T))
    reps = check_sink(w, 4, outs, arrays, layerwise=layerwise)
    print("\n[sink] %s" % par.summarize(reps))


# ---------------------------------------------------------------------------
# out-of-prompt softmax mass: the keys outside the prompt take their share of every row's normaliser
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("dtype,d,G,n_obs,caches,flags", [
    ("f32", 64, 2, 5, ((200, 12), (90, 9)), 0),
    ("bf16", 128, 2, 9, ((300, 20), (777, 100), (1100, 32)), 0),                 # tuned score kernel, several chunks per head
    ("bf16", 128, 5, 32, ((640, 24),), 0),                                       # two query tiles per head
    ("bf16", 128, 2, 9, ((300, 20),), P.binding.OBF_FLAG_GENERIC_PATH)])
def test_out_of_prompt_softmax_mass(dtype, d, G, n_obs, caches, flags):
    w = small("lse", layers=2, kv_heads=2, G=G, n_obs=n_obs, d=d, dtype=dtype, rank=2, caches=caches, seed=71 + G)
    arrays = [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    g = np.random.default_rng(17)
    params = par.params_for(w, flags=flags)
    dev, lses = [], []
    from scipy.special import logsumexp
    for ci, a in enumerate(arrays):
        # around each row's own log-sum-exp over the prompt: between "nearly nothing outside the prompt" and
        # "most of the mass outside it"; one row without any
        Kf = par.f32_view(a["K"], dtype).astype(np.float64)
        Qf = par.f32_view(a["Q"], dtype).astype(np.float64).reshape(w.layers, w.kv_heads, w.n_q, d)
        own = logsumexp(np.einsum("lhqd,lhtd->lhqt", Qf, Kf) / np.sqrt(d), axis=-1)
        le = (own + g.standard_normal(own.shape) * 3).astype(np.float32).reshape(w.layers, w.q_heads, w.n_obs)
        le[0, 0, 0] = -np.inf
        lses.append(le)
        dev.append({"K": par.to_device(a["K"], dtype), "V": par.to_device(a["V"], dtype), "Q": par.to_device(a["Q"], dtype),
                    "budget": w.caches[ci].budget, "lse_extra": torch.from_numpy(le).cuda()})
    outs = P.compress_caches(params, dev, want_scores=True)
    torch.cuda.synchronize()
    assert P.obf_last_device_status(outs[0]["workspace"]) & 0xFF == 0
    bits = np.int16 if dtype == "bf16" else np.int32
    reps = []
    for ci, a in enumerate(arrays):
        Qv = par.f32_view(a["Q"], dtype).reshape(w.layers, w.kv_heads, w.n_q, d)
        le = lses[ci].reshape(w.layers, w.kv_heads, w.n_q)
        diags = P.parse_diag(outs[ci]["diag"])
        for l, h in all_heads(w):
            K, V = par.f32_view(a["K"][l, h], dtype), par.f32_view(a["V"][l, h], dtype)
            ref = oracle.head(K, V, Qv[l, h], w.caches[ci].budget, w.rank, lse_extra=le[l, h])
            assert ref["A"].sum() < w.n_q * 0.999                   # the outside keys did take mass
            out = outs[ci]
            reps.append(par.check_head(
                dtype, K, V, Qv[l, h], w.caches[ci].budget, w.rank, out["idx"][l, h].cpu().numpy(),
                par.out_bits(out["K_out"][l, h]), par.out_bits(out["V_out"][l, h]), par.out_to_f32(out["V_out"][l, h]),
                out["scores"][l, h].cpu().numpy(), out["delta"][l, h].cpu().numpy(), diags[l * w.kv_heads + h],
                a["K"][l, h].view(bits), a["V"][l, h].view(bits), name="lse cache %d layer %d head %d" % (ci, l, h), ref=ref))
    print("\n[lse_extra] %s" % par.summarize(reps))


# ---------------------------------------------------------------------------
# Attn-inject (App. D.2): the back-fill shared out by attention mass
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("dtype,d,caches", [("f32", 64, ((200, 12), (90, 9))), ("bf16", 128, ((300, 20), (1024, 32)))])
def test_attn_inject_shares_the_backfill_by_attention_mass(dtype, d, caches):
    w = small("attn", layers=2, kv_heads=2, G=2, n_obs=6, d=d, dtype=dtype, rank=2, caches=caches, seed=97)
    arrays = [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    outs, _, st = par.run_gpu(w, arrays, flags=P.binding.OBF_FLAG_ATTN_INJECT)
    assert st & 0xFF == 0
    plain, _, _ = par.run_gpu(w, arrays)
    checked = 0
    for ci, a in enumerate(arrays):
        o = outs[ci]
        # selection, keys and delta itself are those of the uniform injection
        assert torch.equal(o["idx"], plain[ci]["idx"]) and torch.equal(o["K_out"], plain[ci]["K_out"])
        assert torch.equal(o["delta"], plain[ci]["delta"])
        Qv = par.f32_view(a["Q"], dtype).reshape(w.layers, w.kv_heads, w.n_q, d)
        for l, h in all_heads(w):
            K, V = par.f32_view(a["K"][l, h], dtype), par.f32_view(a["V"][l, h], dtype)
            ref = oracle.head(K, V, Qv[l, h], w.caches[ci].budget, w.rank)
            idx = o["idx"][l, h].cpu().numpy()
            if not np.array_equal(idx, ref["idx"]) or ref["diag"]["skipped"]:
                continue
            dg = ref["diag"]
            gap = (dg["lam_rho"] - dg["lam_next"]) / dg["lam_1"]
            if gap < 1e-3:
                continue
            expect = oracle.attn_inject(V, ref["A"], idx, ref["delta"])
            share = len(idx) * ref["A"][idx] / (ref["A"][idx].sum() + 1e-12)
            dtol = max(2e-5 if dtype == "f32" else 2e-4, 200.0 * par.U32 / gap * dg["alpha"] * dg["rbar_norm"])
            # the tolerance on delta times the row's share (plus the share's own error: masses to 1e-5), and half a
            # bf16 ulp of the result on the bf16 path
            bound = share[:, None] * (dtol + 2e-5 * np.abs(ref["delta"])[None, :]) + 1e-6
            if dtype == "bf16":
                bound = bound + 2.0 ** -8 * 1.01 * np.abs(expect)
            err = np.abs(par.out_to_f32(o["V_out"][l, h]).astype(np.float64) - expect)
            assert np.all(err <= bound), "cache %d layer %d head %d: max err %.3g" % (ci, l, h, err.max())
            assert not np.allclose(share, 1.0)                      # the shares do differ from the uniform ones
            checked += 1
    assert checked >= 4


# ---------------------------------------------------------------------------
def test_early_out_skips_the_value_pass_of_full_heads_and_changes_nothing():
    # two caches: budget 200 >= head_dim (generic values: every head's retained values span R^d) and budget 40 < head_dim
    # (every head is back-filled).  With OBF_FLAG_EARLY_OUT the span test runs first and the pass over V skips the heads
    # of the first cache: every output must be the same bit for bit, and the back-filled heads must still be back-filled
    w = small("early", layers=2, kv_heads=2, G=4, n_obs=8, d=128, dtype="bf16", rank=2, caches=((1300, 200), (900, 40)),
              seed=53)
    arrays = [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    plain, _, st0 = par.run_gpu(w, arrays)
    early, _, st1 = par.run_gpu(w, arrays, flags=P.binding.OBF_FLAG_EARLY_OUT)
    assert st0 & 0xFF == 0 and st1 & 0xFF == 0
    for a, b in zip(plain, early):
        for key in ("idx", "K_out", "V_out", "delta", "scores"):
            assert torch.equal(a[key], b[key]), key
    assert torch.all(early[0]["delta"] == 0) and torch.all(early[1]["delta"].norm(dim=-1) > 0)
    d0, d1 = P.parse_diag(early[0]["diag"]), P.parse_diag(early[1]["diag"])
    assert all(dg["span_rank"] == 128 for dg in d0) and all(dg["span_rank"] == 40 for dg in d1)


# cache-merging baseline (App. E): deleted values merged into the retained position with the most similar key
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("dtype,d,caches,flags", [
    ("f32", 64, ((200, 12), (90, 9), (70, 70)), 0),
    ("bf16", 128, ((300, 20), (1024, 32), (700, 150)), 0),
    ("bf16", 128, ((512, 28),), P.binding.OBF_FLAG_LAYERWISE)])
def test_cache_merging_baseline(dtype, d, caches, flags):
    w = small("merge", layers=2, kv_heads=2, G=2, n_obs=6, d=d, dtype=dtype, rank=2, caches=caches, seed=101)
    arrays = [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    outs, _, st = par.run_gpu(w, arrays, flags=flags | P.binding.OBF_FLAG_MERGE, want_assign=True)
    assert st & 0xFF == 0
    ev, _, _ = par.run_gpu(w, arrays, evict=True, flags=flags)
    bits = np.int16 if dtype == "bf16" else np.int32
    near_ties = flips = 0
    for ci, a in enumerate(arrays):
        o = outs[ci]
        assert torch.equal(o["idx"], ev[ci]["idx"]) and torch.equal(o["K_out"], ev[ci]["K_out"])    # selection and keys: plain eviction
        assert torch.all(o["delta"] == 0)
        Qv = par.f32_view(a["Q"], dtype).reshape(w.layers, w.kv_heads, w.n_q, d)
        for l in range(w.layers):
            lay = None
            if flags & P.binding.OBF_FLAG_LAYERWISE:
                lay = oracle.layer(par.f32_view(a["K"][l], dtype), par.f32_view(a["V"][l], dtype), Qv[l], w.caches[ci].budget, 0)
            for h in range(w.kv_heads):
                K, V = par.f32_view(a["K"][l, h], dtype), par.f32_view(a["V"][l, h], dtype)
                ref = oracle.merge_head(K, V, Qv[l, h], w.caches[ci].budget)
                idx = o["idx"][l, h].cpu().numpy()
                g_assign = o["assign"][l, h].cpu().numpy()
                if lay is not None:
                    assert np.array_equal(idx, lay["idx"][h])
                elif not np.array_equal(idx, ref["idx"]):
                    continue                                        # a tie inside the selection band
                T = K.shape[0]
                keep = np.zeros(T, bool); keep[idx] = True
                assert np.all(g_assign[keep] == -1) and np.all((g_assign[~keep] >= 0) & (g_assign[~keep] < len(idx)))
                A = lay["A"][h] if lay is not None else ref["A"]
                if lay is None:
                    # routing: equal to the oracle's wherever the two best similarities are further apart than fp32
                    # can blur (1e-5); elsewhere the GPU's choice must be one of the near-best
                    clear = ref["margin"] > 1e-5
                    assert np.array_equal(g_assign[clear & ~keep], ref["assign"][clear & ~keep])
                    near_ties += int((~clear & ~keep).sum())
                    flips += int((g_assign != ref["assign"]).sum())
                    Kd = K.astype(np.float64); Kn = Kd / np.maximum(np.linalg.norm(Kd, axis=1, keepdims=True), 1e-300)
                    for j in np.flatnonzero(g_assign != ref["assign"]):
                        cs = Kn[idx] @ Kn[j]
                        assert cs[g_assign[j]] >= cs.max() - 1e-5
                # merged values: the oracle's step (iii) on the routing the GPU took
                expect = oracle.merge_given(V, A, idx, g_assign)
                absum = np.abs(V[idx].astype(np.float64))
                for j in np.flatnonzero(~keep):
                    absum[g_assign[j]] += A[j] / (A[idx[g_assign[j]]] + 1e-12) * np.abs(V[j].astype(np.float64))
                # fp32 accumulation of the weighted sum (weights carry the masses' 1e-5) and one rounding of the result
                bound = 4e-5 * absum + 1e-6
                if dtype == "bf16":
                    bound = bound + 2.0 ** -8 * 1.01 * np.abs(expect)
                err = np.abs(par.out_to_f32(o["V_out"][l, h]).astype(np.float64) - expect)
                assert np.all(err <= bound), "cache %d layer %d head %d: merged values off by %.3g" % (ci, l, h, err.max())
                assert np.array_equal(par.out_bits(o["K_out"][l, h]), a["K"][l, h].view(bits)[idx])
    print("\n[merge] near-tie routings %d, of which the GPU chose another near-best slot %d" % (near_ties, flips))


@pytest.mark.parametrize("d,caches", [(64, ((65, 1), (257, 64), (300, 65))), (128, ((255, 63), (129, 8), (513, 200)))])
def test_cache_merging_around_the_tiles_of_the_tensor_core_routing(d, caches):
    # positions come in tiles of 16, 64 and 256, slots in groups of 8 and 64
    test_cache_merging_baseline("bf16", d, caches, 0)


# ---------------------------------------------------------------------------
# int8 copy of the compacted relay (post-hoc quantisation stacked on the compression, App. E)
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("dtype,d,caches,flags", [
    ("f32", 64, ((200, 12), (90, 90)), 0),
    ("bf16", 128, ((300, 20), (777, 140)), 0),
    ("bf16", 128, ((512, 28),), P.binding.OBF_FLAG_LAYERWISE)])
def test_int8_copy_of_the_relay(dtype, d, caches, flags):
    w = small("q8", layers=2, kv_heads=2, G=2, n_obs=6, d=d, dtype=dtype, rank=2, caches=caches, seed=83)
    arrays = [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    outs, _, st = par.run_gpu(w, arrays, flags=flags, want_int8=True)
    assert st & 0xFF == 0
    plain, _, _ = par.run_gpu(w, arrays, flags=flags)
    injected = 0
    for ci, a in enumerate(arrays):
        o = outs[ci]
        # the usual outputs do not depend on the int8 copy being asked for
        for key in ("idx", "K_out", "V_out"):
            assert torch.equal(o[key], plain[ci][key]), key
        Kf, Vf = o["K_out"].float().cpu().numpy(), o["V_out"].float().cpu().numpy()
        for name, X in (("K", Kf), ("V", Vf)):
            codes, scales = oracle.quantize_rows(X)                     # the oracle's quantiser on the relay as it left
            assert np.array_equal(o[name + "_q8"].cpu().numpy(), codes), "%s codes differ" % name
            assert np.array_equal(o[name + "_scale"].cpu().numpy(), scales), "%s scales differ" % name
            back = codes.astype(np.float64) * scales.astype(np.float64)[..., None]
            # x / scale is rounded to fp32 before the rounding to a code: 127 * 2^-24 of a step on top of half a step
            assert np.all(np.abs(back - X) <= 0.5 * scales[..., None] * (1 + 2.0 ** -15))
        # the keys are exact copies of the inputs: their codes are those of the oracle's own gather
        idx = o["idx"].cpu().numpy()
        Kin = par.f32_view(a["K"], dtype)
        for l, h in all_heads(w):
            assert np.array_equal(o["K_q8"][l, h].cpu().numpy(), oracle.quantize_rows(Kin[l, h][idx[l, h]])[0])
        injected += int((o["delta"].abs().sum(dim=-1) > 0).sum())
    assert injected > 0                                                 # some values were quantised after an injection


def test_sink_prefix_longer_than_the_prompt_keeps_everything():
    w = small("sink_all", d=64, dtype="f32", rank=1, caches=((6, 3),), heavy=0)
    arrays = [synth.gen_cache(w, 0)]
    outs, _, st = par.run_gpu(w, arrays, flags=P.binding.OBF_FLAG_SINK(10))
    assert st & 0xFF == 0
    assert outs[0]["idx"].shape[-1] == 6
    assert torch.equal(outs[0]["idx"][0, 0].cpu(), torch.arange(6, dtype=torch.int32))


# ---------------------------------------------------------------------------
# fixed three-iteration Gram subspace path (an approximation: compared with the oracle's same iteration)
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("dtype,d,rank,caches", [("f32", 64, 2, ((200, 12), (90, 9))), ("f32", 128, 4, ((300, 20),)),
                                                 ("bf16", 128, 4, ((1024, 32), (300, 20))), ("f32", 64, 8, ((150, 10),))])
def test_fast_path_matches_the_oracles_same_iteration(dtype, d, rank, caches):
    w = small("fast", layers=2, kv_heads=2, G=2, n_obs=6, d=d, dtype=dtype, rank=rank, caches=caches, seed=61)
    arrays = [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    outs, _, st = par.run_gpu(w, arrays, flags=P.binding.OBF_FLAG_FAST_PATH)
    assert st & 0xFF == 0
    worst = 0.0
    for ci in range(len(w.caches)):
        a, out = arrays[ci], outs[ci]
        Qv = a["Q"].reshape(w.layers, w.kv_heads, w.n_q, d)
        diags = P.parse_diag(out["diag"])
        for l in range(w.layers):
            for h in range(w.kv_heads):
                K, V, Q = par.f32_view(a["K"][l, h], dtype), par.f32_view(a["V"][l, h], dtype), par.f32_view(Qv[l, h], dtype)
                ref = oracle.head(K, V, Q, w.caches[ci].budget, rank, fast_iters=3)
                g_idx = out["idx"][l, h].cpu().numpy()
                if not np.array_equal(g_idx, ref["idx"]):
                    continue                                        # a tie inside the band: another valid retained set
                gd = out["delta"][l, h].cpu().numpy().astype(np.float64)
                scale = ref["diag"]["alpha"] * ref["diag"]["rbar_norm"]
                err = np.linalg.norm(gd - ref["delta"])
                worst = max(worst, err / scale)
                # three multiplications by an fp32 Gram matrix whose eigenvalues are within a small factor of each
                # other: the error stays near fp32 rounding (measured: 4e-7 of the scale)
                assert err <= 1e-4 * scale + 1e-6, "delta off by %.3g (scale %.3g)" % (err, scale)
                Vk = V[g_idx].astype(np.float64)
                assert np.abs(Vk @ gd).max() <= 1e-4 * np.linalg.norm(Vk, 2) * np.linalg.norm(gd)
                assert np.linalg.norm(gd) <= scale * (1 + 1e-3)
                dg = diags[l * w.kv_heads + h]
                assert dg["rho_eff"] == ref["diag"]["rho_eff"]
                assert abs(dg["revr"] - ref["diag"]["revr"]) <= 1e-3
                gv = par.out_to_f32(out["V_out"][l, h]).astype(np.float64)
                tol = (2e-3 * scale + 1e-4) if dtype == "f32" else (2e-2 * np.abs(ref["V_out"]) + 2e-3 * scale + 1e-3)
                assert np.all(np.abs(gv - ref["V_out"]) <= tol)
    print("\n[fast path] worst relative delta error %.3g" % worst)


# ---------------------------------------------------------------------------
# few retained rows: the selection copies them itself, with more of them a kernel of its own does
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("dtype,d,flags", [("f32", 64, 0), ("f32", 128, 0), ("bf16", 64, 0), ("bf16", 128, 0),
                                           ("bf16", 128, P.binding.OBF_FLAG_LAYERWISE)])
@pytest.mark.parametrize("caches", [((300, 1),), ((64, 64), (701, 63)), ((1500, 64),), ((300, 65), (90, 7))])
def test_retained_rows_are_copied_whoever_copies_them(dtype, d, flags, caches):
    w = small("copies", layers=2, d=d, dtype=dtype, rank=1, caches=caches, seed=71)
    arrays = [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    for evict in (True, False):
        outs, _, st = par.run_gpu(w, arrays, evict=evict, flags=flags)
        assert st & 0xFF == 0
        for a, o in zip(arrays, outs):
            idx = o["idx"].cpu().numpy()
            assert np.all(np.diff(idx, axis=-1) > 0)
            for l, h in all_heads(w):
                assert np.array_equal(o["K_out"][l, h].float().cpu().numpy(), par.f32_view(a["K"][l, h], dtype)[idx[l, h]])
                if evict:
                    assert np.array_equal(o["V_out"][l, h].float().cpu().numpy(), par.f32_view(a["V"][l, h], dtype)[idx[l, h]])


@pytest.mark.parametrize("dtype,d", [("f32", 64), ("bf16", 64), ("bf16", 128)])
@pytest.mark.parametrize("budgets", [(127,), (128,), (129, 31), (255, 130), (256,), (257,)])
def test_retained_rows_of_few_heads_copied_by_the_selection(dtype, d, budgets):
    # few heads: up to 128 rows of keys and values, up to 256 of the values where a span test waits for them; a full span keeps
    # the values as they are, so that both outputs are copies
    w = small("few", layers=2, d=d, dtype=dtype, rank=1, caches=tuple((700, b) for b in budgets), seed=72)
    arrays = [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    for evict in (True, False):
        outs, _, st = par.run_gpu(w, arrays, evict=evict)
        assert st & 0xFF == 0
        for a, o, b in zip(arrays, outs, budgets):
            idx = o["idx"].cpu().numpy()
            for l, h in all_heads(w):
                assert np.array_equal(o["K_out"][l, h].float().cpu().numpy(), par.f32_view(a["K"][l, h], dtype)[idx[l, h]])
                if evict or b >= d + 60:
                    assert np.array_equal(o["V_out"][l, h].float().cpu().numpy(), par.f32_view(a["V"][l, h], dtype)[idx[l, h]])


# ---------------------------------------------------------------------------
# selection: masses so close together that one bin of the first count holds most of them (further counts), or spread
# (the bin's keys are ranked at once)
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("flags", [0, P.binding.OBF_FLAG_LAYERWISE, P.binding.OBF_FLAG_SINK(4)])
@pytest.mark.parametrize("T,budget", [(257, 100), (3001, 500), (16384, 1700)])
@pytest.mark.parametrize("spread", [0.0, 1e-5, 1e-3, 0.3])
def test_selection_of_close_masses(flags, T, budget, spread):
    w = small("close", dtype="bf16", d=128, caches=((T, budget),), heavy=0, seed=73)
    a = synth.gen_cache(w, 0)
    a["K"] = synth.to_bf16_bits(synth.bf16_bits_to_f32(a["K"]) * np.float32(spread))
    out = par.run_gpu(w, [a], evict=True, flags=flags)[0][0]
    scores = out["scores"].float().cpu().numpy().reshape(w.kv_heads, T)
    sink = 4 if flags == P.binding.OBF_FLAG_SINK(4) else 0
    for h in range(w.kv_heads):
        s = scores[h].copy()
        if flags == P.binding.OBF_FLAG_LAYERWISE:
            s = scores[0].copy()
            for g in range(1, w.kv_heads):
                s = s + scores[g]
        s[:sink] = np.inf
        idx = out["idx"][0, h].cpu().numpy()
        # the largest masses, the lowest positions among equals
        assert np.array_equal(idx, np.sort(np.lexsort((np.arange(T), -s))[:len(idx)])), (h, spread)


@pytest.mark.parametrize("dtype,d", [("f32", 64), ("bf16", 128)])
def test_int8_copy_of_merged_values(dtype, d):
    w = small("q8m", layers=2, d=d, dtype=dtype, caches=((300, 63), (200, 65), (90, 1)), seed=87)
    arrays = [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    outs, _, st = par.run_gpu(w, arrays, flags=P.binding.OBF_FLAG_MERGE, want_int8=True)
    assert st & 0xFF == 0
    for o in outs:
        for name in ("K", "V"):
            codes, scales = oracle.quantize_rows(o[name + "_out"].float().cpu().numpy())
            assert np.array_equal(o[name + "_q8"].cpu().numpy(), codes) and np.array_equal(o[name + "_scale"].cpu().numpy(), scales)


# ---------------------------------------------------------------------------
# query rows of a head: up to 32 (64) of a tile are worked on as four (two) copies, each on its share of the keys
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("n_obs", [1, 16, 17, 32, 33, 64, 65, 80, 81, 96, 97, 128])
def test_query_rows(d, n_obs):
    run_and_check(small("rows", G=2, n_obs=n_obs, d=d, dtype="bf16", caches=((700, 40), (129, 20)) * (9 if n_obs == 80 else 1), seed=91))


# ---------------------------------------------------------------------------
# scale of the values: delta is linear in them, and Eq. 2 and Eq. 5 depend on directions only
# ---------------------------------------------------------------------------
def _scaled(a, dtype, factor):
    if dtype == "f32":
        return a * np.float32(factor)
    return synth.to_bf16_bits(synth.bf16_bits_to_f32(a) * np.float32(factor))


def _falling_values(w, seed):
    """Values whose channels fall off by 0.7 each (eigenvalues of the residual a factor of two apart), down to 1e-2."""
    d, rng = w.head.head_dim, np.random.default_rng(seed)
    v = rng.standard_normal((w.layers, w.kv_heads, w.caches[0].T, d)) * np.maximum(0.7 ** np.arange(d), 1e-2)
    return v.astype(np.float32) if w.dtype == "f32" else synth.to_bf16_bits(v.astype(np.float32))


@pytest.mark.parametrize("dtype,d", [("f32", 64), ("f32", 128), ("bf16", 64), ("bf16", 128)])
@pytest.mark.parametrize("rank,flags", [(2, 0), (9, 0), (2, P.binding.OBF_FLAG_FAST_PATH)])
def test_scale_of_the_values_scales_the_backfill(dtype, d, rank, flags):
    w = small("scale", d=d, dtype=dtype, rank=rank, caches=((700, 20),), seed=101)
    a = synth.gen_cache(w, 0)
    a["V"] = _falling_values(w, 102)
    params = par.params_for(w, None, flags)
    params.eps = 0.0                                                 # (the epsilon of Eq. 4 and Eq. 6 has a scale of its own)

    def run(arrays):
        dev = {name: par.to_device(arrays[name], dtype) for name in "KVQ"}
        out = P.compress_caches(params, [dict(dev, budget=w.caches[0].budget)])[0]
        torch.cuda.synchronize()
        assert P.obf_last_device_status(out["workspace"]) & 0xFF == 0
        return out["idx"].cpu().numpy(), out["delta"].cpu().numpy().astype(np.float64)

    idx, want = run(a)
    assert np.all(np.linalg.norm(want, axis=-1) > 0)
    rows = np.median(np.linalg.norm(par.f32_view(a["V"], dtype), axis=-1))
    # (the last two: retained rows on both sides of the norms 1e-12 and 1e12, where the kernel begins to rescale rows)
    exps = (-45, 32, round(np.log2(1e-12 / rows)), round(np.log2(1e12 / rows)))
    runs = [(2.0 ** e, dict(a, V=_scaled(a["V"], dtype, 2.0 ** e))) for e in exps]
    tiny = a["V"].copy()                                             # the retained rows alone: the same span
    for h in range(w.kv_heads):
        tiny[0, h, idx[0, h]] = _scaled(a["V"][0, h, idx[0, h]], dtype, 2.0 ** -66)
    runs.append((1.0, dict(a, V=tiny)))
    for factor, b in runs:
        got = run(b)[1] / factor
        # fp32 rounding against eigenvalues that lie apart by a tenth of the largest or more down to the second, and by
        # 0.5^9 of it at the ninth: 2^-24 / 0.002 = 3e-5, times three for the roundings of G and of the solve
        err = np.linalg.norm(got - want, axis=-1)
        tol = 1e-4 * np.linalg.norm(want, axis=-1)
        if dtype == "bf16":
            # the retained rows' share is taken out of fp32 sums over all rows: a few ulps of the largest retained value
            tol += 2.0 ** -22 * np.array([np.linalg.norm(par.f32_view(a["V"][0, h], dtype)[idx[0, h]], axis=-1).max() for h in range(w.kv_heads)])
        assert np.all(err <= tol), (factor, err, tol)


@pytest.mark.parametrize("large", [10.0, 1000.0])
@pytest.mark.parametrize("flags", [0, P.binding.OBF_FLAG_EARLY_OUT])
def test_heads_of_64_channels_keep_their_precision_beside_large_retained_values(large, flags):
    # the sums of Eq. 3 and Eq. 4 run over the deleted rows alone: retained values a thousand times as large leave no trace in
    # them.  Retained tokens lie anywhere in the tiles of 128, the last tile is ragged, and budgets on both sides of 64 take
    # both copies of the retained rows
    w = small("large64", layers=2, d=64, dtype="bf16", rank=2, caches=((700, 20), (129, 33), (128, 9), (1500, 64)), seed=107)
    arrays = [synth.gen_cache(w, ci) for ci in range(len(w.caches))]
    for ci, a in enumerate(arrays):
        T, rng = w.caches[ci].T, np.random.default_rng(ci)
        # (eigenvalues about 16 : 4 : 0.25 and no small ones, so that the retained rows' span is well conditioned)
        V = rng.standard_normal((w.layers, w.kv_heads, T, 64)) * np.array([4.0, 2.0] + 62 * [0.5])
        Qv = a["Q"].reshape(w.layers, w.kv_heads, w.n_q, 64)
        for l, h in all_heads(w):
            A = oracle.scores(par.f32_view(a["K"][l, h], "bf16"), par.f32_view(Qv[l, h], "bf16"))
            # (of the cache with a budget of head_dim all retained rows are multiples of one another)
            idx = oracle.topk(A, w.caches[ci].budget)[0]
            V[l, h, idx] = large * (V[l, h, idx] if w.caches[ci].budget < 64 else V[l, h, idx[:1]])
        a["V"] = synth.to_bf16_bits(V.astype(np.float32))
    outs, _, st = par.run_gpu(w, arrays, flags=flags)
    assert st & 0xFF == 0
    for a, o in zip(arrays, outs):
        for l, h in all_heads(w):
            ref = oracle.backfill(par.f32_view(a["K"][l, h], "bf16"), par.f32_view(a["V"][l, h], "bf16"),
                                  o["scores"][l, h].cpu().numpy().astype(np.float64), o["idx"][l, h].cpu().numpy(), w.rank)
            gap = (ref["diag"]["lam_rho"] - ref["diag"]["lam_next"]) / ref["diag"]["lam_1"]
            err = np.linalg.norm(o["delta"][l, h].cpu().numpy().astype(np.float64) - ref["delta"]) / np.linalg.norm(ref["delta"])
            # 64 fp32 roundings over the distance of the subspace from the rest (measured before the tensor cores took
            # these heads over: 1e-6)
            assert err <= 64 * par.U32 / gap, (l, h, err, gap)


@pytest.mark.parametrize("T,n_obs", [(128, 1), (700, 1), (2049, 1), (700, 2)])
def test_softmax_rows_of_heads_of_64_channels_add_up_to_one(T, n_obs):
    # with logits of 100 (base 2) a normaliser kept as a logarithm would be rounded to 2^-18: the same error in every weight of
    # the row.  What is left is the exponential's own 2^-22.5, once in the sum and once in a weight that may be most of the row,
    # and three roundings
    w = small("rows64", d=64, dtype="bf16", rank=0, kv_heads=8, G=1, n_obs=n_obs, caches=((T, 20),), seed=109)
    a = synth.gen_cache(w, 0)
    K, Q = par.f32_view(a["K"], "bf16")[0], par.f32_view(a["Q"], "bf16")[0]
    top = np.abs(np.einsum("htd,hqd->hqt", K, Q)).max(axis=(1, 2)) / 8.0 * np.log2(np.e)
    a["Q"] = synth.to_bf16_bits((Q * (100.0 / top)[:, None, None]).astype(np.float32))[None]
    out = par.run_gpu(w, [a], evict=True)[0][0]
    rows = out["scores"].cpu().numpy().astype(np.float64)[0].sum(axis=-1)
    assert np.all(np.abs(rows / n_obs - 1.0) <= 2 * 2.0 ** -22.5 + 3 * par.U32), rows - n_obs


# ---------------------------------------------------------------------------
# the masses of a head depend on the head alone: not on the other heads of the call, the slabs it is cut into or the scratch
# ---------------------------------------------------------------------------
def _random_caches(layers, kv_heads, G, n_obs, d, Ts, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    return [{"K": torch.randn((layers, kv_heads, T, d), generator=g, device="cuda").mul_(2.0).to(tdt),
             "V": torch.randn((layers, kv_heads, T, d), generator=g, device="cuda").to(tdt),
             "Q": torch.randn((layers, kv_heads * G, n_obs, d), generator=g, device="cuda").mul_(2.0).to(tdt)} for T in Ts]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("Ts", [(64, 129), (300, 2100), (1024, 5000), (257,)])
def test_masses_do_not_depend_on_the_other_heads_of_the_call(dtype, Ts):
    # fp32, and bf16 on the shape-generic kernels: 40 layers x 4 heads against their last layer alone
    flags = 0 if dtype == "f32" else P.binding.OBF_FLAG_GENERIC_PATH
    dt = P.OBF_F32 if dtype == "f32" else P.OBF_BF16
    dev = _random_caches(40, 4, 2, 33, 64, Ts, dtype, 113)
    lse = [torch.randn((40, 8, 33), device="cuda") for _ in Ts]
    whole = P.compress_caches(P.make_params(40, 4, 8, 64, 33, 0, dt, flags=flags),
                              [dict(x, budget=20, lse_extra=e) for x, e in zip(dev, lse)], evict=True, want_scores=True)
    for ci, (x, e) in enumerate(zip(dev, lse)):
        part = {name: t[-1:].contiguous() for name, t in x.items()}
        for heads in (slice(0, 4), slice(2, 3)):
            one = {"K": part["K"][:, heads].contiguous(), "V": part["V"][:, heads].contiguous(),
                   "Q": part["Q"][:, 2 * heads.start:2 * heads.stop].contiguous(),
                   "lse_extra": e[-1:, 2 * heads.start:2 * heads.stop].contiguous()}
            n = heads.stop - heads.start
            out = P.compress_caches(P.make_params(1, n, 2 * n, 64, 33, 0, dt, flags=flags), [dict(one, budget=20)],
                                    evict=True, want_scores=True)[0]
            assert torch.equal(out["scores"], whole[ci]["scores"][-1:, heads])
            assert torch.equal(out["idx"], whole[ci]["idx"][-1:, heads])


def test_host_entry_point_on_fp32_layers_matches_the_device_entry_point():
    # 37 layers: slabs of 9 and 10, whose heads share the chip differently from those of the whole call
    dev = _random_caches(37, 8, 1, 8, 64, (700,), "f32", 117)[0]
    params = P.make_params(37, 8, 8, 64, 8, 2, P.OBF_F32)
    ref = P.compress_caches(params, [dict(dev, budget=12)], want_scores=True)[0]
    h = {n: t.cpu().pin_memory() for n, t in dev.items()}
    oK, oV = torch.empty((37, 8, 12, 64)).pin_memory(), torch.empty((37, 8, 12, 64)).pin_memory()
    oI, oS = torch.empty((37, 8, 12), dtype=torch.int32).pin_memory(), torch.empty((37, 8, 700)).pin_memory()
    c = P.make_cache(h["K"], h["V"], h["Q"], 700, 12, oK, oV, oI, None, oS)
    arena = torch.empty(P.obf_host_arena_bytes(params, [c]), dtype=torch.uint8, device="cuda")
    P.obf_compress_host(params, [c], arena)
    assert torch.equal(oS, ref["scores"].cpu()) and torch.equal(oI, ref["idx"].cpu()) and torch.equal(oK, ref["K_out"].cpu())
    assert torch.allclose(oV, ref["V_out"].cpu(), rtol=1e-4, atol=4e-6)


# ---------------------------------------------------------------------------
# calls of different shapes from several host threads: a kernel's shared-memory limit is one for all of them
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("what", ["selection", "algebra"])
def test_threads_with_different_shared_memory_needs(what):
    # long against short prompts (64 KB of selection keys or 1 KB); full eigen-decompositions against a single vector (200 KB or
    # 60 KB of the dense algebra).  Every call has to be accepted
    import threading
    shapes = [(16384, 20, 0, 64), (256, 20, 0, 64)] if what == "selection" else [(200, 20, 9, 128), (200, 2, 1, 128)]
    failures, start = [], threading.Barrier(len(shapes))

    def worker(T, budget, rank, d):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            x = _random_caches(1, 1, 1, 1, d, (T,), "f32", 127)[0]
            params = P.make_params(1, 1, 1, d, 1, rank, P.OBF_F32)
            out = P.compress_caches(params, [dict(x, budget=budget)], stream=stream)[0]
            stream.synchronize()
            start.wait()
            for i in range(600 if what == "selection" else 100):
                rc = P.obf_compress(params, out["cache_structs"], out["workspace"], stream=stream, check=False)
                if rc != P.binding.OBF_OK:
                    failures.append((T, rank, i, rc))
                    break
            stream.synchronize()

    threads = [threading.Thread(target=worker, args=s) for s in shapes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures


def test_a_call_that_fails_halfway_leaves_no_work_unjoined():
    # More heads than a grid has rows: the copy of the retained rows is refused at its launch, after the call has forked to the
    # library's stream.  The call is captured and the graph never launched, so nothing runs; a fork that is not joined again
    # would make the end of the capture fail.
    n = 65536
    params = P.make_params(n, 1, 1, 128, 1, 1, P.OBF_BF16)
    buf = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    ptr = (buf.data_ptr() + 255) // 256 * 256
    cache = P.make_cache(ptr, ptr, ptr, 256, 130, ptr, ptr, ptr)
    warm = small("warm", d=128, dtype="bf16", caches=((256, 130),))       # (streams and events exist before the capture)
    par.run_gpu(warm, [synth.gen_cache(warm, 0)])
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph(keep_graph=True)                         # (never instantiated)
    rc = None
    with torch.cuda.graph(graph, stream=stream):
        rc = P.obf_compress(params, [cache], ptr, P.obf_workspace_bytes(params, [cache]), stream=stream, check=False)
    assert rc == P.binding.OBF_ERR_CUDA
    del graph
    ok = par.run_gpu(warm, [synth.gen_cache(warm, 0)])                    # the next call is accepted
    assert ok[2] & 0xFF == 0


@pytest.mark.parametrize("d,G,n_obs,caches", [
    (128, 1, 1, ((128, 9), (256, 9), (257, 9), (385, 9))),          # one query, whole and barely begun chunks of 256 keys and halves
    (128, 2, 16, ((129, 9), (160, 9), (1025, 9))),                  # 32 queries: four copies, a piece of 32 keys with one key
    (128, 3, 11, ((255, 9), (300, 9))),                             # 33: two copies
    (64, 8, 8, ((383, 9), (512, 9))),                               # 64
    (64, 5, 13, ((287, 9),)),                                       # 65: one copy, an odd number of queries
    (128, 8, 16, ((4100, 9), (140, 9))),                            # 128, more than sixteen chunks of a head
    (64, 3, 43, ((200, 9), (4400, 9))),                             # 129: a second tile of one query
    (128, 8, 32, ((8500, 9),)),                                     # 256, chunks fetched in two sweeps
])
def test_score_kernel_at_the_edges_of_its_chunks_pieces_and_copies(d, G, n_obs, caches):
    # masses, positions and outputs against the oracle (run_and_check: 2e-7 + 1e-5 of the mass, fp32 sums and exponentials)
    w = small("chunks", layers=1, kv_heads=3, G=G, n_obs=n_obs, d=d, dtype="bf16", rank=1, caches=caches, n_outlier=3, n_sink=4,
              heavy=5, seed=900 + G * n_obs)
    a, _, _ = run_and_check(w)
    assert "k_score_tc" in [n for n, _ in P.obf_compress_profiled(par.params_for(w), a[0]["cache_structs"], a[0]["workspace"])]


def test_masses_of_a_head_do_not_depend_on_the_rest_of_the_call():
    # chunks are dealt over the whole call: the order in which a row's statistics are added is the head's alone
    g = torch.Generator(device="cuda").manual_seed(3)
    K, V, Q = (torch.randn((5, 4, rows, 128), generator=g, device="cuda", dtype=torch.bfloat16) for rows in (2900, 2900, 40))
    params = P.make_params(5, 4, 4, 128, 40, 0, P.OBF_BF16)
    whole = P.compress_caches(params, [dict(K=K, V=V, Q=Q, budget=30)], evict=True, want_scores=True)[0]
    for l in range(5):
        one = [x[l:l + 1].contiguous() for x in (K, V, Q)]
        part = P.compress_caches(P.make_params(1, 4, 4, 128, 40, 0, P.OBF_BF16), [dict(K=one[0], V=one[1], Q=one[2], budget=30)],
                                 evict=True, want_scores=True)[0]
        assert torch.equal(part["scores"][0], whole["scores"][l]) and torch.equal(part["idx"][0], whole["idx"][l])


@pytest.mark.parametrize("caches", [((300, 1), (200, 31)), ((700, 32), (161, 33)), ((400, 63),), ((130, 130), (500, 40))])
@pytest.mark.parametrize("rank", [2, 9])
def test_reflectors_found_beside_the_pass_over_values(caches, rank):
    # bf16 heads of 64 channels, every budget below 64 (but in the last case, whose first cache is kept whole): batches of 32 rows
    # with remainders, the tridiagonal and the Jacobi route of the dense algebra behind them
    w = small("rows", layers=2, kv_heads=3, G=4, n_obs=4, d=64, dtype="bf16", rank=rank, caches=caches, seed=61 + rank)
    a, _, _ = run_and_check(w)
    names = [n for n, _ in P.obf_compress_profiled(par.params_for(w), a[0]["cache_structs"], a[0]["workspace"])]
    assert ("k_obf_rows" in names) == all(min(b, T) < 64 for T, b in caches)


@pytest.mark.parametrize("G,n_obs,d", [(1, 20, 128), (2, 25, 64), (4, 25, 128), (3, 50, 64)])      # four copies, two, one, a second tile
def test_masses_of_a_head_do_not_depend_on_the_number_of_caches(G, n_obs, d):
    # seventeen caches: more than the score kernel has two tensor maps of the queries for
    caches = tuple((129 + 71 * i, 9) for i in range(17))
    w = small("many", layers=1, kv_heads=2, G=G, n_obs=n_obs, d=d, dtype="bf16", rank=1, caches=caches, heavy=5, seed=300 + n_obs)
    a, _, arrays = run_and_check(w)
    for ci in range(17):
        one = dataclasses.replace(w, caches=(w.caches[ci],))
        b, _, st = par.run_gpu(one, [arrays[ci]])
        assert st & 0xFF == 0
        assert torch.equal(a[ci]["scores"], b[0]["scores"]) and torch.equal(a[ci]["idx"], b[0]["idx"]), ci


@pytest.mark.parametrize("d", [64, 128])
def test_a_wait_that_runs_out_between_two_query_tiles(d):
    # every slot has a second tile of queries to load and multiply when the wait of the first one runs out (20 ms): the block lets
    # what it started come to its end, and the call after it finds everything as it should be
    w = small("expire2", layers=1, kv_heads=4, G=8, n_obs=32, d=d, dtype="bf16", rank=1, caches=((2000, 40),), heavy=5, seed=17)
    arrays = [synth.gen_cache(w, 0)]
    outs, dev, st = par.run_gpu(w, arrays, flags=P.binding.OBF_FLAG_TEST_WAIT_EXPIRES)
    assert st & P.binding.OBF_DEV_TIMEOUT
    ws = outs[0]["workspace"]
    good = P.compress_caches(par.params_for(w), dev, want_scores=True, workspace=ws)
    torch.cuda.synchronize()
    assert P.obf_last_device_status(ws) & 0xFF == 0
    par.check_cache(w, 0, arrays[0], good[0], all_heads(w))


@pytest.mark.parametrize("d,G,n_obs,caches", [
    (128, 2, 16, ((8192, 9), (8193, 9), (300, 9))),                # 32 chunks: folded in one step; 33: a last sixteen of one; a short one
    (64, 4, 32, ((12288, 9),)),                                    # three whole sixteens
    (128, 4, 40, ((12289, 9),)),                                   # and a chunk more, with two tiles of queries
    (64, 1, 50, ((75776, 9),)),                                    # as many as there are slots on 148 multiprocessors
])
def test_score_kernel_folds_long_heads_in_two_steps(d, G, n_obs, caches):
    w = small("longer", layers=1, kv_heads=2, G=G, n_obs=n_obs, d=d, dtype="bf16", rank=1, caches=caches, n_outlier=3, n_sink=4,
              heavy=5, seed=700 + n_obs)
    a, _, arrays = run_and_check(w)
    assert "k_score_tc" in [n for n, _ in P.obf_compress_profiled(par.params_for(w), a[0]["cache_structs"], a[0]["workspace"])]
    for ci, c in enumerate(w.caches):                              # the masses of a head do not depend on the length of the others
        b, _, _ = par.run_gpu(dataclasses.replace(w, caches=(c,)), [arrays[ci]])
        assert torch.equal(a[ci]["scores"], b[0]["scores"]) and torch.equal(a[ci]["idx"], b[0]["idx"])


@pytest.mark.parametrize("d,G,n_obs", [(64, 4, 7), (128, 4, 8), (64, 4, 15), (128, 4, 16), (64, 4, 32), (128, 4, 32), (64, 4, 40), (128, 8, 32)])
def test_score_kernel_reuses_its_slots(d, G, n_obs):
    # 48 heads of (2 + 3 + 6) + 8 chunks are 912, three for every slot: both slots of a block, their buffers and barriers met again by
    # last chunks of one half (300 = 256 + 44, 1380 = 5 * 256 + 100) and of two (700 = 2 * 256 + 188, 1950 = 7 * 256 + 158); four, two
    # and one copies, two tiles
    caches = ((300, 9), (700, 9), (1380, 9), (1950, 9))
    w = small("slots", layers=6, kv_heads=8, G=G, n_obs=n_obs, d=d, dtype="bf16", rank=1, caches=caches, heavy=3, n_outlier=3,
              seed=40 + n_obs + d)
    _, reps, _ = run_and_check(w, evict=True, heads=[(l, (3 * l + 1) % 8) for l in range(6)] + [(5, 7)])
    assert len(reps) == 7 * len(caches)


def test_masses_of_a_head_do_not_depend_on_the_other_heads_of_its_slots():
    # 800 chunks of ten a head: slots are used again, and by which chunk follows from all that comes before
    g = torch.Generator(device="cuda").manual_seed(4)
    K, V, Q = (torch.randn((10, 8, rows, 64), generator=g, device="cuda", dtype=torch.bfloat16) for rows in (2500, 2500, 70))
    whole = P.compress_caches(P.make_params(10, 8, 8, 64, 70, 0, P.OBF_BF16), [dict(K=K, V=V, Q=Q, budget=30)], evict=True, want_scores=True)[0]
    for l in range(10):
        one = [x[l:l + 1].contiguous() for x in (K, V, Q)]
        part = P.compress_caches(P.make_params(1, 8, 8, 64, 70, 0, P.OBF_BF16), [dict(K=one[0], V=one[1], Q=one[2], budget=30)],
                                 evict=True, want_scores=True)[0]
        assert torch.equal(part["scores"][0], whole["scores"][l]) and torch.equal(part["idx"][0], whole["idx"][l])
