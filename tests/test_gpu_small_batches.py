"""Parity of the kernel that shares a row between the CTAs of a cluster (batches of up to 74 rows on a
148-SM device), at the batch sizes where the number of CTAs per row changes and at row lengths where
slices, tables and lists have their edges."""
import os

import numpy as np
import pytest
import torch

from oracle import albireo_oracle as O
from paper_2606_01927_b200 import workloads as W

from parity import compare, compare_top_lists, to_host

pytestmark = pytest.mark.gpu

DBG_CAP = 128
_CORES = len(os.sched_getaffinity(0))


@pytest.fixture(scope="module")
def binding():
    from paper_2606_01927_b200 import binding as Bd
    return Bd


@pytest.fixture(scope="module")
def sampler(binding):
    s = binding.Sampler(max_rows=128, max_vocab=160000, max_history_total=1 << 21)
    yield s
    s.close()


def check(binding, sampler, w, flags=0, **kw):
    ref = O.sample(w, threads=_CORES, topk_cap=DBG_CAP)
    t = binding.workload_tensors(w, sampler.device)
    out = sampler.albireo_sample(t.pop("logits"), **t, row_base=w.row_base, num_top=w.num_top, want_counts=True,
                                 dbg_cap=DBG_CAP, want_status=True, flags=flags, **kw)
    torch.cuda.synchronize()
    g = to_host(out)
    rep = compare(w, g, ref, dbg_cap=DBG_CAP)
    assert rep.ok() and not rep.excused, (rep.summary(), rep.failures[:3], rep.excused[:3])
    bad = compare_top_lists(w, g, ref)
    assert not bad, bad[:3]
    return g, ref


# rows per batch around 148 / 16, 148 / 8, 148 / 4 and 148 / 2; lengths with 0 to 14 unaligned ends, one
# vector more or less than a slice boundary, and slices that end up empty
@pytest.mark.parametrize("dtype", [W.F32, W.BF16, W.F16])
@pytest.mark.parametrize("B,V", [(1, 65536), (9, 65537), (10, 65543), (18, 32775), (19, 16391), (37, 33001), (38, 16384),
                                 (74, 8191 * 2), (75, 16384), (3, 131073 + 8)])
def test_mixed_requests_at_the_edges(binding, sampler, B, V, dtype):
    base = W.random_small(1000 + B, B=B, V=V, dtype=W.F32 if dtype == W.F16 else dtype)
    w = W.as_f16(base) if dtype == W.F16 else base
    w.num_top = 5
    check(binding, sampler, w)


@pytest.mark.parametrize("dtype", [W.F32, W.BF16])
@pytest.mark.parametrize("kind", ["topk", "topk_wide", "minp_wide", "topp", "topp_one", "none", "flat"])
def test_rows_without_histories(binding, sampler, dtype, kind):
    """No tables behind the slices; rows off the 16-byte grid, so that CTA 0 lists their ends; rows of
    ties, whose window of the top-p cut has to be split down to single codes."""
    B, V = 23, 33271
    rng = np.random.default_rng(7)
    x = (rng.standard_normal((B, V)) * 2).astype(np.float32)
    if kind == "flat":
        x = np.round(x).astype(np.float32)
        x[0] = 1.5
    par = {"topk": dict(top_k=np.full(B, 40, np.int32)),
           "topk_wide": dict(top_k=np.full(B, 250, np.int32), top_p=np.full(B, 0.9, np.float32)),
           "minp_wide": dict(min_p=np.full(B, 0.004, np.float32), top_p=np.full(B, 0.9, np.float32)),
           "topp": dict(top_p=np.linspace(0.05, 0.999, B).astype(np.float32)),
           "topp_one": dict(top_p=np.zeros(B, np.float32)),
           "none": dict(), "flat": dict(top_p=np.full(B, 0.7, np.float32))}[kind]
    w = W.Workload(kind, B, V, dtype, x if dtype == W.F32 else W.f32_to_bf16_bits(x),
                   temperature=np.full(B, 0.9, np.float32), seeds=np.arange(B, dtype=np.uint64), **par)
    w.num_top = 0 if kind == "none" else 7
    if kind == "flat":
        w.num_top = 0
    check(binding, sampler, w)


def test_a_slice_with_more_distinct_history_ids_than_it_lists(binding, sampler):
    """Ids packed into the head of the vocabulary: one slice has more of them than its list holds (that row
    goes to one CTA), another row just fits, a third repeats the row's unaligned ends."""
    B, V = 4, 120001
    rng = np.random.default_rng(9)
    x = (rng.standard_normal((B, V)) * 2).astype(np.float32)
    rows = [rng.permutation(4000)[:1500], rng.permutation(3500)[:1008], np.array([0, 1, V - 1, V - 1, V - 2, 5, -1, V]), rng.integers(0, V, 9000)]
    off = np.cumsum([0] + [len(r) for r in rows]).astype(np.int32)
    w = W.Workload("dense", B, V, W.BF16, W.f32_to_bf16_bits(x), temperature=np.ones(B, np.float32),
                   top_k=np.array([50, 50, 50, 0], np.int32), top_p=np.full(B, 0.9, np.float32),
                   repetition_penalty=np.full(B, 1.3, np.float32), presence_penalty=np.full(B, 0.4, np.float32),
                   frequency_penalty=np.full(B, 0.2, np.float32), history_ids=np.concatenate(rows).astype(np.int32),
                   history_offsets=off, seeds=np.arange(B, dtype=np.uint64))
    check(binding, sampler, w)


@pytest.mark.parametrize("cut", ["topk", "greedy", "topp", "none"])
def test_full_vocabulary_list(binding, sampler, cut):
    w = W.random_small(1100, B=12, V=40003, dtype=W.BF16)
    w.top_k[:] = 3 if cut == "topk" else 0
    w.top_p[:] = 0.6 if cut == "topp" else 1.0
    w.min_p[:] = 0.0
    w.temperature[:] = 0.0 if cut == "greedy" else 0.8
    w.logprob_full_vocab = True
    w.num_top = 128
    check(binding, sampler, w, flags=binding.FLAG_LOGPROB_FULL_VOCAB)


# ------------------------------------------------------------------ the same rows by one CTA each (batches above 74 rows)

@pytest.mark.parametrize("dtype", [W.F32, W.BF16])
@pytest.mark.parametrize("B,V", [(76, 1000), (80, 16385), (100, 33000)])
def test_mixed_requests_one_cta_per_row(binding, sampler, B, V, dtype):
    w = W.random_small(1200 + B, B=B, V=V, dtype=dtype)
    w.num_top = 5
    check(binding, sampler, w)


@pytest.mark.parametrize("B", [2, 76])
@pytest.mark.parametrize("cut", ["ties", "tail", "none"])
def test_cuts_among_ties_and_far_down_the_tail(binding, sampler, B, cut):
    """A vocabulary whose bulk falls on a few dozen bf16 values (thousands of equal scores at the cut), and
    top-p close to 1 on a long tail."""
    V = 60001
    rng = np.random.default_rng(31)
    x = (rng.standard_normal((B, V)) * 2 - (40.0 if cut == "ties" else 0.0)).astype(np.float32)
    p = {"ties": np.linspace(0.3, 0.97, B), "tail": 1.0 - np.logspace(-2, -5, B), "none": np.ones(B)}[cut].astype(np.float32)
    w = W.Workload(cut, B, V, W.BF16, W.f32_to_bf16_bits(x), temperature=np.full(B, 1.2, np.float32), top_p=p,
                   seeds=np.arange(B, dtype=np.uint64))
    g, ref = check(binding, sampler, w)


@pytest.mark.parametrize("dtype", [W.F32, W.BF16])
@pytest.mark.parametrize("k", [40, 65, 128, 256])
def test_large_top_k_on_gaussian_rows(binding, sampler, dtype, k):
    """Rows without a dense head: the candidate list has to be looked at while it grows."""
    B, V = 80, 150001
    rng = np.random.default_rng(33)
    x = (rng.standard_normal((B, V)) * 3).astype(np.float32)
    w = W.Workload("gauss", B, V, dtype, x if dtype == W.F32 else W.f32_to_bf16_bits(x), temperature=np.full(B, 0.8, np.float32),
                   top_k=np.full(B, k, np.int32), seeds=np.arange(B, dtype=np.uint64))
    g, _ = check(binding, sampler, w)
    assert (g["row_status"] & 1).sum() == 0            # every row on the single-pass path


@pytest.mark.parametrize("B", [6, 76])
@pytest.mark.parametrize("cut", ["none", "topp", "minp", "none_full", "topp_full"])
@pytest.mark.parametrize("near", [1, 3])
def test_lists_longer_than_what_carries_mass(binding, sampler, B, cut, near):
    """Fewer elements than the list wants lie within 2^-42 of the likeliest one's mass: the list goes on with
    the elements behind the gap wherever they are members."""
    V = 20011
    rng = np.random.default_rng(41)
    x = rng.standard_normal((B, V)).astype(np.float32)
    for b in range(B):
        x[b, rng.permutation(V)[:near]] = 14.0 + rng.random(near).astype(np.float32)
    par = {"topp": dict(top_p=np.full(B, 0.9, np.float32)), "minp": dict(min_p=np.full(B, 1e-30, np.float32))}.get(cut.split("_")[0], {})
    w = W.Workload(cut, B, V, W.BF16, W.f32_to_bf16_bits(x), temperature=np.full(B, 0.25, np.float32),
                   seeds=np.arange(B, dtype=np.uint64), **par)
    w.num_top = 5
    w.logprob_full_vocab = cut.endswith("full")
    _, ref = check(binding, sampler, w, flags=binding.FLAG_LOGPROB_FULL_VOCAB if w.logprob_full_vocab else 0)
    if cut != "topp":
        assert (ref.top_ids >= 0).all()


@pytest.mark.parametrize("B", [6, 76])
@pytest.mark.parametrize("dtype", [W.F32, W.BF16])
@pytest.mark.parametrize("T", [0.5, 1.0, 1.7])
@pytest.mark.parametrize("flags", [0, 1], ids=["auto", "general"])
def test_masks_of_the_lowest_value(binding, sampler, B, dtype, T, flags):
    """Tokens masked with the type's lowest finite value: below T = 1 their scores leave the fp32 range and are
    not among the finite ones; sizes of the kept set and of the top-k stage are the oracle's."""
    V = 20003
    rng = np.random.default_rng(43)
    x = rng.standard_normal((B, V)).astype(np.float32)
    low = np.float32(-3.4028234663852886e38 if dtype == W.F32 else -3.3895313892515355e38)
    x[rng.random((B, V)) < 0.9] = low
    x[0] = low
    x[0, 4321] = 1.0
    p = np.where(np.arange(B) % 3 == 0, 1.0, 0.9).astype(np.float32)
    w = W.Workload("masked", B, V, dtype, x if dtype == W.F32 else W.f32_to_bf16_bits(x), temperature=np.full(B, T, np.float32),
                   top_p=p, seeds=np.arange(B, dtype=np.uint64))
    g, ref = check(binding, sampler, w, flags=flags)
    assert (g["num_topk"] == ref.rows["n_topk"]).all()
    assert (g["num_kept"][p == 1.0] == ref.rows["n_keep"][p == 1.0]).all()


@pytest.mark.parametrize("B", [6, 76])
@pytest.mark.parametrize("dtype", [W.F32, W.BF16])
@pytest.mark.parametrize("cut", ["none", "topk", "full"])
@pytest.mark.parametrize("flags", [0, 1], ids=["auto", "general"])
def test_lists_and_top_k_reach_into_masks_of_the_lowest_value(binding, sampler, B, dtype, cut, flags):
    """More entries wanted than tokens are left unmasked: the masked ones follow in the order of their ids."""
    V = 20003
    rng = np.random.default_rng(44)
    x = np.full((B, V), -3.4028234663852886e38 if dtype == W.F32 else -3.3895313892515355e38, np.float32)
    for b in range(B):
        x[b, rng.permutation(V)[:1 + b % 7]] = rng.standard_normal(1 + b % 7).astype(np.float32)
    w = W.Workload("masked", B, V, dtype, x if dtype == W.F32 else W.f32_to_bf16_bits(x), temperature=np.ones(B, np.float32),
                   top_k=np.full(B, 30 if cut == "topk" else 0, np.int32), seeds=np.arange(B, dtype=np.uint64))
    w.num_top = 20
    w.logprob_full_vocab = cut == "full"
    g, ref = check(binding, sampler, w, flags=flags | (binding.FLAG_LOGPROB_FULL_VOCAB if cut == "full" else 0))
    assert (g["num_kept"] == ref.rows["n_keep"]).all() and (ref.top_ids >= 0).all()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("cut", ["topp", "none", "minp_topp", "topp_full", "topk_full"])
def test_results_do_not_depend_on_where_a_row_lies(binding, sampler, dtype, cut):
    """The same rows in batches of other sizes (one CTA per row, clusters of several sizes) and on other offsets from
    the 16-byte grid, with cuts down the tail where an element weighs 1e-6 of the sum: sums are of integers, so
    tokens, kept sizes and log-probabilities are the same bit for bit."""
    B, V = 96, 40009
    g = torch.Generator(device=sampler.device).manual_seed(5)
    x = (torch.randn((B, V), generator=g, device=sampler.device) * 1.5).to(dtype)
    par = dict(temperature=torch.full((B,), 0.9, device=sampler.device), seeds=torch.arange(B, device=sampler.device) * 7 + 1)
    if "topp" in cut:
        par["top_p"] = (1.0 - torch.logspace(-1, -4, B, device=sampler.device)).float()
    if "minp" in cut:
        par["min_p"] = torch.full((B,), 1e-4, device=sampler.device)
    if "topk" in cut:
        par["top_k"] = torch.full((B,), 30, dtype=torch.int32, device=sampler.device)
    flags = binding.FLAG_LOGPROB_FULL_VOCAB if cut.endswith("full") else 0
    whole = to_host(sampler.albireo_sample(x, **par, want_counts=True, flags=flags))
    for lo, n, shift in [(0, 96, 3), (0, 5, 0), (5, 9, 1), (14, 17, 7), (30, 36, 2), (22, 74, 5)]:
        buf = torch.zeros((n * (V + shift) + 8,), dtype=dtype, device=sampler.device)
        view = buf[shift:shift + n * (V + shift)].view(n, V + shift)[:, :V]
        view.copy_(x[lo:lo + n])
        part = to_host(sampler.albireo_sample(view, **{k: v[lo:lo + n] for k, v in par.items()}, row_base=lo, want_counts=True, flags=flags))
        for f in ("tokens", "num_kept", "num_topk"):
            assert (part[f] == whole[f][lo:lo + n]).all(), (f, lo, n, shift)
        assert (part["logprobs"].view(np.uint32) == whole["logprobs"][lo:lo + n].view(np.uint32)).all(), (lo, n, shift)


@pytest.mark.parametrize("dtype", [W.F32, W.BF16])
@pytest.mark.parametrize("extras", [True, False])
def test_top_k_with_a_min_p_floor_that_rises(binding, sampler, dtype, extras):
    """A long candidate list cut at the k-th largest key while the warps have seen different min-p floors."""
    B, V = 120, 68066
    rng = np.random.default_rng(47)
    x = (rng.standard_normal((B, V))).astype(np.float32)
    x[rng.random((B, V)) > 0.02] = -np.inf
    w = W.Workload("topk_minp", B, V, dtype, x if dtype == W.F32 else W.f32_to_bf16_bits(x), temperature=np.ones(B, np.float32),
                   top_k=np.full(B, 200, np.int32), min_p=np.full(B, 0.04, np.float32), top_p=np.linspace(0.3, 0.95, B).astype(np.float32),
                   seeds=np.arange(B, dtype=np.uint64))
    w.num_top = 100
    if extras:
        g, ref = check(binding, sampler, w)
        assert (g["num_kept"] == ref.rows["n_keep"]).sum() >= B - 2
        return
    ref = O.sample(w, threads=_CORES)
    t = binding.workload_tensors(w, sampler.device)
    g = to_host(sampler.albireo_sample(t.pop("logits"), **t, num_top=w.num_top))
    rep = compare(w, g, ref)
    assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3])


@pytest.mark.parametrize("B", [8, 80])
@pytest.mark.parametrize("dtype", [W.F32, W.BF16])
@pytest.mark.parametrize("cut", ["none", "topp", "topk_full"])
def test_masses_of_scores_far_from_zero(binding, sampler, B, dtype, cut):
    """Scores around 1000 / T, where the product with 1 / T is rounded by 1e-4 and more: a mass is that of the rounded
    score (as everywhere else), not of the product before its rounding."""
    V = 17011
    rng = np.random.default_rng(53)
    x = (1000.0 + rng.standard_normal((B, V)) * 3).astype(np.float32)
    x[:, ::3] = np.round(x[:, ::3])
    par = dict(none={}, topp=dict(top_p=np.full(B, 0.9, np.float32)), topk_full=dict(top_k=np.full(B, 20, np.int32)))[cut]
    w = W.Workload("far", B, V, dtype, x if dtype == W.F32 else W.f32_to_bf16_bits(x),
                   temperature=np.linspace(0.07, 1.3, B).astype(np.float32), seeds=np.arange(B, dtype=np.uint64), **par)
    w.logprob_full_vocab = cut.endswith("full")
    check(binding, sampler, w, flags=binding.FLAG_LOGPROB_FULL_VOCAB if w.logprob_full_vocab else 0)
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("cut", ["greedy", "topk", "topp", "minp", "none"])
@pytest.mark.parametrize("B", [8, 80])
def test_infinities_and_nan_give_a_token_in_range(binding, sampler, dtype, cut, B):
    """Rows outside the contract (+inf, NaN, nothing finite): the token is unspecified but an id of the row."""
    V = 33001
    g = torch.Generator(device=sampler.device).manual_seed(3)
    x = torch.randn((B, V), generator=g, device=sampler.device).to(dtype)
    x[0] = float("nan")
    x[1] = float("inf")
    x[2] = -float("inf")
    x[3, ::2] = float("inf")
    x[4, ::3] = float("nan")
    x[5, 7] = float("inf")
    x[6, 33000] = float("nan")
    x[7, :100] = float("inf")
    x[7, 100:] = -float("inf")
    par = dict(greedy=dict(temperature=torch.zeros(B, device=sampler.device)), none={},
               topk=dict(top_k=torch.full((B,), 50, dtype=torch.int32, device=sampler.device)),
               topp=dict(top_p=torch.full((B,), 0.9, device=sampler.device)),
               minp=dict(min_p=torch.full((B,), 0.01, device=sampler.device)))[cut]
    pad = torch.zeros((64 + B * V + 64,), dtype=dtype, device=sampler.device)
    view = pad[64:64 + B * V].view(B, V)
    view.copy_(x)
    for flags in (0, binding.FLAG_FORCE_GENERAL, binding.FLAG_LOGPROB_FULL_VOCAB):
        for num_top in (0, 20):
            o = to_host(sampler.albireo_sample(view, **par, num_top=num_top, flags=flags))
            assert ((o["tokens"] >= 0) & (o["tokens"] < V)).all(), (flags, num_top, o["tokens"])
            if num_top:
                assert ((o["top_ids"] >= -1) & (o["top_ids"] < V)).all(), (flags, num_top)


@pytest.mark.parametrize("B", [8, 80])
def test_size_of_a_top_k_with_ties_below_the_min_p_floor(binding, sampler, B):
    """The top-k stage's size with ties kept, where the k-th largest score lies below the min-p floor (no debug
    list, which changes what the stream may drop)."""
    V = 17003
    rng = np.random.default_rng(59)
    x = np.round(rng.standard_normal((B, V)) * 2).astype(np.float32)
    x[:, :5] = 20.0
    w = W.Workload("ties_minp", B, V, W.BF16, W.f32_to_bf16_bits(x), temperature=np.ones(B, np.float32), top_k=np.full(B, 12, np.int32),
                   min_p=np.full(B, 0.1, np.float32), seeds=np.arange(B, dtype=np.uint64))
    w.topk_keep_ties = True
    ref = O.sample(w, threads=_CORES)
    t = binding.workload_tensors(w, sampler.device)
    g = to_host(sampler.albireo_sample(t.pop("logits"), **t, want_counts=True, flags=binding.FLAG_TOPK_KEEP_TIES))
    assert (g["num_topk"] == ref.rows["n_topk"]).all() and (g["num_kept"] == ref.rows["n_keep"]).all()
    assert compare(w, g, ref).ok()


@pytest.mark.parametrize("B", [2, 12, 24, 50])
@pytest.mark.parametrize("dtype", [W.F32, W.BF16])
def test_long_histories(binding, sampler, B, dtype):
    """Histories with more distinct ids in a slice than its list on chip takes, in clusters of every size: the rows stay
    on their path, with and without a prompt part and with ids outside the vocabulary."""
    V = 120001
    rng = np.random.default_rng(61)
    x = (rng.standard_normal((B, V)) * 2).astype(np.float32)
    rows = [rng.integers(-3, V + 3, 20000) if b % 3 == 0 else rng.integers(0, 6000, 4000) if b % 3 == 1 else
            np.minimum(rng.zipf(1.2, 16000), V - 1) for b in range(B)]
    w = W.Workload("long", B, V, dtype, x if dtype == W.F32 else W.f32_to_bf16_bits(x), temperature=np.ones(B, np.float32),
                   top_k=np.where(np.arange(B) % 2, 50, 0).astype(np.int32), top_p=np.full(B, 0.9, np.float32),
                   repetition_penalty=np.full(B, 1.3, np.float32), presence_penalty=np.full(B, 0.4, np.float32),
                   frequency_penalty=np.full(B, 0.2, np.float32), history_ids=np.concatenate(rows).astype(np.int32),
                   history_offsets=np.cumsum([0] + [len(r) for r in rows]).astype(np.int32), seeds=np.arange(B, dtype=np.uint64))
    w.output_start = np.where(np.arange(B) % 4 == 0, 7000, 0).astype(np.int32)
    w.num_top = 5
    g, ref = check(binding, sampler, w)
    assert (g["num_kept"] == ref.rows["n_keep"]).all()
    assert not (g["row_status"][w.top_k > 0] & binding.ROW_GENERAL_PATH).any()
    assert not (g["row_status"] & binding.ROW_HISTORY_OVERFLOW).any()
