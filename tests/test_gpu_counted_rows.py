"""Rows of bfloat16 logits whose values are counted (top-p, min-p that keeps many, lists): the ends of the table of values,
what has no place in it, cuts in the segments that penalised tokens share, against the oracle.  Only results are compared: a row that is not
counted after all gives the same ones by the passes of other rows."""
import os

import numpy as np
import pytest
import torch

from oracle import albireo_oracle as O
from paper_2606_01927_b200 import workloads as W

from parity import compare, compare_top_lists, to_host

pytestmark = pytest.mark.gpu

_CORES = len(os.sched_getaffinity(0))


@pytest.fixture(scope="module")
def binding():
    from paper_2606_01927_b200 import binding as Bd
    return Bd


@pytest.fixture(scope="module")
def sampler(binding):
    s = binding.Sampler(max_rows=80, max_vocab=140000, max_history_total=1 << 20)
    yield s
    s.close()


def rows(kind, B, V, rng):
    x = rng.standard_normal((B, V)) * 3 - 1.1 * np.log(np.arange(1, V + 1))
    if kind == "ends":                       # the table's last values, and those just outside it
        for b in range(B):
            for v in (-63.75, -63.5, -64.0, -1e4, 2.0 ** -26, -(2.0 ** -26), 2.0 ** -27, -(2.0 ** -27), 1e-39, 0.0, -0.0, 63.75 if b % 3 else 3.0):
                x[b, rng.integers(0, V, 5)] = v
            if b % 4 == 1:
                x[b, rng.integers(0, V)] = 64.0
    elif kind == "zeros":                    # padding logits: up to 254 of them are listed, more are not
        for b in range(B):
            x[b, V - (253 + b % 3):] = 0.0
            x[b, :V // 2] -= 6.0
    elif kind == "masked":
        x[rng.random((B, V)) < 0.6] = -np.inf
    elif kind == "below":                    # all of the row where values are counted together
        x = np.minimum(x - 70.0, -60.0)
    elif kind == "ties":                     # thousands of equal scores at the cut
        x = np.round(rng.standard_normal((B, V)) * 0.7) + 40.0
    elif kind == "flat":
        x = rng.standard_normal((B, V)) * 0.01
    elif kind == "high":
        x = x + 50.0
    return x.astype(np.float32)


# 40 rows: two CTAs to a row, 16: eight (slices just large enough to be counted; of 32760 the last one is 8 ids short of
# that, and of 32752 both are); 80: a CTA to each
@pytest.mark.parametrize("B,V", [(40, 33007), (40, 32760), (40, 32752), (16, 131080), (80, 8211)])
@pytest.mark.parametrize("kind", ["plain", "ends", "zeros", "masked", "below", "ties", "flat", "high"])
@pytest.mark.parametrize("history", [False, True])
def test_counted_rows(binding, sampler, B, V, kind, history):
    rng = np.random.default_rng(500 + B)
    x = rows(kind, B, V, rng)
    cls = np.arange(B) % 5
    w = W.Workload(kind, B, V, W.BF16, W.f32_to_bf16_bits(x), temperature=rng.choice([0.4, 0.9, 1.0, 1.6], B).astype(np.float32),
                   top_p=np.where(cls == 4, 1.0, 1.0 - 10.0 ** rng.uniform(-3, -0.2, B)).astype(np.float32),
                   min_p=np.where(cls >= 3, 10.0 ** rng.uniform(-12, -2, B), 0.0).astype(np.float32),
                   seeds=rng.integers(0, 1 << 62, B).astype(np.uint64), step=9)
    if history:
        lens = rng.integers(0, 1200, B)
        w.history_offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        w.history_ids = np.minimum(rng.zipf(1.15, int(lens.sum())) - 1, V - 1).astype(np.int32)
        w.repetition_penalty, w.presence_penalty, w.frequency_penalty = (np.full(B, v, np.float32) for v in (1.13, 0.21, 0.07))
    for num_top, full in ((0, False), (6, False), (6, True)):
        w.num_top, w.logprob_full_vocab = num_top, full
        if full:
            w.min_p = None
        ref = O.sample(w, threads=_CORES)
        t = binding.workload_tensors(w, sampler.device)
        g = to_host(sampler.albireo_sample(t.pop("logits"), **t, num_top=num_top, want_counts=True, want_status=True,
                                           flags=binding.FLAG_LOGPROB_FULL_VOCAB if full else 0))
        rep = compare(w, g, ref)
        assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])
        bad = compare_top_lists(w, g, ref)
        assert not bad, bad[:3]


@pytest.mark.parametrize("B", [40, 80])
def test_no_cut_and_extreme_temperatures(binding, sampler, B):
    """The race against a reference that is not the maximum: rows whose largest score comes late, and rows whose first
    vectors hold no finite score; temperatures at which the scores of different values meet."""
    V = 40003
    rng = np.random.default_rng(77)
    x = rng.standard_normal((B, V)).astype(np.float32)
    late = np.arange(B) % 4 == 1
    x[late, :20000] -= 50.0
    x[late, 30001] = 60.0
    x[np.arange(B) % 4 == 2, :20000] = -np.inf
    T = np.where(np.arange(B) % 4 == 3, 10.0 ** rng.uniform(-19, 19, B), 1.0).astype(np.float32)
    for top_p in (1.0, 0.7):
        w = W.Workload("none", B, V, W.BF16, W.f32_to_bf16_bits(x), temperature=T, top_p=np.full(B, top_p, np.float32),
                       seeds=np.arange(B, dtype=np.uint64))
        ref = O.sample(w, threads=_CORES)
        t = binding.workload_tensors(w, sampler.device)
        g = to_host(sampler.albireo_sample(t.pop("logits"), **t, want_counts=True, want_status=True))
        rep = compare(w, g, ref)
        assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])


@pytest.mark.parametrize("B", [40, 80])
def test_thousands_of_masses_in_a_segment(binding, sampler, B):
    """Thousands of penalised tokens and zeros of (nearly) the largest mass, all of them in one segment, and the cut far below:
    their sum passes 2^52, and its low word wraps many times.  More than 2048 distinct ids by one CTA per row: their scores lie in
    the workspace."""
    V = 40003
    rng = np.random.default_rng(11)
    x = (-0.5 - 2.5 * rng.random((B, V))).astype(np.float32)
    n = np.where(np.arange(B) % 2 == 0, 3950, 6000)
    for b in range(B):
        x[b, :n[b] + 200] = 0.0
        if b % 3:
            x[b, 20000] = 2.0 ** -(b % 7)
    w = W.Workload("zeros", B, V, W.BF16, W.f32_to_bf16_bits(x), temperature=np.ones(B, np.float32), top_p=np.full(B, 0.9, np.float32),
                   seeds=rng.integers(0, 1 << 62, B).astype(np.uint64), step=3,
                   history_ids=np.concatenate([np.arange(k) for k in n]).astype(np.int32), history_offsets=np.concatenate([[0], np.cumsum(n)]).astype(np.int32),
                   repetition_penalty=np.full(B, 1.1, np.float32), presence_penalty=np.zeros(B, np.float32), frequency_penalty=np.zeros(B, np.float32))
    ref = O.sample(w, threads=_CORES)
    t = binding.workload_tensors(w, sampler.device)
    g = to_host(sampler.albireo_sample(t.pop("logits"), **t, want_counts=True, want_status=True))
    rep = compare(w, g, ref)
    assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])
    # (exponentials to 2^-22: the sum of 8000 to 12000 is off by 0.003 at most, a token at the cut weighs 0.1)
    assert np.abs(g["num_kept"].astype(np.int64) - ref.rows["n_keep"]).max() <= 2


@pytest.mark.parametrize("kind", ["low", "masked", "dense"])
def test_ties_far_above_the_first_vectors(binding, sampler, kind):
    """Rows without a cut by one CTA each are raced before their maximum is known: equal maxima behind the first 4096 ids, at
    temperatures that take them up to 1e9 above all that lies ahead (`low`), behind ids that are masked, and hundreds of thousands of units above
    rows of which half is at the maximum (`dense`).  Only the generator's words tell them apart; the same rows by clusters give the same bits."""
    B, V = 80, 40003
    rng = np.random.default_rng(5)
    x = rng.standard_normal((B, V)).astype(np.float32)
    x[:, :4200] = -np.inf if kind == "masked" else -5.0
    for b in range(B):
        if kind == "dense":
            x[b, 4200:][rng.random(V - 4200) < 0.5] = 8.0
        else:
            x[b, rng.integers(4200, V, 40)] = 8.0
            start = 4200 + 8 * int(rng.integers(0, 4000))
            x[b, start:start + 24] = 8.0
    T = np.where(np.arange(B) % 2 == 0, 10.0 ** rng.uniform(-8, -4, B), 10.0 ** rng.uniform(-4, 0, B)).astype(np.float32)
    w = W.Workload("ties", B, V, W.BF16, W.f32_to_bf16_bits(x), temperature=T, seeds=rng.integers(0, 1 << 62, B).astype(np.uint64), step=5)
    ref = O.sample(w, threads=_CORES)
    t = binding.workload_tensors(w, sampler.device)
    logits, step = t.pop("logits"), t.pop("step")
    g = to_host(sampler.albireo_sample(logits, **t, step=step, want_counts=True, want_status=True))
    rep = compare(w, g, ref)
    assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])
    for lo in (0, 40):
        part = to_host(sampler.albireo_sample(logits[lo:lo + 40], **{k: v[lo:lo + 40] for k, v in t.items() if v is not None}, step=step, row_base=lo,
                                              want_counts=True))
        for f in ("tokens", "num_kept", "num_topk"):
            assert (part[f] == g[f][lo:lo + 40]).all(), (f, lo)
        assert (part["logprobs"].view(np.uint32) == g["logprobs"][lo:lo + 40].view(np.uint32)).all(), lo


@pytest.mark.parametrize("B", [40, 80])
def test_penalised_scores_without_a_place(binding, sampler, B):
    """Penalties that take scores beyond every value of the logits' type, up (a negative presence penalty) or down: such a token has no place
    in the table, whichever thread comes upon it."""
    V = 40003
    rng = np.random.default_rng(3)
    x = rng.standard_normal((B, V)).astype(np.float32)
    n = 1 + np.arange(B) * 37
    w = W.Workload("beyond", B, V, W.BF16, W.f32_to_bf16_bits(x), temperature=np.ones(B, np.float32), top_p=np.full(B, 0.7, np.float32),
                   seeds=rng.integers(0, 1 << 62, B).astype(np.uint64), step=3,
                   history_ids=np.concatenate([rng.permutation(V)[:k] for k in n]).astype(np.int32), history_offsets=np.concatenate([[0], np.cumsum(n)]).astype(np.int32),
                   repetition_penalty=np.ones(B, np.float32), frequency_penalty=np.zeros(B, np.float32),
                   presence_penalty=np.where(np.arange(B) % 2 == 0, -3.4e38, 3.4e38).astype(np.float32))
    ref = O.sample(w, threads=_CORES)
    t = binding.workload_tensors(w, sampler.device)
    g = to_host(sampler.albireo_sample(t.pop("logits"), **t, want_counts=True, want_status=True))
    rep = compare(w, g, ref)
    assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])


@pytest.mark.parametrize("B,V", [(40, 33007), (80, 8211)])
@pytest.mark.parametrize("kind", ["half zeros", "tall", "too many tall", "all tall", "tiny"])
@pytest.mark.parametrize("history", [False, True])
def test_values_without_a_place(binding, sampler, B, V, kind, history):
    """Values that the table does not hold: zeros of both signs by the thousand, up to 254 others that are listed (64 and more; nearer to zero than
    2^-26), more of them than that; cuts among values of 64 and more, and below them, at temperatures that spread the mass over either."""
    rng = np.random.default_rng(900 + B)
    x = (rng.standard_normal((B, V)) * 3).astype(np.float32)
    for b in range(B):
        n = {"half zeros": V // 2, "tall": 1 + 31 * (b % 8), "too many tall": 255 + b, "all tall": V, "tiny": 245 + b % 16}[kind]
        at = rng.permutation(V)[:n]
        x[b, at] = {"half zeros": np.where(rng.random(n) < 0.5, 0.0, -0.0), "tiny": rng.choice([-1.0, 1.0], n) * 2.0 ** rng.uniform(-60, -27, n)}.get(
            kind, rng.uniform(56, 100, n))
        if kind == "tall" and b % 4 == 3:
            x[b, rng.integers(0, V, 300)] = rng.uniform(57, 63.9, 300)
    w = W.Workload(kind, B, V, W.BF16, W.f32_to_bf16_bits(x), temperature=np.where(np.arange(B) % 3 == 0, 1.0, rng.choice([8.0, 30.0], B)).astype(np.float32),
                   top_p=rng.choice([0.01, 0.1, 0.5, 0.9, 0.99], B).astype(np.float32), seeds=rng.integers(0, 1 << 62, B).astype(np.uint64), step=4)
    if history:
        lens = rng.integers(0, 1200, B)
        w.history_offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        w.history_ids = rng.integers(0, V, int(lens.sum())).astype(np.int32)
        w.repetition_penalty, w.presence_penalty, w.frequency_penalty = (np.full(B, v, np.float32) for v in (1.13, 0.0, 0.0))
    for num_top, full in ((0, False), (6, False), (6, True)):
        w.num_top, w.logprob_full_vocab = num_top, full
        ref = O.sample(w, threads=_CORES)
        t = binding.workload_tensors(w, sampler.device)
        g = to_host(sampler.albireo_sample(t.pop("logits"), **t, num_top=num_top, want_counts=True, want_status=True,
                                           flags=binding.FLAG_LOGPROB_FULL_VOCAB if full else 0))
        rep = compare(w, g, ref)
        assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])
        bad = compare_top_lists(w, g, ref)
        assert not bad, bad[:3]
