"""Batches of more rows than are on the device at once, wide ones among them, and histories around the sizes of the candidate path's hash table of ids,
against the oracle; a workspace that holds fewer distinct ids than a row has."""
import os
from contextlib import closing

import numpy as np
import pytest
import torch

from oracle import albireo_oracle as O
from paper_2606_01927_b200 import workloads as W

from parity import compare, to_host

pytestmark = pytest.mark.gpu

_CORES = len(os.sched_getaffinity(0))


@pytest.fixture(scope="module")
def binding():
    from paper_2606_01927_b200 import binding as Bd
    return Bd


@pytest.fixture(scope="module")
def sampler(binding):
    s = binding.Sampler(max_rows=1100, max_vocab=40000, max_history_total=1 << 20)
    yield s
    s.close()


def against_oracle(binding, sampler, w):
    ref = O.sample(w, threads=_CORES)
    t = binding.workload_tensors(w, sampler.device)
    g = to_host(sampler.albireo_sample(t.pop("logits"), **t, want_status=True))
    rep = compare(w, g, ref)
    assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])
    return g


# more than 296 rows: one more, and over three rounds of them.  Wide rows: none, a few at the end, most, all
@pytest.mark.parametrize("B,V", [(297, 20011), (1024, 4000), (1060, 4096)])
@pytest.mark.parametrize("wide", [0.0, 0.03, 0.7, 1.0])
@pytest.mark.parametrize("dtype", [W.BF16, W.F32])
def test_wide_rows_first(binding, sampler, B, V, wide, dtype):
    rng = np.random.default_rng(B + int(100 * wide))
    x = (rng.standard_normal((B, V)) * 2.5).astype(np.float32)
    is_wide = rng.random(B) < wide if wide != 0.03 else np.arange(B) >= B - 9
    lens = rng.integers(0, 60, B)
    w = W.Workload("ordered", B, V, dtype, W.f32_to_bf16_bits(x) if dtype == W.BF16 else x, temperature=np.where(is_wide | (np.arange(B) % 5 > 0), 0.9, 0.0).astype(np.float32),
                   top_k=np.where(is_wide, 0, rng.integers(1, 90, B)).astype(np.int32), top_p=rng.uniform(0.5, 1.0, B).astype(np.float32),
                   min_p=np.where(np.arange(B) % 3 == 0, 10.0 ** rng.uniform(-4, -1, B), 0.0).astype(np.float32),
                   seeds=rng.integers(0, 1 << 62, B).astype(np.uint64), step=5)
    w.history_offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    w.history_ids = rng.integers(0, V, int(lens.sum())).astype(np.int32)
    w.repetition_penalty, w.presence_penalty, w.frequency_penalty = (np.full(B, v, np.float32) for v in (1.2, 0.3, 0.1))
    against_oracle(binding, sampler, w)


# 2048 ids are staged on chip, 3584 are hashed at most, 4096 distinct ones are more than the rank tables hold on chip
@pytest.mark.parametrize("ids", ["distinct", "few", "outside"])
@pytest.mark.parametrize("B,dtype", [(80, W.BF16), (160, W.F32), (300, W.F16)])
def test_histories(binding, sampler, ids, B, dtype):
    V = 39999
    rng = np.random.default_rng(B)
    x = (rng.standard_normal((B, V)) * 3).astype(np.float32)
    lens = np.array([0, 1, 2047, 2048, 2049, 3583, 3584, 3585, 4096, 700])[np.arange(B) % 10]
    rows = []
    for n in lens:
        if ids == "distinct":
            rows.append(rng.permutation(V)[:n])
        elif ids == "few":
            rows.append(np.minimum(rng.zipf(1.3, n) - 1, V - 1))
        else:
            rows.append(rng.integers(-50, V + 50, n))
    w = W.Workload("histories", B, V, W.F32 if dtype == W.F16 else dtype, W.f32_to_bf16_bits(x) if dtype == W.BF16 else x, temperature=np.full(B, 0.8, np.float32),
                   top_k=rng.integers(1, 120, B).astype(np.int32), top_p=np.full(B, 0.95, np.float32), seeds=rng.integers(0, 1 << 62, B).astype(np.uint64), step=6)
    w.history_offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    w.history_ids = np.concatenate(rows).astype(np.int32)
    w.repetition_penalty, w.presence_penalty, w.frequency_penalty = (np.full(B, v, np.float32) for v in (0.7, -0.4, -0.05))      # (penalised tokens come out ahead)
    w.output_start = np.where(np.arange(B) % 4 == 0, lens // 2, 0).astype(np.int32)
    against_oracle(binding, sampler, W.as_f16(w) if dtype == W.F16 else w)


# Every kind of row in one batch, around the sizes of the hash table (1025 to 3584 ids, 2048 of them staged on chip); the min-p rows outgrow the candidate list, so that their
# tables are built anew over the hashed ones.  80 rows have an SM each, 300 are more than are on the device at once.
_LENGTHS = np.array([0, 59, 1023, 1024, 1025, 2047, 2048, 2049, 3584, 3585, 4096])


@pytest.mark.parametrize("B,V,pieces", [(80, 39999, 1), (300, 39999, 1), (300, 40000, 4)])
@pytest.mark.parametrize("dtype", [W.BF16, W.F16])
def test_histories_of_mixed_rows(binding, sampler, B, V, pieces, dtype):
    rng = np.random.default_rng(B + pieces)
    x = (rng.standard_normal((B, V)) * 3).astype(np.float32)
    lens, cls = _LENGTHS[np.arange(B) % len(_LENGTHS)], (np.arange(B) // len(_LENGTHS)) % 4
    w = W.Workload("mixed", B, V, W.F32 if dtype == W.F16 else dtype, W.f32_to_bf16_bits(x) if dtype == W.BF16 else x, temperature=np.where(cls == 0, 0.0, 0.9).astype(np.float32),
                   top_k=np.where(cls == 1, rng.integers(1, 100, B), 0).astype(np.int32), top_p=np.where(cls == 2, rng.uniform(0.5, 1.0, B), 1.0).astype(np.float32),
                   min_p=np.where(cls == 3, 1e-4, 0.0).astype(np.float32), seeds=rng.integers(0, 1 << 62, B).astype(np.uint64), step=7)
    w.history_offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    w.history_ids = rng.integers(0, V, int(lens.sum())).astype(np.int32)
    w.repetition_penalty, w.presence_penalty, w.frequency_penalty = (np.full(B, v, np.float32) for v in (0.7, -0.4, -0.05))      # (penalised tokens come out ahead)
    w.output_start = np.where(np.arange(B) % 3 == 0, lens // 2, 0).astype(np.int32)
    if dtype == W.F16:
        w = W.as_f16(w)
    ref = O.sample(w, threads=_CORES)
    t = binding.workload_tensors(w, sampler.device)
    lg = t.pop("logits")
    if pieces > 1:
        lg = torch.stack([lg[:, j * (V // pieces):(j + 1) * (V // pieces)] for j in range(pieces)]).contiguous()
    g = to_host(sampler.albireo_sample(lg, **t, want_status=True))
    rep = compare(w, g, ref)
    assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])
    assert not (g["row_status"] & binding.ROW_HISTORY_OVERFLOW).any()


# a vocabulary whose bitmap leaves room for the hash table beside two CTAs per SM, and one that does not
@pytest.mark.parametrize("V", [175072, 175073])
def test_histories_of_the_largest_hashed_vocabulary(binding, V):
    B, n = 152, 2000
    rng = np.random.default_rng(V)
    w = W.Workload("bitmap", B, V, W.BF16, W.f32_to_bf16_bits((rng.standard_normal((B, V)) * 3).astype(np.float32)), temperature=np.full(B, 0.8, np.float32), top_k=np.full(B, 40, np.int32),
                   seeds=np.arange(B, dtype=np.uint64), history_ids=rng.integers(0, V, B * n).astype(np.int32), history_offsets=(np.arange(B + 1) * n).astype(np.int32),
                   repetition_penalty=np.full(B, 0.7, np.float32), presence_penalty=np.full(B, -0.4, np.float32), frequency_penalty=np.zeros(B, np.float32))
    with closing(binding.Sampler(max_rows=B, max_vocab=V, max_history_total=B * n)) as s:
        against_oracle(binding, s, w)


@pytest.mark.parametrize("B", [80, 300])
@pytest.mark.parametrize("dtype", [W.BF16, W.F16])
def test_workspace_shorter_than_a_rows_ids(binding, B, dtype):
    """Rows with more than 2048 distinct ids and no room for them in the workspace are sampled without penalties and marked, whatever table their length would have; all others have theirs."""
    V = 20000
    rng = np.random.default_rng(B)
    lens = np.array([2048, 2049, 0, 3584, 1025, 3585, 2300])[np.arange(B) % 7]
    few = np.arange(B) % 14 >= 7                           # (long histories of few ids)
    rows = [rng.integers(0, 1500, n) if f else rng.permutation(V)[:n] for n, f in zip(lens, few)]
    over = np.array([np.unique(r).size > 2048 for r in rows])
    x = (rng.standard_normal((B, V)) * 2).astype(np.float32)

    def workload(rows):
        w = W.Workload("short", B, V, W.F32 if dtype == W.F16 else dtype, W.f32_to_bf16_bits(x) if dtype == W.BF16 else x, temperature=np.full(B, 0.9, np.float32), top_k=np.full(B, 64, np.int32),
                       repetition_penalty=np.full(B, 1.3, np.float32), presence_penalty=np.full(B, 0.5, np.float32), frequency_penalty=np.full(B, 0.2, np.float32),
                       seeds=np.arange(B, dtype=np.uint64) + 5, history_ids=np.concatenate(rows).astype(np.int32), history_offsets=np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32))
        return W.as_f16(w) if dtype == W.F16 else w
    w, marked = workload(rows), workload([r[:0] if o else r for r, o in zip(rows, over)])
    ref = O.sample(marked, threads=_CORES)
    with closing(binding.Sampler(max_rows=B, max_vocab=V, max_history_total=1000)) as s:
        t = binding.workload_tensors(w, s.device)
        g = to_host(s.albireo_sample(t.pop("logits"), **t, want_status=True))
    rep = compare(marked, g, ref)
    assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])
    assert (((g["row_status"] & binding.ROW_HISTORY_OVERFLOW) != 0) == over).all() and over.any()
