"""Passes of one CTA over a row in global memory, and the end of a cut among equal scores: row lengths around whole rounds of the passes' loads, rows in pieces,
kept sets of more vectors than wait in the last pass at a time, hundreds of elements at the score of the cut, against the oracle."""
import os
from contextlib import closing

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
    s = binding.Sampler(max_rows=80, max_vocab=131072, max_history_total=1 << 18)
    yield s
    s.close()


# 80 rows: a CTA to each (a round is 4 vectors of each of 512 threads: 16384 elements of 16 bits, 8192 of fp32); 40: two CTAs to a row.
@pytest.mark.parametrize("B,V,pieces", [(80, 16384, 1), (80, 16376, 1), (80, 32776, 1), (80, 36865, 1), (80, 131072, 1), (80, 36864, 4), (80, 20480, 2), (40, 131072, 1)])
@pytest.mark.parametrize("dtype", [W.BF16, W.F32])
@pytest.mark.parametrize("history", [False, True])
def test_wide_rows(binding, sampler, B, V, pieces, dtype, history):
    rng = np.random.default_rng(V + B)
    x = (rng.standard_normal((B, V)) * 3).astype(np.float32)
    x[::4] = np.round(x[::4] * 2) / 2                  # thousands of equal scores
    x[1::4] -= 12.0                                    # hundreds of bfloat16 values' worth of equals
    cls = np.arange(B) % 5
    w = W.Workload("wide", B, V, dtype, W.f32_to_bf16_bits(x) if dtype == W.BF16 else x, temperature=rng.choice([0.6, 1.0, 2.5], B).astype(np.float32),
                   top_p=np.where(cls == 4, 1.0, rng.uniform(0.5, 0.999, B)).astype(np.float32),
                   min_p=np.where(cls == 3, 10.0 ** rng.uniform(-5, -3, B), 0.0).astype(np.float32), seeds=rng.integers(0, 1 << 62, B).astype(np.uint64), step=3)
    if history:
        lens = rng.integers(0, 900, B)
        w.history_offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        w.history_ids = rng.integers(0, V, int(lens.sum())).astype(np.int32)
        w.repetition_penalty, w.presence_penalty, w.frequency_penalty = (np.full(B, v, np.float32) for v in (1.2, 0.3, 0.1))
    ref = O.sample(w, threads=_CORES)
    t = binding.workload_tensors(w, sampler.device)
    lg = t.pop("logits")
    if pieces > 1:
        lg = torch.stack([lg[:, j * (V // pieces):(j + 1) * (V // pieces)] for j in range(pieces)]).contiguous()
    g = to_host(sampler.albireo_sample(lg, **t, want_counts=True, want_status=True))
    rep = compare(w, g, ref)
    assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])


# Rows so short that some or all of them have no whole aligned vector of 16 bytes (and rows of one vector and two among them): nothing is copied for
# those.  1 and 80 rows are on the device at once, 300 are not.
@pytest.mark.parametrize("V", [1, 2, 3, 7, 9, 14, 15, 17])
@pytest.mark.parametrize("dtype", [W.BF16, W.F16, W.F32])
@pytest.mark.parametrize("history,num_top", [(False, 0), (True, 0), (False, 3)])
def test_rows_without_a_whole_vector(binding, dtype, V, history, num_top):
    with closing(binding.Sampler(max_rows=300, max_vocab=32, max_history_total=1 << 16)) as sampler:
        for B in (1, 80, 300):
            base = W.random_small(2000 + 16 * B + V, B=B, V=V, dtype=W.F32 if dtype == W.F16 else dtype, with_history=history)
            if B == 1:
                base.temperature[:], base.top_k[:], base.top_p[:] = 0.9, 0, 0.8
            base.num_top = num_top
            w = W.as_f16(base) if dtype == W.F16 else base
            ref = O.sample(w, threads=_CORES)
            t = binding.workload_tensors(w, sampler.device)
            g = to_host(sampler.albireo_sample(t.pop("logits"), **t, num_top=num_top, want_status=True))
            rep = compare(w, g, ref)
            assert rep.ok() and not rep.excused, (B, rep.summary(), rep.failures[:3], rep.excused[:3])
            assert not (g["row_status"] & binding.ROW_TIMEOUT).any(), B
            assert not compare_top_lists(w, g, ref), B


# A floor and no top-p: so many elements above it as wait in the last pass at a time (7168 vectors), fewer and more, some of them penalised, lists with and without
@pytest.mark.parametrize("B,V", [(80, 131072), (80, 65537), (24, 131072)])
@pytest.mark.parametrize("num_top,history", [(0, False), (0, True), (5, False)])
def test_floor_alone(binding, sampler, B, V, num_top, history):
    rng = np.random.default_rng(V + B)
    kept = np.array([1100, 2050, 7167, 7168, 7169, 7680, 20000, 60000])[np.arange(B) % 8]
    x = rng.uniform(-9, -6, (B, V)).astype(np.float32)
    for b in range(B):
        x[b, rng.permutation(V)[:kept[b]]] = rng.uniform(2, 5, kept[b]).astype(np.float32)
    w = W.Workload("floor", B, V, W.BF16, W.f32_to_bf16_bits(x), temperature=np.ones(B, np.float32), min_p=np.full(B, 1e-3, np.float32), seeds=rng.integers(0, 1 << 62, B).astype(np.uint64), step=4)
    w.num_top = num_top
    if history:
        lens = rng.integers(0, 900, B)
        w.history_offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        w.history_ids = rng.integers(0, V, int(lens.sum())).astype(np.int32)
        w.repetition_penalty, w.presence_penalty, w.frequency_penalty = (np.full(B, v, np.float32) for v in (1.2, 0.3, 0.1))
    ref = O.sample(w, threads=_CORES)
    t = binding.workload_tensors(w, sampler.device)
    g = to_host(sampler.albireo_sample(t.pop("logits"), **t, num_top=num_top, want_counts=True, want_status=True))
    rep = compare(w, g, ref)
    assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])
    assert (g["num_kept"] == ref.rows["n_keep"]).all()
    assert not compare_top_lists(w, g, ref)
