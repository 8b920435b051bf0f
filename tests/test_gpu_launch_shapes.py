"""Which kernel a batch gets, read from captured graphs: CTAs per row up to the longest rows whose slices fit the shared memory,
whatever the kernel keeps in front of them; and results there."""
import os

import numpy as np
import pytest
import torch

from oracle import albireo_oracle as O
from paper_2606_01927_b200 import workloads as W

from parity import compare, to_host

pytestmark = pytest.mark.gpu

_CORES = len(os.sched_getaffinity(0))
_TORCH = {W.F32: torch.float32, W.BF16: torch.bfloat16, W.F16: torch.float16}


@pytest.fixture(scope="module")
def binding():
    from paper_2606_01927_b200 import binding as Bd
    return Bd


@pytest.fixture(scope="module")
def sampler(binding):
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the table below is for 148 SMs")
    s = binding.Sampler(max_rows=80, max_vocab=400000, max_history_total=1 << 18)
    yield s
    s.close()


def launched(sampler, *args, **kw):
    """CTAs and mangled name of the one kernel that a call launches (captured, not run)."""
    from cuda.bindings import driver
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        out = sampler.albireo_sample(*args, **kw)
    err, nodes, count = driver.cuGraphGetNodes(driver.CUgraph(graph.raw_cuda_graph()), 8)
    assert err == driver.CUresult.CUDA_SUCCESS and count == 1, (err, count)
    err, p = driver.cuGraphKernelNodeGetParams(nodes[0])
    assert err == driver.CUresult.CUDA_SUCCESS, err
    err, name = driver.cuFuncGetName(p.func) if int(p.func) else driver.cuKernelGetName(p.kern)
    assert err == driver.CUresult.CUDA_SUCCESS, err
    del out
    return int(p.gridDimX), name.decode()


def batch(sampler, B, V, dtype, history, **par):
    dev = sampler.device
    if history:
        par.update(history_ids=torch.arange(B * 64, dtype=torch.int32, device=dev), history_offsets=torch.arange(0, 64 * B + 1, 64, dtype=torch.int32, device=dev))
    return torch.zeros((B, V), dtype=_TORCH[dtype], device=dev), dict(par, temperature=torch.ones(B, device=dev))


# the longest rows that are shared by so many CTAs
@pytest.mark.parametrize("dtype,history,B,V,team", [
    (W.BF16, False, 64, 197632, 2), (W.F16, False, 34, 197632, 2), (W.BF16, True, 74, 177152, 2), (W.F16, True, 34, 177152, 2),
    (W.BF16, False, 33, 395264, 4), (W.F16, True, 16, 354304, 4), (W.F32, False, 74, 98816, 2), (W.F32, False, 33, 197632, 4),
    (W.F32, True, 34, 91584, 2), (W.F32, True, 16, 183168, 4),
    (W.BF16, False, 64, 200000, 1), (W.BF16, False, 75, 32768, 1), (W.BF16, False, 64, 152064, 2)])
def test_ctas_per_row(binding, sampler, dtype, history, B, V, team):
    logits, par = batch(sampler, B, V, dtype, history, top_p=torch.full((B,), 0.9, device=sampler.device))
    ctas, name = launched(sampler, logits, **par)
    assert ctas == B * team, (ctas / B, name)
    assert ("cluster" in name) == (team > 1), name


@pytest.mark.parametrize("dtype,history,B,V", [(W.BF16, False, 34, 197632), (W.BF16, True, 34, 177152), (W.BF16, False, 34, 195000), (W.F32, False, 34, 98816),
                                               (W.F16, True, 34, 177152), (W.BF16, False, 34, 197640)])
def test_longest_slices(binding, sampler, dtype, history, B, V):
    """Slices that fill the shared memory, with the table of values in front of them and without, and rows just too long for that."""
    rng = np.random.default_rng(V)
    x = (rng.standard_normal((B, V)) * 3).astype(np.float32)
    lg = x if dtype == W.F32 else W.f32_to_bf16_bits(x) if dtype == W.BF16 else x.astype(np.float16).view(np.uint16)
    w = W.Workload("long", B, V, dtype, lg, temperature=np.full(B, 0.9, np.float32), top_p=np.where(np.arange(B) % 3 == 2, 1.0, 0.9).astype(np.float32),
                   seeds=rng.integers(0, 1 << 62, B).astype(np.uint64), step=2)
    if history:
        lens = rng.integers(0, 3000, B)
        w.history_offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        w.history_ids = rng.integers(0, V, int(lens.sum())).astype(np.int32)
        w.repetition_penalty, w.presence_penalty, w.frequency_penalty = (np.full(B, v, np.float32) for v in (1.13, 0.21, 0.07))
    ref = O.sample(w, threads=_CORES)
    t = binding.workload_tensors(w, sampler.device)
    rep = compare(w, to_host(sampler.albireo_sample(t.pop("logits"), **t, want_counts=True, want_status=True)), ref)
    assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])


@pytest.mark.parametrize("cut", ["top_k", "top_k and top_p"])
def test_distinct_ids_that_a_slice_holds(binding, cut):
    """64 rows of 152064 with 8500 distinct ids, some of them twice, in one half of the vocabulary: their scores still lie on chip (the ids in the
    workspace), in the kernel with the table of values as well, and the rows are done in a single pass."""
    B, V, n = 64, 152064, 8600
    s = binding.Sampler(max_rows=B, max_vocab=V, max_history_total=B * n)
    rng = np.random.default_rng(1)
    w = W.Workload("many ids", B, V, W.BF16, W.f32_to_bf16_bits((rng.standard_normal((B, V)) * 3).astype(np.float32)), temperature=np.ones(B, np.float32),
                   top_k=np.full(B, 40, np.int32), top_p=np.full(B, 0.9, np.float32) if "top_p" in cut else None, seeds=np.arange(B, dtype=np.uint64),
                   history_ids=np.concatenate([np.tile(rng.permutation(V // 2)[:8500], 2)[:n] for _ in range(B)]).astype(np.int32), history_offsets=(np.arange(B + 1) * n).astype(np.int32),
                   repetition_penalty=np.full(B, 1.2, np.float32), presence_penalty=np.zeros(B, np.float32), frequency_penalty=np.full(B, 0.1, np.float32))
    ref = O.sample(w, threads=_CORES)
    t = binding.workload_tensors(w, s.device)
    g = to_host(s.albireo_sample(t.pop("logits"), **t, want_status=True))
    rep = compare(w, g, ref)
    assert rep.ok() and not rep.excused, (rep.summary(), rep.failures[:3], rep.excused[:3])
    assert not (g["row_status"] & (binding.ROW_GENERAL_PATH | binding.ROW_HISTORY_OVERFLOW)).any()
    s.close()


@pytest.mark.parametrize("par,counted", [(("top_p",), True), (("num_top",), True), (("top_k", "top_p"), True), ((), False), (("top_k",), False), (("min_p",), False)])
def test_table_of_values_only_where_a_row_may_need_it(binding, sampler, par, counted):
    B, V = 64, 152064
    dev = sampler.device
    values = dict(top_p=torch.full((B,), 0.9, device=dev), top_k=torch.full((B,), 40, dtype=torch.int32, device=dev), min_p=torch.full((B,), 0.1, device=dev), num_top=5)
    logits, rest = batch(sampler, B, V, W.BF16, False, **{k: values[k] for k in par})
    ctas, name = launched(sampler, logits, **rest)
    assert ctas == 2 * B and ("ILi1ELb1E" in name) == counted, name


# Batches around one and two rounds of the rows that are on the device at once: requests that all have a top-k, or a min-p, get the kernel of smaller and larger batches
@pytest.mark.parametrize("par", [("top_k", "top_p"), ("min_p",), ()])
@pytest.mark.parametrize("dtype", [W.BF16, W.F16, W.F32])
def test_one_kernel_for_a_cta_per_row(binding, par, dtype):
    s = binding.Sampler(max_rows=593, max_vocab=4096)
    dev, names = s.device, set()
    for B in (148, 296, 297, 592, 593):
        values = dict(top_p=torch.full((B,), 0.9, device=dev), top_k=torch.full((B,), 40, dtype=torch.int32, device=dev), min_p=torch.full((B,), 0.1, device=dev))
        logits, rest = batch(s, B, 4096, dtype, False, **{k: values[k] for k in par})
        ctas, name = launched(s, logits, **rest)
        assert ctas == B, (B, ctas, name)
        names.add(name)
    s.close()
    assert len(names) == 1 and "albireo_sample_kernel" in names.pop(), names


# Histories have hash tables where these fit beside two CTAs per SM; calls without histories keep the kernel without the code for them
@pytest.mark.parametrize("dtype,V,history,hashed", [(W.BF16, 175072, True, True), (W.BF16, 175073, True, False), (W.F16, 40000, True, True), (W.BF16, 40000, False, False), (W.F32, 40000, True, False)])
def test_kernel_of_hashed_histories(binding, dtype, V, history, hashed):
    B = 150
    s = binding.Sampler(max_rows=B, max_vocab=V, max_history_total=64 * B)
    logits, par = batch(s, B, V, dtype, history, top_k=torch.full((B,), 40, dtype=torch.int32, device=s.device))
    ctas, name = launched(s, logits, **par)
    s.close()
    assert ctas == B and ("Lb0ELb1E" in name) == hashed, name
