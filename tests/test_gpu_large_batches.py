"""Parity of the kernel that ordinary calls with more than 74 rows run (one CTA per row, nothing asked for beyond tokens,
log-probabilities and top-N lists), and of the same rows with counts, which another instantiation serves."""
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
    s = binding.Sampler(max_rows=192, max_vocab=80000, max_history_total=1 << 20)
    yield s
    s.close()


def every_kind_of_request(B, V, dtype, history, seed):
    rng = np.random.default_rng(seed)
    x = (rng.standard_normal((B, V)) * 2.5 - 1.1 * np.log(np.arange(1, V + 1))).astype(np.float32)
    x[1::7] = np.round(x[1::7])                        # rows of ties
    cls = np.arange(B) % 8                             # greedy, top-k (small, large), both, min-p, top-p, nothing, top-k with min-p
    w = W.Workload("mixed", B, V, W.F32 if dtype == W.F16 else dtype, x if dtype != W.BF16 else W.f32_to_bf16_bits(x),
                   temperature=np.where(cls == 0, 0.0, rng.uniform(0.5, 1.3, B)).astype(np.float32),
                   top_k=np.select([cls == 1, cls == 2, cls == 3, cls == 7], [rng.integers(1, 65, B), rng.integers(65, 257, B), 40, 100], 0).astype(np.int32),
                   top_p=np.where((cls == 3) | (cls == 5), rng.uniform(0.3, 0.98, B), 1.0).astype(np.float32),
                   min_p=np.where((cls == 4) | (cls == 7), 10.0 ** rng.uniform(-4, -1, B), 0.0).astype(np.float32),
                   seeds=rng.integers(0, 1 << 62, B).astype(np.uint64), step=77)
    if history:
        lens = rng.integers(0, 1500, B)
        w.history_offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
        w.history_ids = np.minimum(rng.zipf(1.2, int(lens.sum())) - 1, V - 1).astype(np.int32)
        w.repetition_penalty, w.presence_penalty, w.frequency_penalty = (np.full(B, v, np.float32) for v in (1.2, 0.4, 0.2))
        w.output_start = np.where(np.arange(B) % 3 == 0, 300, 0).astype(np.int32)
    return W.as_f16(w) if dtype == W.F16 else w


def against_oracle(w, g):
    ref = O.sample(w, threads=_CORES)
    rep = compare(w, g, ref)
    assert rep.ok() and len(rep.excused) <= 1, (rep.summary(), rep.failures[:3], rep.excused[:3])
    bad = compare_top_lists(w, g, ref)
    assert not bad, bad[:3]


# 90 rows: a deep ring, an SM to each row; 160: two rows per SM.  70001: rows off the 16-byte grid; 4 to 9 tiles
@pytest.mark.parametrize("B", [90, 160])
@pytest.mark.parametrize("dtype", [W.F32, W.BF16, W.F16])
@pytest.mark.parametrize("history", [False, True])
@pytest.mark.parametrize("layout", ["rows", "pieces", "buffers"])
def test_ordinary_calls(binding, sampler, B, dtype, history, layout):
    V = 70001 if layout == "rows" else 70016
    w = every_kind_of_request(B, V, dtype, history, 71)
    t = binding.workload_tensors(w, sampler.device)
    lg = t.pop("logits")
    args = {"logits": lg}
    if layout != "rows":
        pieces = [lg[:, j * (V // 4):(j + 1) * (V // 4)].contiguous() for j in range(4)]
        args = dict(logits=torch.stack(pieces)) if layout == "pieces" else dict(logits=pieces[0], segment_tensors=pieces, B=B, V=V)
    for num_top in (0, 6):
        w.num_top = num_top
        plain = to_host(sampler.albireo_sample(**args, **t, num_top=num_top))
        more = to_host(sampler.albireo_sample(**args, **t, num_top=num_top, want_counts=True, want_status=True))
        assert (plain["tokens"] == more["tokens"]).all()
        assert (plain["logprobs"].view(np.uint32) == more["logprobs"].view(np.uint32)).all()
        if num_top:
            assert (plain["top_ids"] == more["top_ids"]).all()
            # (the kept sizes of the call with counts say which rows' lists can be compared)
            plain["num_kept"] = more["num_kept"]
            against_oracle(w, plain)


@pytest.mark.parametrize("dtype", [W.F32, W.BF16])
@pytest.mark.parametrize("option", ["exp1", "keep_ties", "full", "full_list"])
def test_options_beyond_the_ordinary(binding, sampler, dtype, option):
    B, V = 80, 40003
    w = every_kind_of_request(B, V, dtype, True, 73)
    w.num_top = 0 if option == "full" else 6
    flags = 0
    if option == "exp1":
        w = W.with_exp1(w, seed=9)
    if option == "keep_ties":
        w.topk_keep_ties, flags = True, binding.FLAG_TOPK_KEEP_TIES
    if option.startswith("full"):
        w.logprob_full_vocab, flags = True, binding.FLAG_LOGPROB_FULL_VOCAB
    t = binding.workload_tensors(w, sampler.device)
    g = to_host(sampler.albireo_sample(t.pop("logits"), **t, num_top=w.num_top, want_counts=True, flags=flags))
    against_oracle(w, g)


@pytest.mark.parametrize("B", [5, 40, 90])
def test_a_call_sees_what_the_kernel_ahead_of_it_wrote(binding, sampler, B):
    """The kernel may be scheduled while the one ahead of it still runs: logits and parameters written just before
    the call, and results read just after it, in a stream and in a captured graph with a side stream."""
    V, n = 60000, 6
    g = torch.Generator(device=sampler.device).manual_seed(2)
    src = torch.randn((n, B, V), generator=g, device=sampler.device) * 3
    temps = torch.rand((n, B), generator=g, device=sampler.device) + 0.3
    ks = torch.randint(1, 100, (n, B), generator=g, device=sampler.device, dtype=torch.int32)
    seeds = torch.arange(B, device=sampler.device)
    want = []
    for i in range(n):
        torch.cuda.synchronize()
        want.append(sampler.albireo_sample(src[i], temperature=temps[i], top_k=ks[i], seeds=seeds).tokens)
    want = torch.stack(want)
    x, T, k = torch.empty((B, V), device=sampler.device), torch.empty(B, device=sampler.device), torch.empty(B, dtype=torch.int32, device=sampler.device)
    tok, lp = torch.empty(B, dtype=torch.int32, device=sampler.device), torch.empty(B, device=sampler.device)
    got = torch.empty((n, B), dtype=torch.int32, device=sampler.device)

    def steps(stream, side):
        for i in range(n):
            torch.add(src[i], 0.0, out=x)              # a kernel that takes longer than the launch of the next
            if side is not None:                       # (and one on another stream that the call depends on too)
                side.wait_stream(stream)
                with torch.cuda.stream(side):
                    torch.mul(temps[i], 1.0, out=T)
                stream.wait_stream(side)
            else:
                torch.mul(temps[i], 1.0, out=T)
            k.copy_(ks[i])
            sampler.albireo_sample(x, temperature=T, top_k=k, seeds=seeds, out_tokens=tok, out_logprobs=lp, stream=stream)
            torch.add(tok, 0, out=got[i])
            sampler.albireo_sample(x, temperature=T, top_k=k, seeds=seeds, out_tokens=tok, out_logprobs=lp, stream=stream)   # (back to back)

    st, side = torch.cuda.Stream(device=sampler.device), torch.cuda.Stream(device=sampler.device)
    for s2 in (None, side):
        got.fill_(-1)
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            steps(st, s2)
        torch.cuda.synchronize()
        assert torch.equal(got, want)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            steps(st, s2)
        for _ in range(2):
            got.fill_(-1)
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(got, want)
