"""What a user of the sampler has it do, as a list of cases that can be timed and compared.

One pass of a case is one call of ``Sampler.albireo_sample`` (or, where the logits start in host
memory, ``Sampler.albireo_sample_host``): the sampling step that follows every decode step.  Logits,
sampling parameters, histories and seeds are in place before the call, as the LM head and the
scheduler leave them; the handle is kept for the life of the program.  Values follow the generators
of ``paper_2606_01927_b200/workloads.py`` (a Gaussian bulk, a Zipf-ranked prior over token ids, a few
dominant tokens, Zipf-distributed histories), made on the GPU.

Fields of a case:
  entry     "device" (all tensors on the GPU) or "host" (pinned host tensors, copies included)
  B, V      rows and vocabulary
  dtype     "f32", "bf16" or "f16"
  logits    "zipf" (Gaussian + Zipf-ranked bias), "spikes" (Gaussian + ten dominant ids),
            "extremes" (Gaussian with near-flat and one-hot-like rows among them)
  cut       which parameters the requests carry: "topk_topp", "topk", "minp_topp", "topp", "none",
            "greedy", or "mixed" (row classes greedy / top-k / top-p / min-p in turn)
  T         temperature of every row (0: drawn per row from U[0.3, 1.5])
  k, p      top-k and top-p of the cuts that use them (p = 0: drawn per row from U[0.5, 1])
  hist      history ids per row, with all three penalties (ragged: U{0..hist} per row); 0: none
  ragged    whether history lengths differ between rows
  num_top   length of the top-N list returned per row
  full      log-probabilities relative to the whole vocabulary
  pieces    1, or the number of vocabulary pieces a row arrives in (sequence-parallel sampling)
"""
import math

import torch

from paper_2606_01927_b200 import binding

_DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
_DEFAULT = dict(entry="device", dtype="bf16", logits="zipf", cut="topk_topp", T=0.7, k=40, p=0.9, hist=0, ragged=False,
                num_top=0, full=False, pieces=1)


def _case(name=None, **kw):
    c = dict(_DEFAULT, **kw)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # one user at a console: a single row, where launch and latency are everything
        _case("single_row", B=1, V=152064),
        # a small batch of fp32 rows with a small vocabulary (configuration 1)
        _case("config1_small_f32", B=8, V=32000, dtype="f32", logits="spikes", cut="topk", T=0.8, k=50),
        # a small batch with an odd vocabulary (rows not 16-byte aligned) and every kind of request in it
        _case("odd_vocab_mixed", B=13, V=50257, cut="mixed", T=0, k=100, p=0, hist=700, ragged=True),
        # requests that set top_p alone, the commonest setting of chat clients
        _case("nucleus", B=32, V=128256, cut="topp", T=1.0, p=0.95),
        # requests that set nothing: plain softmax sampling at temperature 1
        _case("plain_softmax", B=64, V=152064, cut="none", T=1.0),
        # the metric workload: a full decode batch, top-k and top-p
        _case("metric_topk_topp", B=256, V=152064),
        # penalties from 2048-id histories, min-p and top-p (configuration 3)
        _case("config3_penalties", B=256, V=128256, logits="spikes", cut="minp_topp", T=1.0, p=0.95, hist=2048),
        # a large batch in which every request has its own settings (configuration 4)
        _case("config4_mixed", B=512, V=152064, cut="mixed", T=0, k=100, p=0, hist=4096, ragged=True),
        # the largest batch: fp32 rows, penalties, top-20 lists (configuration 5)
        _case("config5_large_f32", B=1024, V=129280, dtype="f32", logits="extremes", T=0.6, k=20, p=0.8, hist=1024, num_top=20),
        # log-probabilities of the model itself and the five likeliest tokens with each, as completion APIs return them
        _case("api_logprobs", B=64, V=128256, cut="topp", T=1.0, p=0.95, num_top=5, full=True),
        # rows in four pieces, as the all-to-all of sequence-parallel sampling leaves them, fp16
        _case("pieces_f16", B=128, V=128256, dtype="f16", T=0.8, k=50, p=0.95, pieces=4),
        # logits that start in pinned host memory
        _case("host_entry", entry="host", B=32, V=152064),
    ]


_MOST_BYTES = 1024 * 129280 * 4      # the logits of the largest listed case


def draw(rng):
    """One more case: batch and vocabulary over their logarithms, every option in its share."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    dtype = rng.choice(["bf16", "bf16", "bf16", "f16", "f32"])
    size = 4 if dtype == "f32" else 2
    V = log_int(16000, 262144)
    if rng.random() < 0.6:
        V -= V % 64                    # vocabularies are padded more often than not
    B = min(log_int(1, 1024), max(1, _MOST_BYTES // (V * size)))
    cut = rng.choice(["topk_topp", "topk_topp", "topk", "minp_topp", "topp", "none", "greedy", "mixed"])
    c = _case(B=B, V=V, dtype=dtype, cut=cut, logits=rng.choice(["zipf", "zipf", "spikes", "extremes"]),
              T=round(rng.uniform(0.5, 1.2), 3), k=log_int(1, 200), p=round(rng.uniform(0.7, 0.98), 3),
              hist=log_int(64, 4096) if rng.random() < 0.5 else 0, ragged=rng.random() < 0.5)
    if cut == "mixed":
        c.update(T=0, p=0)
    extra = rng.random()
    if extra < 0.15:
        c.update(num_top=rng.randint(1, 20), full=rng.random() < 0.5)
    elif extra < 0.3 and V % 64 == 0:
        c.update(pieces=rng.choice([2, 4, 8]))
    elif extra < 0.4 and B * V * size <= 1 << 25:
        c.update(entry="host")
    return c


def _bias(V, s, dev):
    return torch.arange(1, V + 1, dtype=torch.float64, device=dev).log_().mul_(-s).to(torch.float32)


def _logits(case, gen, dev):
    B, V, kind = case["B"], case["V"], case["logits"]
    out = torch.empty((B, V), dtype=_DTYPES[case["dtype"]], device=dev)
    bias = _bias(V, 1.1, dev) if kind == "zipf" else None
    for lo in range(0, B, 128):        # fp32 draws in slices, so that a large batch of 16-bit rows stays small
        n = min(128, B - lo)
        x = torch.randn((n, V), generator=gen, device=dev)
        if kind == "extremes":
            x *= 4.0
            row = torch.arange(lo, lo + n, device=dev) % 100
            x[row == 0] *= 0.0025
            hot = torch.randint(0, V, (n,), generator=gen, device=dev)
            x[torch.arange(n, device=dev), hot] += torch.where(row == 1, 30.0, 0.0)
        else:
            x *= 3.0
            if kind == "zipf":
                x += bias
            else:
                ids = torch.randint(0, V, (n, 10), generator=gen, device=dev)
                x.scatter_add_(1, ids, 6.0 + 4.0 * torch.rand((n, 10), generator=gen, device=dev))
        out[lo:lo + n] = x
    return out


def _parameters(case, gen, dev):
    """The per-row arrays that the case's requests carry; an absent array means "off for every row"."""
    B, cut = case["B"], case["cut"]

    def full(v, dtype=torch.float32):
        return torch.full((B,), v, dtype=dtype, device=dev)

    def uniform(lo, hi):
        return lo + (hi - lo) * torch.rand(B, generator=gen, device=dev)

    par = dict(temperature=full(case["T"]) if case["T"] > 0 else uniform(0.3, 1.5))
    p = full(case["p"]) if case["p"] > 0 else uniform(0.5, 1.0)
    if cut in ("topk", "topk_topp"):
        par["top_k"] = full(case["k"], torch.int32)
    if cut in ("topp", "topk_topp", "minp_topp"):
        par["top_p"] = p
    if cut == "minp_topp":
        par["min_p"] = full(0.05)
    if cut == "greedy":
        par["temperature"] = full(0.0)
    if cut == "mixed":
        cls = torch.arange(B, device=dev) % 4
        k = torch.randint(1, max(2, case["k"] + 1), (B,), generator=gen, device=dev, dtype=torch.int32)
        par["temperature"] = torch.where(cls == 0, 0.0, par["temperature"])
        par["top_k"] = torch.where(cls == 1, k, 0)
        par["top_p"] = torch.where(cls == 2, p, 1.0)
        par["min_p"] = torch.where(cls == 3, uniform(0.01, 0.2), 0.0)
    if case["hist"]:
        lens = (torch.randint(0, case["hist"] + 1, (B,), generator=gen, device=dev) if case["ragged"]
                else torch.full((B,), case["hist"], device=dev))
        off = torch.zeros(B + 1, dtype=torch.int64, device=dev)
        off[1:] = torch.cumsum(lens, 0)
        cdf = torch.cumsum(torch.exp(_bias(case["V"], 1.2, dev).double()), 0)
        n = max(1, int(off[-1]))
        u = torch.rand(n, generator=gen, device=dev, dtype=torch.float64) * cdf[-1]
        par["history_ids"] = torch.searchsorted(cdf, u).clamp_(max=case["V"] - 1).to(torch.int32)
        par["history_offsets"] = off.to(torch.int32)
        par["repetition_penalty"], par["presence_penalty"], par["frequency_penalty"] = full(1.1), full(0.5), full(0.3)
    par["seeds"] = torch.randint(0, 1 << 62, (B,), generator=gen, device=dev)
    return par


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(seed)
    logits = _logits(case, gen, dev)
    par = _parameters(case, gen, dev)
    par["step"] = seed % 4096
    host = case["entry"] == "host"
    if host:
        logits = logits.cpu().pin_memory()
        par = {k: v.cpu().pin_memory() if isinstance(v, torch.Tensor) else v for k, v in par.items()}
    if case["pieces"] > 1:
        t = case["pieces"]
        logits = logits.view(case["B"], t, case["V"] // t).transpose(0, 1).contiguous()
    n_hist = int(par["history_ids"].numel()) if case["hist"] else 0
    sampler = binding.Sampler(max_rows=case["B"], max_vocab=case["V"], max_history_total=n_hist, device=dev, host_staging=host)
    if case["num_top"]:
        par["num_top"] = case["num_top"]
    if case["full"]:
        par["flags"] = binding.FLAG_LOGPROB_FULL_VOCAB
    return dict(call=sampler.albireo_sample_host if host else sampler.albireo_sample, logits=logits, par=par)


def run(state):
    out = state["call"](state["logits"], **state["par"])
    if out.top_ids is None:
        return out.tokens, out.logprobs
    return out.tokens, out.logprobs, out.top_ids, out.top_logprobs


def work(case):
    """Each logit, history id and per-row parameter read once, each result written once; a multiplication
    and a comparison per logit."""
    B, V = case["B"], case["V"]
    size = 4 if case["dtype"] == "f32" else 2
    hist = B * case["hist"] * (0.5 if case["ragged"] else 1.0) * 4 + (B + 1) * 4 if case["hist"] else 0
    return {"bytes": B * V * size + hist + B * 40 + B * (8 + 8 * case["num_top"]), "flops": 2.0 * B * V}


def tolerance(case):
    """Tokens and list ids are whole numbers, equal unless two race scores or the mass at a cut come within
    fp32 rounding of each other.  Log-probabilities are fp32 logarithms of fp32 sums."""
    return {"rel": 1e-5, "max": 1e-4, "differ": 1e-3}
