"""The Python binding beside a server's other threads."""
import threading
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    from paper_2606_01927_b200 import binding as Bd
    return Bd


def test_a_launch_that_waits_for_the_queue_lets_other_threads_run(binding):
    """With the device busy and the launch queue full a call blocks; another thread goes on meanwhile."""
    s = binding.Sampler(max_rows=4, max_vocab=1000)
    x = torch.zeros((4, 1000), device=s.device)
    s.albireo_sample(x)
    torch.cuda.synchronize()
    ticks, stop = [], threading.Event()

    def tick():
        while not stop.is_set():
            ticks.append(time.perf_counter())
            time.sleep(0.005)

    t = threading.Thread(target=tick)
    t.start()
    out = (torch.empty(4, dtype=torch.int32, device=s.device), torch.empty(4, device=s.device))
    torch.cuda._sleep(int(1.5e9))                      # a spin of a fixed number of cycles, 0.8 s
    t0 = time.perf_counter()
    longest = 0.0
    for _ in range(4000):                              # several times what the queue takes
        a = time.perf_counter()
        s.albireo_sample(x, out_tokens=out[0], out_logprobs=out[1])
        longest = max(longest, time.perf_counter() - a)
    t1 = time.perf_counter()
    stop.set()
    t.join()
    torch.cuda.synchronize()
    s.close()
    seen = [v for v in ticks if t0 <= v <= t1]
    gap = max(b - a for a, b in zip([t0] + seen, seen + [t1]))
    assert longest > 0.2, longest                      # a call did block
    assert gap < 0.5 * longest, (gap, longest)


def test_out_of_memory_is_torchs(binding):
    s = binding.Sampler(max_rows=4, max_vocab=1000)
    x = torch.zeros((4, 1000), device=s.device)
    with pytest.raises(torch.cuda.OutOfMemoryError):
        s.albireo_sample(x, B=1 << 45)                 # the outputs alone are more than any device holds
    s.close()


def test_host_arrays_off_their_alignment_and_shared_with_results(binding):
    """Through the C ABI: pinned seeds at a 4-byte offset, and results written over an input array, give what plain
    arrays give (such arrays are copied, not read in place)."""
    import ctypes as C
    B, V = 40, 5000
    s = binding.Sampler(max_rows=B, max_vocab=V, host_staging=True)
    g = torch.Generator().manual_seed(1)
    x = torch.randn((B, V), generator=g).pin_memory()
    k = torch.randint(1, 60, (B,), generator=g, dtype=torch.int32).pin_memory()
    seeds = torch.randint(0, 1 << 62, (B,), generator=g).pin_memory()
    want = s.albireo_sample_host(x, top_k=k, seeds=seeds)

    def call(top_k_at, seeds_at, tok_at, lp_at):
        st = torch.cuda.current_stream(s.device)
        rc = binding.LIB.albireo_sample_host(s._handle, x.data_ptr(), B, V, binding.F32, None, top_k_at, None, None, None, None, None,
                                             None, None, 0, seeds_at, 0, tok_at, lp_at, st.cuda_stream, None)
        assert rc == binding.OK, s.last_error()

    off = torch.zeros(8 * B + 8, dtype=torch.uint8).pin_memory()
    C.memmove(off.data_ptr() + 4, seeds.data_ptr(), 8 * B)
    tok, lp = torch.zeros(B, dtype=torch.int32).pin_memory(), torch.zeros(B).pin_memory()
    call(k.data_ptr(), off.data_ptr() + 4, tok.data_ptr(), lp.data_ptr())
    assert (tok == want.tokens).all() and (lp == want.logprobs).all()
    both = torch.zeros(2 * B, dtype=torch.int32).pin_memory()
    both[B // 2:B // 2 + B] = k
    call(both.data_ptr() + 4 * (B // 2), seeds.data_ptr(), both.data_ptr(), lp.data_ptr())      # tokens over half of top_k
    assert (both[:B] == want.tokens).all() and (lp == want.logprobs).all()
    s.close()
