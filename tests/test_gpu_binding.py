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
