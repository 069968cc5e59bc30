"""The Python module of the native calls: built against the torch it is loaded beside, other threads run meanwhile, and
arguments are taken as before it existed."""
import threading
import time

import pytest
import torch

from paper_2607_27735_b200 import binding, build


def test_module_of_another_torch_is_rebuilt_and_not_loaded(monkeypatch):
    assert build._native_current()
    assert binding._nat().abi == build.native_abi()
    monkeypatch.setattr(torch, "__version__", "0.0.0+other")
    assert not build._native_current()  # by content, whatever its date
    monkeypatch.setattr(binding, "_native", None)
    with pytest.raises(ImportError, match="0.0.0"):
        binding._nat()


@pytest.mark.gpu
def test_a_launch_that_waits_for_room_leaves_other_threads_running():
    state = torch.tensor([1.0, 4.0], device="cuda")
    entropy = torch.rand(8, device="cuda")
    m = torch.tensor([3], dtype=torch.int32, device="cuda")
    binding.spec_controller_update(state, entropy, m, 0.9)
    torch.cuda.synchronize()
    gaps, stop = [], threading.Event()

    def tick():
        last = time.perf_counter()
        while not stop.is_set():
            time.sleep(0.002)
            now = time.perf_counter()
            gaps.append(now - last)
            last = now

    t = threading.Thread(target=tick)
    t.start()
    try:
        torch.cuda._sleep(1_000_000_000)  # half a second on the device; the launches behind it fill the queue
        longest = 0.0
        for _ in range(6000):
            t0 = time.perf_counter()
            binding.spec_controller_update(state, entropy, m, 0.9)
            longest = max(longest, time.perf_counter() - t0)
        torch.cuda.synchronize()
    finally:
        stop.set()
        t.join()
    assert longest > 0.1, "no launch had to wait: the test shows nothing"
    assert max(gaps) < 0.5 * longest


@pytest.mark.gpu
def test_the_bound_of_the_lengths_may_be_a_float():
    committed = torch.tensor([50, 995], dtype=torch.int32, device="cuda")
    binding.spec_advance_lengths(committed, None, 8, max_len=1000.0)
    assert committed.tolist() == [50, 991]
