"""Other Python threads run while a call of the native module waits for the device."""
import threading
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["quantize", "dequantize"])
def test_a_full_launch_queue_does_not_stop_the_other_threads(name):
    """The device is kept busy for about half a second, and more kernels are enqueued behind that than a stream's launch
    queue holds, so that the enqueueing thread has to wait in a launch; another thread counts on meanwhile."""
    from paper_2503_18893_b200 import xkv
    x = torch.randn(4, 64, device="cuda").to(torch.bfloat16)
    codes, meta = xkv.xkv_quantize_rtn(x)
    call = (lambda: xkv.xkv_quantize_rtn(x)) if name == "quantize" else (lambda: xkv.xkv_dequantize_rtn(codes, meta))
    call()
    torch.cuda.synchronize()
    stamps, stop = [], threading.Event()

    def count():
        while not stop.is_set():
            stamps.append(time.perf_counter())
            time.sleep(0.002)

    t = threading.Thread(target=count)
    t.start()
    time.sleep(0.02)
    torch.cuda._sleep(1_000_000_000)                       # cycles: half a second at 1.9 GHz
    begin = time.perf_counter()
    for _ in range(4000):
        call()
    end = time.perf_counter()
    stop.set()
    t.join()
    torch.cuda.synchronize()
    assert end - begin > 0.3                               # the queue was full: the calls had to wait for the device
    inside = [begin] + [s for s in stamps if begin < s < end] + [end]
    assert max(b - a for a, b in zip(inside, inside[1:])) < 0.3     # with the lock held: all of it
