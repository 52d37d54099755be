"""The binding lets other Python threads run while a call waits inside the library, as it does where the launch queue is full."""
import threading
import time

import pytest
import torch

import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.workloads import make_inputs, small_config

pytestmark = pytest.mark.gpu


def test_a_call_that_waits_for_the_launch_queue_lets_other_threads_run():
    cfg = small_config("threads", 1, 16, 16, 1, 32, 8, 4, 4)
    x = {k: v.cuda() for k, v in make_inputs(cfg).items()}
    d = terra.make_desc(cfg)
    o, lse = terra.terra_swin_attn_fwd(d, x["q"], x["k"], x["v"], x["bias"])
    torch.cuda.synchronize()
    longest, stop = [0.0], threading.Event()

    def tick():
        last = time.perf_counter()
        while not stop.is_set():
            time.sleep(0.001)
            now = time.perf_counter()
            longest[0], last = max(longest[0], now - last), now

    ticker = threading.Thread(target=tick)
    ticker.start()
    begin = time.perf_counter()
    torch.cuda._sleep(2_000_000_000)                # about a second of the GPU's clock; the calls behind it fill the queue
    slowest = 0.0
    for _ in range(4000):
        t = time.perf_counter()
        terra.terra_swin_attn_fwd(d, x["q"], x["k"], x["v"], x["bias"], o=o, lse=lse)
        slowest = max(slowest, time.perf_counter() - t)
    stop.set()
    ticker.join()
    torch.cuda.synchronize()
    assert slowest > 0.3, f"no call waited (the longest took {slowest:.3f} s of {time.perf_counter() - begin:.3f}): the test shows nothing"
    assert longest[0] < 0.5 * slowest, f"another thread stood still for {longest[0]:.3f} s while a call waited {slowest:.3f} s"
