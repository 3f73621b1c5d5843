"""The binding gives up the interpreter lock around the launches: a thread that waits for a place in a full launch queue
does not hold up the others."""
import threading
import time

import pytest
import torch

from paper_2411_09909_b200 import amx

pytestmark = pytest.mark.gpu


def test_a_blocked_launch_does_not_stop_other_threads():
    x = torch.randn(16, 512, device="cuda").to(torch.bfloat16)
    codes, scales = amx.quantize(torch.randn(64, 512, device="cuda").to(torch.bfloat16))
    for _ in range(3):
        amx.quant_gemm(x, codes, scales)
    torch.cuda.synchronize()
    longest = []

    def launches():
        for _ in range(1500):                             # two launches each; the queue holds about a thousand
            t = time.perf_counter()
            amx.quant_gemm(x, codes, scales)
            longest.append(time.perf_counter() - t)

    torch.cuda._sleep(int(1.6e9))                         # one kernel of about a second ahead of them
    worker = threading.Thread(target=launches)
    gaps, last = [], time.perf_counter()
    worker.start()
    while worker.is_alive():
        time.sleep(0.002)
        now = time.perf_counter()
        gaps.append(now - last)
        last = now
    torch.cuda.synchronize()
    assert max(longest) > 0.2, "no launch waited for the queue"
    assert max(gaps) < 0.5 * max(longest), (max(gaps), max(longest))
