"""The binding gives up the interpreter lock around the launches: a thread that waits for a place in a full launch queue
does not hold up the others, and threads are inside the library at the same time."""
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


def test_threads_on_their_own_streams_do_not_disturb_each_other():
    """Two threads inside the library at once, each on its own stream with its own operands, across the entry points that
    allocate, configure kernels and encode tensor maps: the results of one thread alone."""
    def problem(seed):
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        bf = lambda *s: torch.randn(*s, device="cuda", generator=g).to(torch.bfloat16)
        x, w, q, k, v = bf(200, 1024), bf(512, 1024), bf(4, 544, 128), bf(2, 544, 128), bf(2, 544, 128)

        def calls():
            codes, scales = amx.quantize(w)
            prepared = amx.quantize_prepared(w, True)[2]
            a = amx.quantize_prepared(x, False)[2]
            return [amx.quant_gemm(x, codes, scales), amx.quant_gemm(x[:3], codes, scales), amx.quant_gemm(x, w_bf16=w, flags=amx.GEMM_FP4),
                    amx.gemm_prepared(a, prepared, 200, 512, 1024), amx.attention_heads(q, k, v, amx.ATTN_CAUSAL)]
        return calls

    problems = [problem(1), problem(2)]
    want = [p() for p in problems]
    torch.cuda.synchronize()
    got = [[], []]

    def run(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(20):
                got[i].append(problems[i]())
            torch.cuda.current_stream().synchronize()

    threads = [threading.Thread(target=run, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(2):
        assert len(got[i]) == 20
        assert all(torch.equal(g, w) for r in got[i] for g, w in zip(r, want[i]))
