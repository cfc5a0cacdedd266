"""A launch that fills its time with further chunks ends for those who wait for
it: a short request beside a long one is admitted and handed back as if each
launch ran one chunk, and a cancelled one stops."""
import time

import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    return need_gpu()


@pytest.mark.parametrize("use_graph", [True, False])
def test_short_request_beside_a_long_one(lbm, use_graph):
    # chunks of 0.1 to 0.2 ms (25 reference steps); a launch with nothing
    # waiting runs them for 2 ms.  A request waits for the launch it arrives in
    # and is done with the next: two chunks and the host's work, under 0.5 ms;
    # 2 ms and more if either launch ran its time out
    s = lbm.Server(mem_budget_bytes=1 << 28, max_slots=64, chunk_steps=25, use_graph=use_graph)
    bg = s.submit(lbm.make_request("D2Q37", 256, 0.002, 0.1, tol=1e-30, max_steps=10_000_000))
    time.sleep(0.05)
    rng, ms = np.random.default_rng(0), []
    for _ in range(40):
        time.sleep(rng.uniform(0.0, 0.004))
        t = time.perf_counter()
        rid = s.submit(lbm.make_request("D2Q17", 64, 0.1, 0.1, tol=1e-30, max_steps=150))
        while True:
            done = [r.id for r in s.poll(8)]
            assert bg not in done
            if rid in done:
                break
        ms.append(1e3 * (time.perf_counter() - t))
    cancels = []
    for _ in range(5):
        t = time.perf_counter()
        s.cancel(bg)
        while not s.poll(8):
            pass
        cancels.append(1e3 * (time.perf_counter() - t))
        bg = s.submit(lbm.make_request("D2Q37", 256, 0.002, 0.1, tol=1e-30, max_steps=10_000_000))
        time.sleep(0.02 + rng.uniform(0.0, 0.004))
    s.close()
    assert np.median(ms) < 1.0 and np.median(cancels) < 1.0, (ms, cancels)
