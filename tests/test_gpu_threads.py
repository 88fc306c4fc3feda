"""The torch-tensor calls let other Python threads run while a launch waits for room in the stream's queue."""
import threading
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bd():
    from paper_2304_11267_b200 import binding
    from paper_2304_11267_b200 import build
    build.build()
    binding.load()
    return binding


@pytest.mark.parametrize("what", ["attention", "geglu", "groupnorm", "conv"])
def test_a_full_queue_does_not_stop_other_threads(bd, what):
    x = torch.zeros(1, 8, 16, 64, dtype=torch.float16, device="cuda")
    if what == "attention":
        a, out = bd.Attention(), torch.empty_like(x)
        call = lambda: a.forward(x, x, x, out=out)  # noqa: E731
    elif what == "geglu":
        out = torch.empty(1, 8, 16, 32, dtype=torch.float16, device="cuda")
        call = lambda: bd.geglu(x, out=out)  # noqa: E731
    elif what == "groupnorm":
        out = torch.empty_like(x)
        call = lambda: bd.groupnorm(x, 4, out=out)  # noqa: E731
    else:
        layer, out = bd.WinogradConv3x3(torch.zeros(64, 3, 3, 64, dtype=torch.float16, device="cuda")), torch.empty_like(x)
        call = lambda: layer(x, out=out)  # noqa: E731
    call()
    torch.cuda.synchronize()
    ticks, stop = [], threading.Event()

    def tick():
        while not stop.wait(0.002):
            ticks.append(time.perf_counter())

    other = threading.Thread(target=tick)
    other.start()
    time.sleep(0.05)
    begin = time.perf_counter()
    torch.cuda._sleep(1_500_000_000)    # 0.75 s and more of GPU time in front of the calls
    for _ in range(3000):               # (a stream's queue holds about a thousand launches)
        call()
    end = time.perf_counter()
    torch.cuda.synchronize()
    stop.set()
    other.join()
    assert end - begin > 0.5, "the calls did not wait: nothing was tested"
    during = [begin] + [t for t in ticks if begin < t < end] + [end]
    longest = max(b - a for a, b in zip(during, during[1:]))
    assert longest < 0.25, "the other thread stood still for %.2f s" % longest
