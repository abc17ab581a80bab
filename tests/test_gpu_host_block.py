"""The pinned block that a host thread's results come back through: taken on the thread's first
such call, handed on when the thread ends, with no CUDA call that another thread's stream
capture forbids."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1003_1123_gb300 import gbrng
    gbrng.lib()
    return gbrng


def system(G, kind="taus", n=5000):
    s = G.LdSystem(G.rng_init(kind, 5, n), torch.zeros((n, 3), device="cuda"), torch.zeros((n, 3), device="cuda"))
    G.ld_init_equilibrium(s)
    return s


def capture(G, a, inside):
    """inside() while this thread captures a run of `a` on a side stream (other threads' calls are
    restricted too, torch's default), then the replay."""
    G.ld_run(a, 10, stats=False)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=torch.cuda.Stream()):
        G.ld_run(a, 10, stats=False)
        inside()
    x = a.x.clone()
    g.replay()
    torch.cuda.synchronize()
    assert not torch.equal(a.x, x)


def test_thread_ends_while_another_captures(G):
    a, b = system(G), system(G)
    ran, leave = threading.Event(), threading.Event()

    def work():
        G.ld_run(b, 10)
        ran.set()
        leave.wait()

    t = threading.Thread(target=work)
    t.start()
    ran.wait()

    def end():
        leave.set()
        t.join()

    capture(G, a, end)


def test_first_call_of_a_thread_while_another_captures(G):
    """Refused, as it synchronises its stream, with that call's error, whether the thread has a
    block or not."""
    b = system(G)
    G.ld_run(b, 10)
    torch.cuda.synchronize()
    codes = []

    def call():
        for _ in range(2):
            try:
                with torch.cuda.stream(torch.cuda.Stream()):
                    G.ld_run(b, 10)
            except G.GbrngError as e:
                codes.append(e.code)

    def other():
        t = threading.Thread(target=call)
        t.start()
        t.join()

    try:
        capture(G, system(G), other)
    except RuntimeError:
        pass          # the refused call ends the capture
    torch.cuda.synchronize()
    assert codes and set(codes) == {-3}
    G.ld_run(b, 10)


def test_many_threads_one_after_another_and_at_once(G):
    """More threads than blocks are kept: every one gets its own run's statistics."""
    import numpy as np
    systems = [system(G, n=1000 + 8 * i) for i in range(80)]
    got = {}

    def work(i):
        for _ in range(3):
            with torch.cuda.stream(torch.cuda.Stream()):
                got[i] = G.ld_run(systems[i], 20)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(80)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for i, s in enumerate(systems):
        v = s.v.double().cpu().numpy()
        assert abs(got[i]["sum_v2"] - (v * v).sum()) <= 2 * v.size * 2.0**-53 * (v * v).sum() + 1e-9
        assert np.isfinite(got[i]["energy_time_avg"])
