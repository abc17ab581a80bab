"""Lagged Fibonacci handles one after another and side by side: a destroyed handle's ring goes to
the next of its row, and every handle's sequence is its seed's all the same."""
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
    yield gbrng
    gbrng.gbrng_set_lfg_order(0)


def words(G, r, n=40000):
    return G.rng_fill_u32(r, n)


@pytest.mark.parametrize("row", range(10))
def test_reused_rings_give_the_seeds_sequence(G, row):
    first = {seed: words(G, G.rng_init_lfg(seed, 1000, row)) for seed in (1, 2, 3)}
    blob = G.rng_get_state(G.rng_init_lfg(2, 1000, row))
    for _ in range(3):
        keep = [G.rng_init_lfg(seed, 1000, row) for seed in (3, 1, 2)]
        copy = G.rng_clone(keep[1])
        for r, seed in zip(keep + [copy], (3, 1, 2, 1)):
            assert torch.equal(words(G, r), first[seed])
        del keep, copy, r
        r = G.rng_init_lfg(9, 1000, row)
        words(G, r, 12345)
        G.rng_set_state(r, blob)
        assert torch.equal(words(G, r), first[2])
        del r


def test_rings_of_other_sizes(G):
    """The last row's ring is larger where order 4 was set: no handle takes the other's."""
    want = words(G, G.rng_init_lfg(5, 10**6, 9), 9 * 10**6)
    for order in (4, 0, 4, 0):
        G.gbrng_set_lfg_order(order)
        assert torch.equal(words(G, G.rng_init_lfg(5, 10**6, 9), 9 * 10**6), want)
    G.gbrng_set_lfg_order(0)


def test_threads_make_and_destroy_handles(G):
    """Eight threads, each on a stream of its own, taking and leaving rings of three rows."""
    want = {row: words(G, G.rng_init_lfg(4, 100, row), 5000) for row in (0, 3, 6)}
    torch.cuda.synchronize()
    bad = []

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            for i in range(12):
                row = (0, 3, 6)[(i + k) % 3]
                r = G.rng_init_lfg(4, 100, row)
                got = words(G, r, 5000)
                if not torch.equal(got, want[row]):
                    bad.append((k, i))
                del r

    threads = [threading.Thread(target=work, args=(k,)) for k in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_kept_rings_are_bounded(G):
    """Forty handles' rings (480 MB and more) are not all kept."""
    import gc
    gc.collect()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    keep = [G.rng_init_lfg(k, 10**6, 9) for k in range(40)]
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] > 40 * (40 << 20)
    del keep
    gc.collect()
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= 128 << 20
