"""The sums of records and statistics, which halve the values before the lanes: records at
every step, several and one to a chunk of 32 steps and one beyond it, by the teams and by
the kernels of one particle a thread with 128- and 256-thread blocks (the last block
partial), against binary64 sums of the positions that runs of `every` steps leave.  Sums of
n terms in any order differ by at most 2 n eps sum|terms|."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
EPS = 2.0**-53


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1003_1123_gb300 import gbrng
    gbrng.lib()
    return gbrng


def ou(G, kind, n):
    R = torch.linspace(-3, 11, n, dtype=torch.float32, device="cuda")
    return G.OuSystem(G.rng_init(kind, 3, n), R, k_sp=0.01, xi=1.0, kT=4.1, dt=1.0)


@pytest.mark.parametrize("kind", ["taus", "ran2", "lcg", "lagfib"])
@pytest.mark.parametrize("n,steps,every", [(17, 99, 1), (1000, 97, 3), (4863, 70, 31), (20001, 65, 32),
                                           (40001, 67, 33), (100003, 9, 2)])
def test_records_are_the_positions_sums(G, kind, n, steps, every):
    a, b = ou(G, kind, n), ou(G, kind, n)
    mean, corr = G.ou_run(a, steps, every)
    R0 = b.R.double().cpu().numpy()
    for r in range(steps // every + 1):
        if r:
            G.ou_run(b, every, every)
        R = b.R.double().cpu().numpy()
        for got, terms in ((mean[r], R), (corr[r], R * R0)):
            assert abs(got * n - terms.sum()) <= 2 * n * EPS * np.abs(terms).sum()


@pytest.mark.parametrize("kind", ["taus", "ran2", "lagfib"])
@pytest.mark.parametrize("n,steps", [(1, 20), (9, 300), (4099, 17), (32801, 3), (200003, 2)])
def test_statistics_are_the_states_sums(G, kind, n, steps):
    """One block, several, and more than the last block adds up."""
    r = G.rng_init(kind, 8, n)
    x = torch.zeros((n, 3), dtype=torch.float32, device="cuda")
    s = G.LdSystem(r, x, torch.zeros_like(x))
    G.ld_init_equilibrium(s)
    st = G.ld_run(s, steps)
    X, V = s.x.double().cpu().numpy(), s.v.double().cpu().numpy()
    for got, terms in ((st["sum_x2"], X * X), (st["sum_v2"], V * V), (st["sum_xv"], X * V)):
        assert abs(got - terms.sum()) <= 2 * terms.size * EPS * np.abs(terms).sum()
