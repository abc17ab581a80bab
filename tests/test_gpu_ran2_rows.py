"""Ran2's shuffle-table entry from the negated output (sum and shifts in place of a
division) and its output from an unsigned maximum: states whose next entry lies at either
edge of each of the 32 intervals of the output, and whose difference of the two generators
is 0, 1 or as large as it gets, continue as the oracle's, in the fills, the one- and
two-oscillator runs (an odd count leaves the second lane a shadow), the paper form and the
overdamped run.  Integers are compared bit for bit; trajectories with the bound that the
transform's 4 ulp give over the steps (as in the other trajectory tests)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

M1, NDIV = 2147483563, 67108862
TRAJ_TOL = 1e-5


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1003_1123_gb300 import gbrng
    gbrng.lib()
    return gbrng


def edge_states(n, seed):
    """The oracle's generator with iy on the intervals' edges and its entry chosen so that
    the next output is the smallest, the largest or the one that wraps."""
    g = oracle.Gen("ran2", seed, n)
    edges = sorted({min(max(j * NDIV + d, 1), M1 - 1) for j in range(33) for d in (-1, 0, 1)})
    for s in range(n):
        st = g.state[s]
        iy = edges[s % len(edges)]
        st[2] = iy
        idum2 = oracle.ran2_schrage(int(st[1]), 1)       # of the next draw
        old = [idum2, idum2 + 1, idum2 - 1, 1, M1 - 1, int(st[3 + iy // NDIV])][s // len(edges) % 6]
        st[3 + iy // NDIV] = min(max(old, 1), M1 - 1)
    return g


def handle(G, g, n):
    r = G.rng_init("ran2", 1, n)
    blob = G.rng_get_state(r)
    payload = G.parse_state(blob)[1]
    G.rng_set_state(r, blob[:len(blob) - len(payload)] + g.state.tobytes())
    return r


def check_state(G, r, g):
    assert G.parse_state(G.rng_get_state(r))[1] == g.state.tobytes()


def rel_err(got, exp):
    got, exp = np.asarray(got, np.float64), np.asarray(exp, np.float64)
    rms = float(np.sqrt((exp * exp).mean())) or 1.0
    return float((np.abs(got - exp) / np.maximum(np.abs(exp), rms)).max())


@pytest.mark.parametrize("n", [1, 33, 594, 1187])
def test_draws_from_edge_states(G, n):
    g = edge_states(n, 5)
    r = handle(G, g, n)
    for items in (n, 3 * n + n // 2, 37 * n):            # one draw, the loop's tail, the loop
        assert np.array_equal(G.rng_fill_u32(r, items).cpu().numpy().view(np.uint32), g.fill_u32(items))
    got = G.rng_fill_uniform(r, 9 * n).cpu().numpy()
    assert np.array_equal(got.view(np.uint32), g.fill_uniform(9 * n).view(np.uint32))
    check_state(G, r, g)


@pytest.mark.parametrize("n,steps", [(1, 19), (595, 7), (77825, 3)])
def test_runs_from_edge_states(G, n, steps):
    """77825 oscillators run two a thread on a GPU of 152 SMs, the last alone."""
    g = edge_states(n, 9)
    r = handle(G, g, n)
    x = torch.ones((n, 3), dtype=torch.float32, device="cuda")
    s = G.LdSystem(r, x, torch.zeros_like(x))
    xo, vo = np.ones((n, 3), np.float32), np.zeros((n, 3), np.float32)
    p = oracle.params()
    for run in (G.ld_run, G.ld_run_stepwise):
        run(s, steps)
        oracle.ld_run_f32(g, xo, vo, p, steps)
        check_state(G, r, g)
        assert rel_err(s.x.cpu().numpy(), xo) < TRAJ_TOL and rel_err(s.v.cpu().numpy(), vo) < TRAJ_TOL
    R = torch.full((n,), 10.0, dtype=torch.float32, device="cuda")
    ou = G.OuSystem(r, R, k_sp=0.01, xi=1.0, kT=4.1, dt=1.0)
    G.ou_run(ou, steps, every=steps)
    Ro = np.full(n, 10.0, np.float32)
    oracle.ou_run_f32(g, Ro, oracle.ou_params(k_sp=0.01, xi=1.0, kT=4.1, dt=1.0), steps, steps)
    check_state(G, r, g)
    assert rel_err(R.cpu().numpy(), Ro) < TRAJ_TOL
