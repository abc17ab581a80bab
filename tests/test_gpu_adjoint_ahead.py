"""The reverse sweep loads the normals of several steps ahead: segments shorter than,
as long as and longer than that, and a last segment of each length, give the same
gradients and end state from kept noise as from regenerated noise."""
import pytest
import torch

from paper_1003_1123_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1003_1123_gb300 import gbrng
    gbrng.lib()
    yield gbrng
    gbrng.ld_set_adjoint_history_limit(-1)


@pytest.mark.parametrize("kind", ["taus", "ran2"])
@pytest.mark.parametrize("steps,ckpt", [(2, 1), (9, 2), (23, 8), (24, 8), (25, 8), (33, 9), (50, 16), (97, 17)])
def test_kept_equals_regenerated(G, kind, steps, ckpt):
    n = 777
    got = []
    for limit in (-1, 0):
        G.ld_set_adjoint_history_limit(limit)
        s = G.LdSystem(G.rng_init(kind, 3, n), *(torch.from_numpy(a).cuda() for a in W.initial_state(n, 4)),
                       K_per=torch.from_numpy(W.spring_constants(n, 5)).cuda())
        r = G.ld_backward(s, steps, ckpt)
        got.append((r["dK"], s.x, s.v, r["loss"], r["dgamma"], r["dkT"], G.rng_get_state(s.rng)))
    a, b = got
    assert all(torch.equal(p, q) for p, q in zip(a[:3], b[:3])) and a[6] == b[6]
    # the same binary32 terms in compensated sums, added up in binary64
    assert all(abs(p - q) <= 1e-12 * abs(q) for p, q in zip(a[3:6], b[3:6]))
