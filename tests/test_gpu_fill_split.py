"""Fills of few streams cut each stream's draws into segments (generators jumped
ahead): the words, normals and states equal those of short fills, which take one
thread a stream, bit for bit, at the edges of the segments."""
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


@pytest.mark.parametrize("kind", ["taus", "lcg"])
@pytest.mark.parametrize("op", ["u32", "uniform", "normal"])
@pytest.mark.parametrize("streams,items", [
    (1, 5000), (7, 64), (7, 65 * 64 + 3), (9, 32 * 128 + 1), (1000, 2047), (1025, 2049), (4096, 256),
    (50001, 130), (60800, 65), (60801, 130),
])
def test_split_equals_short_fills(G, kind, op, streams, items):
    fill = {"u32": G.rng_fill_u32, "uniform": G.rng_fill_uniform, "normal": G.rng_fill_normal}[op]
    per = 2 if op == "normal" else 1
    n = (streams * items - streams // 3) * per     # a last, partial row of items
    a, b = G.rng_init(kind, 41, streams), G.rng_init(kind, 41, streams)
    whole = fill(a, n)
    row = 60 * streams * per                       # fewer than 64 items a stream
    parts = torch.cat([fill(b, min(row, n - k)) for k in range(0, n, row)])
    assert torch.equal(whole.view(torch.int32), parts.view(torch.int32))
    # a partial last row leaves the streams' own counts: compare the next draws too
    assert G.rng_get_state(a) == G.rng_get_state(b)
