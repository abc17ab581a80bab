"""Lagged Fibonacci launches whose dynamic shared memory fills the 48 KB that a kernel has without
asking, to the byte or but for its static part: each in a process of its own, as a larger
launch before it would have asked for more."""
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUNS = {
    # 32 units of 64 oscillators a CTA (152 SMs)
    "resident": """
n = 305000
s = G.LdSystem(G.rng_init("lagfib", 3, n), torch.zeros((n, 3), device="cuda"), torch.zeros((n, 3), device="cuda"))
G.ld_run(s, 3)
assert bool(torch.isfinite(s.x).all()) and bool((s.v != 0).any())
""",
    # 34 oscillators a CTA, three normals of 120 steps: 48960 bytes and 488 of its own
    "small systems": """
n = 5000
for row in range(6, 10):
    s = G.LdSystem(G.rng_init_lfg(3, n, row), torch.zeros((n, 3), device="cuda"), torch.zeros((n, 3), device="cuda"))
    G.ld_run(s, 120)
    assert bool((s.v != 0).any())
""",
    # 6144 particles a CTA, R and R(0)
    "overdamped": """
n = 928107
o = G.OuSystem(G.rng_init("lagfib", 3, n), torch.zeros(n, device="cuda"))
mean, corr = G.ou_run(o, 3, 1)
assert len(mean) == 4
""",
    # rows 7, 8, 9: 24 units of 64 offsets eight deep, 32 of 96 four deep, of 192 two deep
    "fills": """
for row, n in ((7, 230000), (8, 460000), (9, 920000)):
    for fill in (G.rng_fill_u32, G.rng_fill_uniform, G.rng_fill_normal):
        fill(G.rng_init_lfg(3, 1000, row), n)
""",
}


@pytest.mark.parametrize("what", list(RUNS))
def test_first_launch_of_48_kb(what):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    code = "import torch\nfrom paper_1003_1123_gb300 import gbrng as G\n" + RUNS[what] + "torch.cuda.synchronize()\n"
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr[-600:]


def test_threads_with_launches_of_several_sizes():
    """Threads that launch the same kernels with more and with less shared memory: neither takes
    the other's limit away."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import threading
    from paper_1003_1123_gb300 import gbrng as G
    errors = []
    fills = [(G.rng_init_lfg(k, 1000, 9), n) for k, n in enumerate((10**6, 15 * 10**5, 21 * 10**5))]
    runs = []
    for n in (310000, 600000, 900000):
        runs.append(G.LdSystem(G.rng_init("lagfib", 3, n), torch.zeros((n, 3), device="cuda"),
                               torch.zeros((n, 3), device="cuda")))
    torch.cuda.synchronize()

    def work(f):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(60):
                    f()
        except G.GbrngError as e:
            errors.append(str(e))

    jobs = [lambda r=r, n=n: G.rng_fill_uniform(r, n) for r, n in fills]
    jobs += [lambda s=s: G.ld_run(s, 2, stats=False) for s in runs]
    threads = [threading.Thread(target=work, args=(f,)) for f in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
