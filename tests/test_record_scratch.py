"""The overdamped runs' record scratch keeps to what the header promises, 16 bytes per record
and 256 particles or 256 MiB where that is more, whatever number of slots a kernel takes, and
the calls refused are those of the rule by blocks of 256 particles."""
import os
import subprocess

import numpy as np
import pytest
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RULES = r"""
#include <cassert>
#include <cstdio>
#include "records.h"
using namespace gb;
int main()
{
    const int sms = 152;
    const int64_t counts[] = {1, 2, 11, 1001, 100001, 10000001, 100000001, 268435456, 268435457, 0x7fffffffll,
                              0x80000000ll, 1ll << 40};
    for (int64_t n = 1; n <= 2000000; n += n < 5000 ? 1 : n < 100000 ? 7 : 331) {
        const int64_t b256 = (n + 255) / 256;
        for (int64_t r : counts) {
            const double promise = std::max(16.0 * (double)r * (double)b256, 256.0 * 1048576);
            // refused: 2^31 records, or more than 4 GiB at one slot for 256 particles
            assert(records_refused(r, record_blocks(n)) == (r > 0x7fffffff || 16.0 * (double)r * (double)b256 > 4294967296.0));
            for (int order : {1, 2, 4})
                assert(lfg_record_blocks(n, sms, order) == std::min<int64_t>(b256, (order == 4 ? 4 : 5) * sms));
            // the kernels of more slots, where they may run
            for (int64_t per : {8, 16, 128, 256}) {
                const int64_t slots = (n + per - 1) / per;
                if (records_fit(r, slots, n)) assert(16.0 * (double)r * (double)slots <= promise);
                if (per == 256) assert(records_fit(r, slots, n));
            }
        }
        // one launch of the shared sequence, whichever of its kernels: a slot a CTA, or one a using warp
        const int64_t share = lfg_share(n, sms), most = lfg_launch_records(n, sms);
        assert(share % 2 == 0 && share * sms >= n && most >= 2);
        for (int unit : {32, 64}) {
            const int slots = lfg_record_slots(share, unit);
            assert(slots >= 1 && slots <= kOuWarps);
            assert(16 * most * sms * slots <= kRecordScratch);
        }
    }
    puts("ok");
}
"""


def test_rules(tmp_path):
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    src.write_text(RULES)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1003_1123_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout == "ok\n"


@pytest.mark.gpu
@pytest.mark.parametrize("kind,n,steps,sparse", [
    ("lagfib", 100, 250001, 50),      # a slot a CTA: three launches
    ("lagfib", 100000, 15000, 25),    # a slot a using warp: three launches
    ("taus", 10000, 60000, 100),      # too many for the teams' slots: one particle a thread
    ("lcg", 10000, 60000, 100),
])
def test_many_records(kind, n, steps, sparse):
    """A record after every step against one every `sparse` steps, which fits one launch: the same
    positions and states, the same sums up to their order; and the scratch within its bound."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1003_1123_gb300 import gbrng as G
    kw = dict(k_sp=0.01, xi=1.0, kT=4.1, dt=1.0)
    R0 = torch.linspace(-3, 4, n, device="cuda")
    a = G.OuSystem(G.rng_init(kind, 7, n), R0.clone(), **kw)
    b = G.OuSystem(G.rng_init(kind, 7, n), R0.clone(), **kw)
    mean_b, corr_b = G.ou_run(b, steps, sparse)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    mean_a, corr_a = G.ou_run(a, steps, 1)
    used = free - torch.cuda.mem_get_info()[0]
    assert used <= max(16 * (steps + 1) * ((n + 255) // 256), 256 << 20) + (16 << 20)   # 16 MiB: the sums and R(0)
    assert torch.equal(a.R, b.R)
    assert G.rng_get_state(a.rng) == G.rng_get_state(b.rng)
    # any order of n terms' sum: 2 n eps of the terms' mean size, which is below 50
    tol = 2 * n * 2.0**-53 * 50
    assert np.abs(np.asarray(mean_a)[::sparse] - mean_b).max() <= tol
    assert np.abs(np.asarray(corr_a)[::sparse] - corr_b).max() <= 4 * tol
    # and the last record against the positions themselves
    if steps % sparse == 0:
        assert abs(mean_a[-1] - a.R.double().mean().item()) <= tol
        assert abs(corr_a[-1] - (a.R.double() * R0.double()).mean().item()) <= 4 * tol


@pytest.mark.gpu
def test_refused_record_counts():
    """2^28 + 1 records of one block of particles are refused, with nothing run."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import ctypes as C
    from paper_1003_1123_gb300 import gbrng as G
    for kind in ("taus", "ran2", "lcg", "lagfib"):
        s = G.OuSystem(G.rng_init(kind, 7, 256), torch.ones(256, device="cuda"), k_sp=0.01, xi=1.0, kT=4.1, dt=1.0)
        before = G.rng_get_state(s.rng)
        cs, one = s.c_struct(), np.zeros(1)
        rc = G.lib().ou_run(C.byref(cs), 2**28, 1, one.ctypes.data, one.ctypes.data, None)
        assert rc == -1 and one[0] == 0.0
        assert bool((s.R == 1).all()) and G.rng_get_state(s.rng) == before
