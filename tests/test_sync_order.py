"""Orderings that the kernels need and that no run can be relied on to miss: read from the
sources, as which of a block's warps comes first is the hardware's choice."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1003_1123_gb300", "csrc")


def source(name):
    """A source file without its comments."""
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def body(text, name):
    """The definition of a function, from its name to the brace that closes it."""
    at = re.search(r"\b%s\([^;{]*\)\s*\{" % name, text)
    assert at, name
    depth, i = 1, at.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[at.start():i]


def test_team_states_are_loaded_before_any_is_stored():
    """Every producer warp of a block loads all its oscillators' generator states; the warp of
    the run's last chunk stores the end states to the same words.  A barrier of all producer
    warps has to lie between, and before any of them may leave."""
    f = body(source("team.cu"), "team_produce")
    loads = [m.end() for m in re.finditer(r"=\s*(?:taus_load\()?a\.(?:taus|lcg)\[i\]", f)]
    stores = [m.start() for m in re.finditer(r"a\.(?:taus|lcg)\[idx\[j\]\]\s*=", f)]
    leaves = [m.start() for m in re.finditer(r"\breturn\b", f)]
    barrier = [m.start() for m in re.finditer(r"bar_sync\(BAR_LOADED, S::kProducers\)", f)]
    assert len(loads) == 2 and len(stores) == 2 and len(barrier) == 1 and leaves
    assert max(loads) < barrier[0] < min(stores + leaves)
    s = source("team.cu")
    assert re.search(r"threadIdx\.x < S::kProducers\)\s*team_produce", s)   # all of them, and no other warp


def test_last_block_reads_partials_behind_the_fence():
    """The last block's lane 0 counts the blocks and fences; the other lanes read what the
    other blocks left only after a warp barrier, which orders memory (a shuffle does not)."""
    f = body(source("device.cuh"), "store_stats")
    count, read = f.index("atomicAdd(s.ticket"), f.index("__ldcg(s.partials")
    fence = f.index("__threadfence()", count)
    assert count < fence < f.index("__syncwarp()", fence) < read


def test_aligned_barriers_are_taken_by_whole_warps():
    """The aligned barriers want the warp converged: each stands in a helper that brings it
    together first, and nowhere else."""
    helpers = ("bar_sync", "bar_arrive", "cluster_sync")
    device = source("device.cuh")
    for name in helpers:
        f = body(device, name)
        assert "__syncwarp()" in f and f.index("__syncwarp()") < f.index("asm volatile"), name
        device = device.replace(f, "")
    texts = {n: source(n) for n in sorted(os.listdir(CSRC)) if n.endswith((".cu", ".cuh"))}
    texts["device.cuh"] = device
    for n, text in texts.items():
        assert not re.search(r'"[^"]*\bbar(?:rier)?\.', text), n


def test_warps_leave_a_failed_launch_by_its_round():
    """A wait that ran out in round r + 1 can be recorded before a using warp has looked past
    round r's barrier; it may leave only for round r's failure, as round r + 1's barrier
    counts on it.  So no flag: the round, and every warp inside the rounds asks for its own."""
    head = source("lfg.cuh")
    assert "<= r" in body(head, "round_failed")
    assert re.search(r"failed\s*=\s*r;", body(head, "wait_warp"))
    for name, kernels in (("lfg.cu", 1), ("lfg_run.cu", 2), ("lfg_ou.cu", 1), ("lfg_team.cu", 1)):
        text = source(name)
        assert text.count("__shared__ int64_t s_failed;") == kernels == text.count("s_failed = kNoRound;")
        assert not re.search(r"if \((?:\*\(volatile[^)]*\)&)?s_failed\)", text)      # as a flag
        # past each BAR_GO, the round of the loop that it closes
        for at in (m.end() for m in re.finditer(r"bar_sync\(BAR_GO, T\);", text)):
            assert re.match(r"\s*if \(round_failed\(&s_failed, [rp]\)\) (?:break|return);", text[at:]), name
