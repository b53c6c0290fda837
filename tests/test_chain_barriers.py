"""The chain kernels' named barriers, read from their source (a broken hand-over
must not be tried on a GPU).

barrier.cta.*.aligned wants every lane of a warp at the same instruction, and the
code around the hand-overs branches per lane.  So the aligned forms occur only in
bar_sync and bar_arrive, and both bring the warp together (__syncwarp) directly
before the instruction.  Arrivals and waits use the thread counts that the
barriers' descriptions give: one count per barrier, the same in both kernels."""
import os
import re

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2507_21239_gb300", "csrc")
CHAINS = ["mcd_collide_chain.cuh", "mcd_collide_chain64.cuh"]


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_aligned_barriers_start_from_a_whole_warp():
    helper = re.compile(r"void (bar_sync|bar_arrive)\(int id, int count\)\s*\{\s*__syncwarp\(\);\s*"
                        r"asm volatile\(\"barrier\.cta\.(sync|arrive)\.aligned %0, %1;\"[^;]*;\s*\}")
    found = helper.findall(_source(CHAINS[0]))
    assert sorted(found) == [("bar_arrive", "arrive"), ("bar_sync", "sync")]
    for name in sorted(os.listdir(CSRC)):
        assert _source(name).count("barrier.cta") == (len(found) if name == CHAINS[0] else 0), name


def test_one_thread_count_per_barrier():
    for name in CHAINS:
        counts = {}
        for bar, n in re.findall(r"bar_(?:sync|arrive)\((kBar\w+), ([^)]*)\)", _source(name)):
            counts.setdefault(bar, set()).add(n)
        assert counts and all(len(c) == 1 for c in counts.values()), (name, counts)
