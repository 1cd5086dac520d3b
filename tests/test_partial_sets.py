"""The bookkeeping of a workspace's two sets of tile partials (csrc/sdv_sets.h), on the CPU:
a call may skip the wait before its stores (fresh = 0) only where nothing but calls of its
own layout, in its own set, has written since the workspace became known."""
import os
import random
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2606_13426_gb300", "csrc")


@pytest.fixture(scope="module")
def replay(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("sets") / "partial_sets_check")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + CSRC, os.path.join(HERE, "partial_sets_check.cpp"), "-o", exe],
                   check=True)

    def run(calls):
        text = "".join("%d %d\n" % c for c in calls)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return run


def _blocks(slots, chosen):
    """The 256-byte blocks of a set: 20 bytes a slot, rounded up; set 1 follows set 0."""
    n = -(-20 * slots // 256)
    return range(chosen * n, (chosen + 1) * n)


def _check(calls, got):
    last = {}                                        # (workspace, block) -> (layout, set) that wrote it last
    for (ws, slots), (chosen, fresh) in zip(calls, got):
        for blk in _blocks(slots, chosen):
            if not fresh:
                assert last.get((ws, blk)) == (slots, chosen), (ws, slots, chosen, blk)
            last[ws, blk] = (slots, chosen)


# A large call, a small one whose set 1 lies inside the large one's set 0, and the large one
# again: its set's last own layout is its own, yet the small call has written there.
@pytest.mark.parametrize("sizes", [(2048, 640, 2048), (640, 2048, 640, 2048), (2048, 2048, 640, 2048, 2048),
                                   (100, 101, 100, 101, 100)])
def test_a_set_that_another_layout_wrote_is_fresh(replay, sizes):
    calls = [(4096, s) for s in sizes]
    _check(calls, replay(calls))


def test_random_runs_of_calls(replay):
    rng = random.Random(3)
    # 4096 and 4096 + 64 * 256 share a place in the table, so that one makes the other forgotten
    calls = [(rng.choice([4096, 4096, 8192, 4096 + 64 * 256]), rng.choice([64, 640, 700, 2048])) for _ in range(4000)]
    _check(calls, replay(calls))


def test_a_run_of_one_layout_alternates_and_waits_only_at_its_start(replay):
    got = replay([(4096, 640)] * 8)
    assert [s for s, _ in got] == [0, 1] * 4
    assert [f for _, f in got] == [1, 1] + [0] * 6
