"""Rules of the kernels' barrier code that no run on a GPU can show broken (a missing order between a wait and what it
guards, a wait where only a look is meant): read from the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_15383_b200", "csrc")


def sources():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            yield name, re.sub(r"//[^\n]*", "", f.read())


def test_a_warp_goes_on_only_when_every_lane_has_seen_the_barrier():
    """A lane's memory accesses are ordered behind its own successful wait on an mbarrier, not behind another lane's: a vote
    on the outcome has to ask for all lanes."""
    votes = [(name, v) for name, text in sources() for v in re.findall(r"__(any|all)_sync\(\s*0xffffffffu\s*,\s*mbar_", text)]
    assert votes and all(v == "all" for _, v in votes), votes


def test_the_issue_loop_only_looks_ahead():
    """mbarrier.try_wait may suspend its thread: outside the waits themselves (mbar.cuh's, and loops that spin on it) a
    barrier is looked at with test_wait, so that work in hand is not held back by a barrier that is not due yet."""
    for name, text in sources():
        if name == "mbar.cuh":
            continue
        ahead = [line.strip() for line in text.splitlines() if re.search(r"mbar_try(_at)?\(", line) and not re.search(r"\bwhile\s*\(", line)]
        assert not ahead, (name, ahead)


def test_a_refused_launch_is_not_dropped():
    """A launcher that answers whether it launched is [[nodiscard]], and no call of one stands by itself: what comes behind it
    would read the buffers of an earlier call."""
    launchers = set()
    for name, text in sources():
        if name == "common.cuh":
            for mark, fn in re.findall(r"^(\[\[nodiscard\]\] )?bool (launch_\w+)\(", text, re.M):
                assert mark, fn
                launchers.add(fn)
    assert {"launch_stream_wave", "launch_tc_stream_wave", "launch_prefill_wave"} <= launchers
    for name, text in sources():
        for fn in launchers:
            alone = re.findall(r"[;{})]\s*%s\(" % fn, text)
            assert not alone, (name, fn)
