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


# const __restrict__ parameters of kernels that wait for the kernel in front of them: data that are complete before they start
COMPLETE_BEFORE = {
    "w_router": None, "bias": None, "w": None, "maps": None, "bank": None,                 # never written by a kernel of a serving loop
    # written by the router, and read by kernels in front of these, which let them start only behind their own wait
    "topk_w": {"decode_gemm_kernel", "token_down_kernel", "token_down_bulk_kernel", "prefill_gemm_kernel", "tc_stream_kernel",
               "epilogue_prefetch"},
    "ids": {"combine_kernel"},
}


def test_nothing_read_behind_a_launch_dependency_counts_as_read_only():
    """A load through const __restrict__ may move in front of griddepcontrol.wait, where its data are still being written: only
    parameters that are complete before the kernel starts have it, and so with the device functions that such kernels call."""
    seen = set()
    for name, text in sources():
        if not re.search(r"grid_dependency_wait\(\)|griddepcontrol\.wait", text):
            continue
        text = re.sub(r"__launch_bounds__\([^)]*\)", "", text)
        functions = list(re.finditer(r"(__global__|__device__)[^;{}]*?(\w+)\(([^{};]*)\)\s*\{", text))
        for i, m in enumerate(functions):
            end = functions[i + 1].start() if i + 1 < len(functions) else len(text)
            if m[1] == "__global__" and not re.search(r"grid_dependency_wait\(\)|griddepcontrol\.wait", text[m.end():end]):
                continue                                       # an ordinary launch: everything in front of it is complete
            for param in re.findall(r"const [\w ]+\*\s*__restrict__ (\w+)", m[3]):
                assert param in COMPLETE_BEFORE and m[2] in (COMPLETE_BEFORE[param] or {m[2]}), (name, m[2], param)
            seen.add(m[2])
    assert {"route_kernel", "route_token_kernel", "route_mma_kernel", "group_small_kernel", "plan_gather_kernel", "combine_kernel",
            "stream_gemm_kernel", "tc_stream_kernel", "pair_gateup_wide_kernel", "fetch_misses_kernel"} <= seen


def test_kernels_of_many_ctas_keep_the_next_one_out():
    """A kernel that releases its dependents at its start shares its SMs with their waiting CTAs: the row copy has thousands of
    CTAs, and behind it stands a GEMM whose one CTA per SM takes half of the threads."""
    text = dict(sources())
    for name, kernel in (("prefill.cu", "gather_rows_kernel"), ("plan.cu", "group_chunk_count_kernel"), ("plan.cu", "group_chunk_scatter_kernel")):
        start = text[name].index("\n%s(" % kernel)
        end = text[name].index("\n}\n", start)
        body = text[name][start:end]
        assert "grid_dependency_wait();" in body and "grid_launch_dependents" not in body, kernel


def test_every_programmatic_launch_can_be_switched_off():
    """-DEXMOE_DISABLE_PDL is for timing without programmatic launches: every launcher that asks for one honours it."""
    found = 0
    for name, text in sources():
        for m in re.finditer(r"programmaticStreamSerializationAllowed = 1;", text):
            launch = text[m.end():text.index("cudaLaunchKernelEx(", m.end())]
            assert "#ifdef EXMOE_DISABLE_PDL" in launch, (name, text[:m.start()].count("\n") + 1)
            found += 1
    assert found >= 8
