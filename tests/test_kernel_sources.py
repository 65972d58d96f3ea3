"""Properties of the kernel sources that no run can show reliably: checked on the text."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_00176_b200", "csrc")


def _sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, f)) as h:
                yield f, re.sub(r"//[^\n]*", "", h.read())


def test_kernels_branch_on_barrier_tests_only_through_a_vote():
    # mbar_test_wait answers per lane, and the lanes of a warp may see a phase end at different tests: a kernel that branches
    # on it around a warp-wide wait or tcgen05.ld could leave lanes behind.  Outside ptx.cuh only the voted form is used
    users = [f for f, text in _sources() if f != "ptx.cuh" and re.search(r"\bmbar_test_wait\s*\(", text)]
    assert users == []
    ptx = dict(_sources())["ptx.cuh"]
    assert re.search(r"bool mbar_test_wait_warp\([^)]*\) \{\s*return __all_sync\(0xffffffffu, mbar_test_wait\(", ptx)


def test_strip_convolution_orders_rows_by_completion():
    # consecutive input rows accumulate into overlapping blocks with instructions of different shapes, which have no documented
    # order of their own: a row is issued on the commit of the row before, and no instruction overwrites its accumulator
    text = dict(_sources())["conv3x3_strip_tcgen05.cuh"]
    assert "mma_commit(&turn[me ^ 1])" in text and not re.search(r"mbar_arrive\w*\(&turn", text)
    assert re.search(r"tcgen05\.mma\.[^;]*%3, 1;", text) and len(re.findall(r"tcgen05\.mma\.", text)) == 1


def test_warps_are_together_before_a_ring_goes_on():
    # a role whose leading lane issues behind predicates has nothing but its waits to keep the other lanes from falling behind, and a
    # lane two phases behind waits for a parity that looks like one it has seen.  Behind a wait that lanes leave one by one, the
    # warp is brought together before the commit, arrival or load that lets the barrier's next phase end
    sources = dict(_sources())
    assert set(re.findall(r"\bvoid (mbar_wait\w*)\(", sources["ptx.cuh"])) == {"mbar_wait_lanes", "mbar_wait_warp"}
    assert re.search(r"void mbar_wait_warp\([^)]*\) \{\s*mbar_wait_lanes\(bar, parity, dead\);\s*__syncwarp\(\);\s*\}", sources["ptx.cuh"])
    events = r"\b(mbar_wait_lanes|mbar_wait_warp|__syncwarp|elect_one|elect_leader|mma_commit(?:_pair)?|mbar_arrive\w*|mbar_expect_tx|tma_load_\w+|bulk_commit|continue|void)\b[ (]"
    users = 0
    for name, text in sources.items():
        if name == "ptx.cuh":
            continue
        apart = None
        for m in re.finditer(events, text):
            what, line = m.group(1), text[:m.start()].count("\n") + 1
            if what == "mbar_wait_lanes":
                apart, users = line, users + 1
            elif what in ("mbar_wait_warp", "__syncwarp", "elect_one", "elect_leader", "void"):
                apart = None
            else:
                assert apart is None, (name, apart, line, what)
        assert apart is None, (name, apart)
    assert users >= 15
    # waits of single threads: only in kernels that have roles under one lane
    assert {f for f, text in sources.items() if re.search(r"\bmbar_wait(_limited)?\(", text)} == {
        "ptx.cuh", "gemm_chain_tcgen05.cuh", "conv_stem_tcgen05.cuh", "selftest_mma.cu", "noalloc.cu"}


def test_a_run_starts_behind_everything_before_it():
    # kernels read constants and packed weights ahead of their dependency wait and let their successors start early; what a caller did on
    # the stream before the run (update a constant, prepack) is ordered by the run's first launch: nothing starts before that has waited
    sources = dict(_sources())
    text = sources["exec.cu"]
    assert re.search(r"void __launch_bounds__\(128\) clear_header\([^)]*\) \{\s*ptx::pdl_wait\(\);\s*ptx::pdl_launch\(\);", text)
    body = re.search(r"\nStatus run_plan\(.*?\n\}", text, re.S).group(0)
    first = body.index("L->fn(xs)")
    assert body.index("if (p->uses_header && step_lo <= 0)") < body.index("launch_pdl(clear_header") < first and body.index("cudaMemsetAsync(arena") < first
    # kernels of plans without a header read nothing ahead: those that are programmatic dependents wait before their first load
    for name, kernel in (("kernels_rows.cuh", "chain_elementwise"), ("kernels_compact.cuh", "nonzero_mask"), ("kernels_compact.cuh", "nonzero_write")):
        body = re.search(r"\b%s\(.*?ptx::pdl_wait\(\);" % kernel, sources[name], re.S).group(0)
        assert not re.search(r"->|= ?\*|reinterpret_cast", body), (kernel, body)


def test_row_convolution_hands_tiles_over_between_its_issuers():
    # two warps issue alternate tiles out of one ring.  A warp that does not issue a tile must not wait on its stages: the other's
    # commits let the ring go on whether or not it has looked.  It waits for its turn, which passes behind the tile's last stage
    text = dict(_sources())["conv3x3_tcgen05.cuh"]
    role = text[text.index("warp == 3 || warp == 12"):text.index("warp == 2", text.index("warp == 3 || warp == 12"))]
    assert re.search(r"if \(acc != me\) \{ n \+= kstages; continue; \}\s*if \(j >= 1\) ptx::mbar_wait_warp\(&turn\[me\]", role)
    assert re.search(r"mbar_wait_lanes\(&full\[s\][^;]*;\s*if \(ks \+ 1 == kstages\) \{\s*__syncwarp\(\);\s*if \(lane == 0\) ptx::mbar_arrive\(&turn\[me \^ 1\]\);", role)
    assert role.count("mbar_wait_lanes(&full") == 1 and "mbar_wait_warp(&full" not in role
