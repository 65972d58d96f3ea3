"""Which form of the GEMM and attention kernels a bound shape takes: the ends of the dispatch rules, on the CPU."""
import pytest

from paper_2403_00176_b200 import binding as B
from paper_2403_00176_b200 import workloads as WL


def _gemm(K, N, M):
    g = B.Graph(f"sym M 1 40000\ninput x bf16 [1,M,{K}]\nconst W bf16 [{K},{N}]\nnode MatMul x W -> y\noutput y\n", 0)
    return g.bind_dims(["M"], [[M]]).plan().group_form(0)


@pytest.mark.parametrize("K,N,M,form", [
    # K split over clusters: 8 CTAs up to 15 tiles, 4 up to 33, 2 up to 74, from 24 (4 CTAs: 12) chunks of 64 on
    (3072, 768, 1, "cluster 8"), (3072, 768, 128, "cluster 8"), (3072, 768, 129, "cluster 4"), (3072, 768, 257, "cluster 2"), (3072, 768, 769, "tile 64"),
    (1536, 384, 256, "cluster 8"), (1472, 384, 256, "cluster 4"), (704, 768, 64, "tile 64"), (768, 768, 64, "cluster 4"), (768, 2304, 64, "cluster 2"),
    (768, 2304, 65, "tile 64"), (768, 768, 257, "tile 64"),
    # one wave of 64-column tiles, then 128 or 256 columns by waves
    (768, 768, 1536, "tile 64"), (768, 768, 1537, "tile 128"), (768, 3072, 769, "tile 256"),
    # pairs where their estimate is 2 us below the single CTA's; never below 12 chunks
    (768, 3072, 1806, "pair"), (768, 3072, 2305, "tile 256"), (768, 2304, 2049, "pair"), (3072, 768, 3073, "pair"), (3072, 768, 14072, "pair"),
    (384, 1536, 8228, "tile 256"), (704, 3072, 1806, "tile 256")])
def test_gemm_forms(K, N, M, form):
    assert _gemm(K, N, M) == form


def test_attention_forms():
    g = B.Graph(WL.cfg2(layers=1).ir, 0)
    at = [g.group_info(i)["kind"] for i in range(g.num_groups())].index("attention")
    form = lambda lens, graph=g: graph.bind_dims(["L"], [[n] for n in lens]).plan().group_form(at)
    assert form([2]) == form([512, 16, 127]) == form([1]) == "tcgen05"
    assert form([1, 64]) == "mma.sync"                     # the views of a single token have other strides
    assert form([64] * 64 + [1, 2]) == "mixed"             # a table of 64 requests and one of two
    assert form([64], B.Graph(WL.cfg2(layers=1).ir, B.OPT_LEGACY_ATTENTION)) == "mma.sync"


@pytest.mark.parametrize("K,N,M,tail,form", [
    # GELU: a launch's time, main loop or epilogue, whichever bounds a wave; pairs only where they are within an eighth
    (768, 3072, 1000, "gelu", "tile 128"), (768, 3072, 1806, "gelu", "tile 128"), (768, 3072, 2900, "gelu", "tile 256"), (768, 3072, 12700, "gelu", "pair"),
    (384, 1536, 3600, "gelu", "tile 128"), (384, 1536, 6000, "gelu", "tile 256"),
    # a residual and fewer than 24 chunks; 24 and more by the main loop
    (768, 768, 3600, "residual", "tile 128"), (1472, 768, 2400, "residual", "tile 128"), (1536, 768, 2400, "residual", "tile 128"), (1472, 1920, 3650, "residual", "tile 128"), (1536, 1920, 3650, "residual", "tile 256"),
    (768, 768, 7169, "residual", "pair"),
    # up to 8 chunks whatever the tail
    (512, 1152, 4500, "", "tile 128"), (576, 1152, 4500, "", "tile 256")])
def test_gemm_forms_by_epilogue(K, N, M, tail, form):
    ir = f"sym M 1 40000\ninput x bf16 [1,M,{K}]\n" + (f"input r bf16 [1,M,{N}]\n" if tail == "residual" else "") + f"const W bf16 [{K},{N}]\nnode MatMul x W -> y\n"
    ir += {"gelu": "node Gelu y -> z\noutput z\n", "residual": "node Add y r -> z\noutput z\n", "": "output y\n"}[tail]
    assert B.Graph(ir, 0).bind_dims(["M"], [[M]]).plan().group_form(0) == form


@pytest.mark.parametrize("N,H,W,cout,form", [
    # halo patches for up to 4/3 of the implicit GEMM's waves: as many (whatever the tiles), 5 for 4, 4 for 3; not 7 for 5, 3 for 2, 2 for 1
    (32, 56, 56, 128, "halo"), (74, 16, 8, 128, "halo"), (20, 58, 64, 128, "halo"), (18, 64, 48, 128, "halo"), (25, 58, 64, 128, "implicit GEMM"),
    (10, 58, 64, 128, "implicit GEMM"), (6, 64, 48, 128, "implicit GEMM"), (4, 64, 48, 128, "halo"), (4, 64, 48, 256, "halo"), (5, 64, 48, 256, "implicit GEMM"),
    # row tiles from four fifths of 128 pixels on; tiles of 64 columns stay
    (1, 20, 102, 128, "halo"), (1, 20, 103, 128, "rows"), (1, 20, 102, 192, "implicit GEMM")])
def test_convolution_forms(N, H, W, cout, form):
    ir = f"input x bf16 [{N},128,{H},{W}]\nconst w bf16 [{cout},128,3,3]\nnode Conv x w -> y {{kernel=3 stride=1 pad=1}}\noutput y\n"
    g = B.Graph(ir, 0)
    conv = [g.group_info(i)["kind"] for i in range(g.num_groups())].index("conv")
    assert g.bind_dims([], [[]]).plan().group_form(conv) == form


def test_projection_blocks_copy_no_samples():
    # the executed and the skipped branch of a projection block are convolutions: both read the Switch input and write the Combine
    # output through the id lists, so the groups around them launch nothing; with copies asked for, they do
    wl = WL.cfg5()
    launches = []
    for flags in (0, B.OPT_COPY_REGROUP):
        g = B.Graph(wl.ir, flags)
        p = g.bind_dims([], [[]]).plan()
        kinds = [g.group_info(i)["kind"] for i in range(g.num_groups())]
        launches.append(sum(p.group_cost(i)[1] for i, k in enumerate(kinds) if k == "combine"))
    assert launches[0] == 0 and launches[1] > 0
