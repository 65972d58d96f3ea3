"""Kernel edges on the GPU: sizes at the ends of tiles, items and dispatch rules, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import interp as O
from paper_2403_00176_b200 import binding as B
from paper_2403_00176_b200 import workloads as WL
from paper_2403_00176_b200.session import Session
from paper_2403_00176_b200.workloads import Request, bf16_round
from tests.gpu_harness import lockstep, run_batch
from tests.test_gpu_parity import _check_topk_lockstep

pytestmark = pytest.mark.gpu

F32_TOL, BF16_TOL = 1e-5, 2e-2


@pytest.mark.parametrize("dtype,tol", [("f32", F32_TOL), ("bf16", BF16_TOL)])
def test_chain_vectors_that_straddle_rows_and_tails(dtype, tol):
    # vectors of 8 outputs over the flat index: rows shorter than a vector, rows that end inside one, tiles of 8192 (4096 in fp32) +- 2,
    # tiles inside one row, operands broadcast over the middle, the first and the last dim, ten requests (two tables), rank 4
    ir = (f"sym I 1 4096\nsym J 1 4096\nsym K 1 8192\ninput a {dtype} [I,1,K]\ninput b {dtype} [2,I,J,K]\ninput c {dtype} [J,1]\n"
          "fconst h f32 [] = 0.5\nnode Sigmoid c -> s\nnode Mul s h -> t\nnode Add t a -> u\nnode Add b u -> v\nnode Relu v -> y\noutput y\n")
    rng = np.random.default_rng(21)
    rnd = (lambda a: bf16_round(a.astype(np.float32))) if dtype == "bf16" else (lambda a: a.astype(np.float32))
    sizes = [(1, 1, 1), (3, 5, 7), (2, 3, 8), (1, 1, 4095), (1, 1, 4096), (1, 1, 4097), (2, 3, 8192), (2, 9, 15), (5, 4, 16), (3, 2, 333)]
    reqs = [Request({"I": i, "J": j, "K": k}, {"a": rnd(rng.standard_normal((i, 1, k))), "b": rnd(rng.standard_normal((2, i, j, k))),
                                               "c": rnd(rng.standard_normal((j, 1)))}) for i, j, k in sizes]
    wl = WL.Workload("chain_edges", dtype, ir, {}, ["I", "J", "K"], ["y"], {"batch_fn": lambda j: reqs})
    _, _, outs = run_batch(wl, reqs)
    for r, req in enumerate(reqs):
        ref = O.run(ir, {}, req.inputs)["y"]
        assert outs[r]["y"].shape == ref.shape
        assert O.rel_err(outs[r]["y"], ref) <= tol, req.syms


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("rank", [1, 2, 3, 4])
def test_nonzero_chunks_words_and_ranks(dtype, rank):
    # pieces of 8192 elements +- 1 (32-element words, 16-byte vectors), a request of several chunks, ten requests (two
    # tables), an all-zero one, negative zeros, ranks 1 to 4; the coordinates are whole numbers: exact
    names = ["A", "B", "C", "D"][:rank]
    ir = "".join(f"sym {n} 0 100000\n" for n in names) + f"input x {dtype} [{','.join(names)}]\nnode NonZero x -> nz\noutput nz\n"
    rng = np.random.default_rng(31)
    sizes = [1, 31, 33, 8191, 8192, 8193, 16400, 40001, 7, 640]
    reqs = []
    for i, n in enumerate(sizes):
        shape = {1: (n,), 2: (max(n // 7, 1), 7), 3: (max(n // 15, 1), 5, 3), 4: (max(n // 40, 1), 2, 5, 4)}[rank]
        x = bf16_round(rng.standard_normal(shape).astype(np.float32))
        x[rng.uniform(size=shape) < (1.0 if i == 8 else 0.5)] = -0.0
        reqs.append(Request(dict(zip(names, shape)), {"x": x}))
    wl = WL.Workload("nonzero_edges", dtype, ir, {}, names, ["nz"], {"batch_fn": lambda j: reqs})
    _, p, outs = run_batch(wl, reqs)
    for r, req in enumerate(reqs):
        assert np.array_equal(outs[r]["nz"], np.array(np.nonzero(req.inputs["x"]))), req.syms
    # the counts are read once per run: another run on other data must be read again
    p.in_dev[0].zero_()
    p.run()
    assert all(o["nz"].shape == (rank, 0) for o in p.outputs())
    p.in_dev[0].copy_(torch.from_numpy(p.in_host[0]))
    p.run_graph()
    again = p.outputs()
    assert all(np.array_equal(a["nz"], b["nz"]) for a, b in zip(again, outs))


@pytest.mark.parametrize("shapes", [[(1, 64)], [(2, 127), (3, 128)], [(9, 129)], [(70, 65), (1, 300), (5, 257), (3, 3), (40, 192)], [(300, 66)]])
def test_conv_strips_segments_and_ring(shapes):
    # strips of the 64 -> 64 channel kernel: one row, segments shorter and longer than the accumulator ring (8 rows) and
    # the row ring, column tiles with one pixel, several requests in one launch beside one below its width rule
    wl = WL.cfg4(blocks=2)
    rng = np.random.default_rng(41)
    reqs = [Request({"H": h, "W": w}, {"x": bf16_round(rng.uniform(-1, 1, (1, 64, h, w)).astype(np.float32))}) for h, w in shapes]
    s, p, outs = run_batch(wl, reqs, opt_flags=B.OPT_NO_REUSE)
    for r, req in enumerate(reqs):
        errs = lockstep(wl, s, p, outs, r, BF16_TOL)
        assert max(errs.values()) <= BF16_TOL, (req.syms, errs)
    p.run()
    for a, b in zip(outs, p.outputs()):
        assert all(np.array_equal(a[n], b[n]) for n in a)


@pytest.mark.parametrize("C,shapes", [(128, [(14, 14), (28, 28), (56, 56), (5, 29), (31, 30), (1, 1)]), (256, [(7, 7), (17, 43), (33, 64)]), (384, [(2, 15)]),
                                      (384, [(130, 98)]), (128, [(2400, 14)])])
def test_conv_halo_patches(C, shapes):
    # patches that fill their 128 rows and that do not, images smaller than a patch and a pixel larger, lines of a whole tile, two and
    # three channel tiles; and launches in which CTAs take three tiles (accumulators, bias and residual buffers, and the ring from
    # tile to tile)
    wl = WL.cfg4(blocks=2, C=C)
    rng = np.random.default_rng(61)
    reqs = [Request({"H": h, "W": w}, {"x": bf16_round(rng.uniform(-1, 1, (1, C, h, w)).astype(np.float32))}) for h, w in shapes]
    s, p, outs = run_batch(wl, reqs, opt_flags=B.OPT_NO_REUSE)
    forms = {p.plan.group_form(i) for i in range(s.graph.num_groups()) if s.graph.group_info(i)["kind"] == "conv"}
    assert forms == {"halo"}, forms
    if shapes[0][0] > 100:
        (h, w), = shapes
        patches = min(-(-w // tw) * -(-h // min(128 // (tw + 2), h)) for tw in range(1, min(w, 126) + 1))
        assert patches * (C // 128) > 2 * torch.cuda.get_device_properties(0).multi_processor_count
    for r, req in enumerate(reqs):
        errs = lockstep(wl, s, p, outs, r, BF16_TOL)
        assert max(errs.values()) <= BF16_TOL, (req.syms, errs)
    p.run()
    for a, b in zip(outs, p.outputs()):
        assert all(np.array_equal(a[n], b[n]) for n in a)


@pytest.mark.parametrize("C,H,W", [(128, 310, 110), (192, 450, 128), (128, 5, 103)])
def test_conv_row_tiles_handed_over_between_issuers(C, H, W):
    # row tiles of 128 and 64 channels: three and ten tiles for some CTAs (both issuers in turn, accumulators and ring reused), one for
    # others, with a residual
    wl = WL.cfg4(blocks=1, C=C)
    rng = np.random.default_rng(73)
    req = Request({"H": H, "W": W}, {"x": bf16_round(rng.uniform(-1, 1, (1, C, H, W)).astype(np.float32))})
    s, p, outs = run_batch(wl, [req], opt_flags=B.OPT_NO_REUSE)
    assert {p.plan.group_form(i) for i in range(s.graph.num_groups()) if s.graph.group_info(i)["kind"] == "conv"} == {"rows"}
    errs = lockstep(wl, s, p, outs, 0, BF16_TOL)
    assert max(errs.values()) <= BF16_TOL, errs


@pytest.mark.parametrize("cin", [64, 192, 256, 320, 512])
def test_conv_forms_add_up_in_the_same_order(cin):
    # kernel rows, then 64-channel chunks, then columns: halo patches (chunks resident up to 256 channels and streamed beyond), row tiles
    # and the implicit GEMM give the same bits.  The same pixels with zeros behind them, at sizes that take different forms
    ir = (f"sym H 1 4096\nsym W 1 4096\ninput x bf16 [1,{cin},H,W]\nconst w bf16 [128,{cin},3,3]\nconst b bf16 [128]\n"
          "node Conv x w b -> c {kernel=3 stride=1 pad=1}\nnode Relu c -> y\noutput y\n")
    rng = np.random.default_rng(71)
    consts = {"w": bf16_round((rng.standard_normal((128, cin, 3, 3)) / np.sqrt(9 * cin)).astype(np.float32)), "b": bf16_round(rng.standard_normal(128).astype(np.float32))}
    s = Session(WL.Workload("conv_forms", "bf16", ir, consts, ["H", "W"], ["y"], {}))
    conv = [s.graph.group_info(i)["kind"] for i in range(s.graph.num_groups())].index("conv")
    for h, w, sizes in [(37, 90, [(37, 90, "halo"), (37, 128, "rows")]), (384, 48, [(384, 48, "implicit GEMM"), (384, 50, "halo"), (384, 103, "rows")])]:
        pixels = bf16_round(rng.standard_normal((1, cin, h, w)).astype(np.float32))
        outs = []
        for hh, ww, form in sizes:
            x = np.zeros((1, cin, hh, ww), np.float32)
            x[:, :, :h, :w] = pixels
            p = s.prepare([Request({"H": hh, "W": ww}, {"x": x})])
            assert p.plan.group_form(conv) == form
            p.run()
            p.check_device_status()
            outs.append(p.outputs()[0]["y"][:, :, :h, :w])
        assert all(np.array_equal(outs[0], o) for o in outs[1:])
        if h == 37:
            assert O.rel_err(outs[0], O.run(ir, consts, {"x": pixels})["y"]) <= BF16_TOL


@pytest.mark.parametrize("cin,cout,side,kernel,form", [(64, 64, (20, 70), 3, "strip"), (64, 128, (14, 14), 3, "halo"), (128, 128, (20, 110), 3, "rows"),
                                                       (64, 192, (9, 11), 3, "implicit GEMM"), (128, 128, (9, 11), 1, "implicit GEMM")])
def test_skipped_samples_through_a_convolution(cin, cout, side, kernel, form):
    # a block whose skipped samples go through a convolution with a ReLU, in every form that reads and writes through the skipped ids, and an
    # identity block behind it: against the oracle, against whole-sample copies, without reuse, and with the counts read back
    n, (h, w) = 7, side
    lines, consts, rng = [f"input x bf16 [{n},64,{h},{w}]", "fconst zero f32 [] = 0.0"], {}, np.random.default_rng(79)

    def const(name, shape, scale, at=0.0):
        lines.append(f"const {name} bf16 [{','.join(map(str, shape))}]")
        consts[name] = bf16_round((rng.standard_normal(shape) * scale + at).astype(np.float32))

    const("w", (cin, 64, 1, 1), 1 / 8)
    lines += ["node Conv x w -> stem {kernel=1 stride=1 pad=0}"]
    src, c = "stem", cin
    for b in range(2):
        const(f"gw{b}", (c, 1), 1.0)
        const(f"gb{b}", (1,), 0.0)
        const(f"w{b}", (cout, c, 3, 3), (2 / (9 * c)) ** 0.5)
        const(f"v{b}", (cout, cout, 3, 3), (2 / (9 * cout)) ** 0.5)
        lines += [f"iconst s{b} i64 [2] = {n} {c}", f"node GlobalAveragePool {src} -> p{b}", f"node Reshape p{b} s{b} -> r{b}", f"node MatMul r{b} gw{b} -> m{b}",
                  f"node Add m{b} gb{b} -> z{b}", f"node Greater z{b} zero -> gate{b}", f"node Switch {src} gate{b} -> e{b} k{b}",
                  f"node Conv e{b} w{b} -> c{b} {{kernel=3 stride=1 pad=1}}", f"node Relu c{b} -> d{b}", f"node Conv d{b} v{b} -> f{b} {{kernel=3 stride=1 pad=1}}",
                  f"node Relu f{b} -> y{b}"]
        skipped = f"k{b}"
        if b == 0:
            const("u", (cout, c, kernel, kernel), (2 / (kernel * kernel * c)) ** 0.5)
            const("ub", (cout,), 0.1)
            lines += [f"node Conv k0 u ub -> q {{kernel={kernel} stride=1 pad={kernel // 2}}}", "node Relu q -> t"]
            skipped = "t"
        lines.append(f"node Combine y{b} {skipped} gate{b} -> blk{b}")
        src, c = f"blk{b}", cout
    ir = "\n".join(lines + [f"node GlobalAveragePool {src} -> gap", "output gap", "output gate0", "output gate1"]) + "\n"
    ir = "\n".join(sorted(ir.splitlines(), key=lambda l: {"node": 1, "output": 2}.get(l.split()[0], 0))) + "\n"
    x = rng.standard_normal((n, 64, h, w)) + rng.standard_normal((n, 64, 1, 1))
    wl = WL.Workload("skipped_convolution", "bf16", ir, consts, [], ["gap", "gate0", "gate1"], {})
    # the gates of both blocks near the middle of their samples' logits, by the oracle
    req = Request({}, {"x": bf16_round(x.astype(np.float32))})
    for b in range(2):
        z = np.sort(O.run(ir, consts, req.inputs)[f"z{b}"].reshape(-1))
        consts[f"gb{b}"] = bf16_round(np.array([-(z[3] + z[4]) / 2], np.float32))
    runs = {}
    for flags in (B.OPT_NO_REUSE, 0, B.OPT_COPY_REGROUP):
        s, p, outs = run_batch(wl, [req], opt_flags=flags)
        runs[flags] = outs[0]
        if flags == B.OPT_NO_REUSE:
            errs = lockstep(wl, s, p, outs, 0, BF16_TOL)
            assert {"blk0", "blk1"} <= set(errs) and max(v for v in errs.values()) <= BF16_TOL, errs
        if not flags & B.OPT_COPY_REGROUP:
            forms = {p.plan.group_form(i) for i in range(s.graph.num_groups()) if s.graph.group_info(i)["kind"] == "conv"}
            assert forms - {"implicit GEMM"} == ({form} if kernel == 3 else {"halo"}) - {"implicit GEMM"}     # (the first is 1x1)
            p.run_exact()
            assert all(np.array_equal(a, runs[flags][name]) for name, a in p.outputs()[0].items())
    assert all(0 < runs[0][f"gate{b}"].sum() < n for b in range(2))
    for flags in (0, B.OPT_COPY_REGROUP):
        assert all(np.array_equal(runs[flags][name], runs[B.OPT_NO_REUSE][name]) for name in runs[0]), flags


@pytest.mark.parametrize("lens", [[1], [33, 64], [129, 640], list(range(1, 129, 3)) + [129, 191, 192, 193, 255, 256, 257, 300, 383, 385, 511, 512, 513, 577] + [200] * 8,
                                  list(range(2, 130, 3)) + [128, 129, 191, 192, 193, 255, 256, 257, 300, 383, 385, 511, 512, 513, 577] + [200] * 7])
def test_attention_blocks_items_and_tables(lens):
    # blocks of 64 keys and tiles of 128 rows at their edges, warps without a live row, a CTA's first, second and third
    # item (the last list: 65 requests, two tables, more than two items per CTA in the first; the list before it has a request of
    # one token among others, whose table goes to the mma.sync kernel)
    wl = WL.cfg2(layers=1, D=384, H=6, F=384, n_requests=1, lmin=1, lmax=640)
    rng = np.random.default_rng(43)
    reqs = [Request({"L": n}, {"x": bf16_round(rng.standard_normal((1, n, 384)).astype(np.float32))}) for n in lens]
    s, p, outs = run_batch(wl, reqs, opt_flags=B.OPT_NO_REUSE)
    form = [p.plan.group_form(i) for i in range(s.graph.num_groups()) if s.graph.group_info(i)["kind"] == "attention"]
    assert form == ["mixed" if 1 in lens and len(lens) == 65 else "tcgen05"], form
    for r in range(0, len(reqs), 4 if len(reqs) > 8 else 1):
        errs = lockstep(wl, s, p, outs, r, BF16_TOL)
        bad = {k: v for k, v in errs.items() if not (isinstance(v, float) and v <= BF16_TOL)}
        assert errs and not bad, (reqs[r].syms, bad)
    p.run()
    for a, b in zip(outs, p.outputs()):
        assert np.array_equal(a["y"], b["y"])


def test_issue_behind_predicates_keeps_up_with_the_pipe():
    # cycles per MMA where a warp waits, its leading lane issues a stage behind predicates and commits it, in stages of 4, 8 and 12: the
    # tensor pipe's 64 at 128 columns and 128 at 256 within a tenth; at 64 columns 43 to 69, where the pipe's 48 do not hide all of the
    # issuer's work.  One thread's handshake takes 95 to 162.  Printed with -s
    st = torch.cuda.current_stream().cuda_stream
    rate = {(pair, n, k): [B.sod2_selftest_mma_rate(pair, n, k, hs, st, iters=4032 if k == 12 else 4096) for hs in (2, 3)]
            for pair in (False, True) for n in (64, 128, 256) for k in (4, 8, 12)}
    print({key: [round(v, 1) for v in r] for key, r in rate.items()})
    for (pair, n, k), (thread, warp) in rate.items():
        assert warp <= {64: 74.0, 128: 72.0, 256: 133.0}[n] and warp < thread + 1.0


@pytest.mark.parametrize("D,H", [(64, 1), (256, 4), (320, 5), (512, 8), (576, 9)])
def test_topk_keep_with_the_layernorm_behind_it(D, H):
    # the kept rows of the first layer leave normalised for the second, in the launch that selects them: rows of one and two
    # vectors a lane, whole and ragged, and rows too wide for that (576); chunks of 32 tokens at their edges, a request of one
    # token, one of more tokens than a CTA has threads
    lens = [1, 2, 31, 32, 33, 64, 65, 300]
    wl = WL.cfg3(layers=2, D=D, H=H, F=2 * D)
    rng = np.random.default_rng(67)
    name, sym = wl.ir.split("input ")[1].split()[0], wl.sym_names[0]
    reqs = [Request({sym: n}, {name: bf16_round((rng.standard_normal((1, n, D)) * rng.uniform(0.5, 2.0, (1, n, 1)) + rng.standard_normal((1, n, 1))).astype(np.float32))}) for n in lens]
    s, p, outs = _check_topk_lockstep(wl, reqs, 2)
    kinds = [s.graph.group_info(i)["kind"] for i in range(s.graph.num_groups())]
    assert p.plan.group_form(kinds.index("topk_keep") + 1) == ("in the selection" if D <= 512 else "")
    # with the arena's space reused, which the launch's reads and writes must allow
    _, _, reused = run_batch(wl, reqs)
    for a, b in zip(outs, reused):
        assert all(np.array_equal(a[n], b[n]) for n in a)


@pytest.mark.parametrize("K,N,M,act,residual", [(768, 768, 7169, None, True), (768, 2312, 4224, "Gelu", False), (3072, 768, 4100, "Relu", True), (3072, 776, 11009, None, False), (768, 392, 12700, None, True)])
def test_gemm_pairs_by_rule(K, N, M, act, residual):
    # sizes at which the dispatch takes CTA pairs by itself: tiles of 192 and 256 columns, a ragged last column unit, the last
    # wave's tiles cut in two, row tiles in bands, an odd number of 128-row tiles
    ir = f"sym M 1 20000\ninput x bf16 [1,M,{K}]\n" + (f"input r bf16 [1,M,{N}]\n" if residual else "") + f"const W bf16 [{K},{N}]\nconst b bf16 [{N}]\nnode MatMul x W -> t0\nnode Add t0 b -> t1\n"
    ir += (f"node {act} t1 -> t2\n" if act else "") + (f"node Add {'t2' if act else 't1'} r -> y\n" if residual else "")
    y = "y" if residual else "t2" if act else "t1"
    ir += f"output {y}\n"
    rng = np.random.default_rng(47)
    consts = {"W": bf16_round((rng.standard_normal((K, N)) / np.sqrt(K)).astype(np.float32)), "b": bf16_round(rng.standard_normal(N).astype(np.float32))}
    ins = {"x": bf16_round(rng.standard_normal((1, M, K), dtype=np.float32))}
    if residual:
        ins["r"] = bf16_round(rng.standard_normal((1, M, N), dtype=np.float32))
    reqs = [Request({"M": M}, ins)]
    wl = WL.Workload("gemm_pair_rule", "bf16", ir, consts, ["M"], [y], {"batch_fn": lambda j: reqs})
    _, p, outs = run_batch(wl, reqs)
    assert p.plan.group_form(0) == "pair"
    assert O.rel_err(outs[0][y], O.run(ir, consts, ins)[y]) <= BF16_TOL
    p.run()
    assert np.array_equal(outs[0][y], p.outputs()[0][y])


@pytest.mark.parametrize("K,N,Ms", [(3072, 768, [1, 64, 97, 128]), (1536, 392, [129, 256, 300]), (1600, 776, [513, 640]), (768, 1000, [63, 64, 65]), (832, 2304, [33])])
@pytest.mark.parametrize("act,residual", [("Gelu", False), (None, True)])
def test_gemm_k_split_over_clusters(K, N, Ms, act, residual):
    # clusters of 8, 4 and 2 CTAs: shares of rows with none left for the last ranks, a ragged last column tile, chunk counts the
    # cluster does not divide (25, 13), the ReLU behind the residual, two row tiles with one row in the last
    ir = f"sym M 1 1000\ninput x bf16 [1,M,{K}]\n" + (f"input r bf16 [1,M,{N}]\n" if residual else "") + f"const W bf16 [{K},{N}]\nconst b bf16 [{N}]\nnode MatMul x W -> t0\nnode Add t0 b -> t1\n"
    ir += (f"node {act} t1 -> y\n" if act else "node Add t1 r -> t2\nnode Relu t2 -> y\n") + "output y\n"
    rng = np.random.default_rng(53)
    consts = {"W": bf16_round((rng.standard_normal((K, N)) / np.sqrt(K)).astype(np.float32)), "b": bf16_round(rng.standard_normal(N).astype(np.float32))}
    wl = WL.Workload("gemm_cluster", "bf16", ir, consts, ["M"], ["y"], {"batch_fn": lambda j: []})
    for M in Ms:
        ins = {"x": bf16_round(rng.standard_normal((1, M, K)).astype(np.float32))}
        if residual:
            ins["r"] = bf16_round(rng.standard_normal((1, M, N)).astype(np.float32))
        _, p, outs = run_batch(wl, [Request({"M": M}, ins)])
        assert p.plan.group_form(0) == f"cluster {8 if K == 3072 or (K == 1536 and M <= 256) else 4 if K in (768, 1536) else 2}", M
        assert O.rel_err(outs[0]["y"], O.run(ir, consts, ins)["y"]) <= BF16_TOL, M
        p.run()
        assert np.array_equal(outs[0]["y"], p.outputs()[0]["y"])


@pytest.mark.parametrize("n,k,D", [(1, 1, 64), (31, 7, 64), (32, 32, 64), (33, 32, 768), (300, 211, 768), (1025, 40, 64), (7000, 4900, 64)])
def test_topk_selection_digits_ties_and_chunks(n, k, D):
    # the radix selection: all scores equal, two values, scores that differ only in their low bits, over the whole exponent
    # range, distinct ones; chunks of 32 tokens at their edges, everything kept, more shared memory than the default, rows
    # wider than the prefetch.  Sums of few squares of powers of two are exact in fp64 whatever their order
    ir = (f"sym N 1 8000\ninput y bf16 [1,N,{D}]\niconst k i64 [1] = {k}\niconst i_m1 i64 [1] = -1\n"
          "node ReduceSumSquare y -> sc {axis=-1 keepdims=0}\nnode TopK sc k -> tv idx {axis=-1 largest=1 order=index}\n"
          "node Reshape idx i_m1 -> ix\nnode Gather y ix -> keep {axis=1}\noutput keep\noutput idx\n")
    rng = np.random.default_rng(59)
    ys = []
    for kind in range(5):
        y = np.zeros((1, n, D), np.float32)
        y[..., 0] = 1.0
        if kind == 1: y[0, :, 1] = rng.integers(0, 2, n)
        if kind == 2: y[0, :, 1] = 2.0 ** -rng.integers(18, 25, n)
        if kind == 3: y[0, :, 0] = 2.0 ** rng.integers(-60, 60, n)
        if kind == 4: y = bf16_round(rng.standard_normal((1, n, D)).astype(np.float32))
        ys.append(y)
    reqs = [Request({"N": n}, {"y": y}) for y in ys]
    wl = WL.Workload("topk_edges", "bf16", ir, {}, ["N"], ["keep", "idx"], {"batch_fn": lambda j: reqs})
    _, p, outs = run_batch(wl, reqs)
    for r, y in enumerate(ys):
        sc = (y[0].astype(np.float64) ** 2).sum(-1)
        want = np.sort(np.argsort(-sc, kind="stable")[:k])
        assert np.array_equal(outs[r]["idx"][0], want), (r, n, k)
        assert np.array_equal(outs[r]["keep"][0], y[0][want]), (r, n, k)


@pytest.mark.parametrize("C", [64, 192])
def test_layout_changes_of_rows_that_start_anywhere(C):
    # channels-last and back around an identity 1x1 convolution: image sizes of every remainder modulo 8, below and past a
    # 64-pixel tile, mixed with aligned ones in one launch; exact
    ir = f"sym H 1 64\nsym W 1 64\ninput x bf16 [1,{C},H,W]\nconst w bf16 [{C},{C},1,1]\nnode Conv x w -> y {{kernel=1 stride=1 pad=0}}\noutput y\n"
    rng = np.random.default_rng(67)
    shapes = [(1, 3), (5, 5), (7, 9), (1, 62), (13, 5), (11, 6), (3, 23), (9, 15), (8, 16), (31, 33), (1, 1)]
    reqs = [Request({"H": h, "W": w}, {"x": bf16_round(rng.standard_normal((1, C, h, w)).astype(np.float32))}) for h, w in shapes]
    wl = WL.Workload("layout_any", "bf16", ir, {"w": np.eye(C, dtype=np.float32).reshape(C, C, 1, 1)}, ["H", "W"], ["y"], {"batch_fn": lambda j: reqs})
    _, p, outs = run_batch(wl, reqs)
    for r, req in enumerate(reqs):
        assert np.array_equal(outs[r]["y"], req.inputs["x"]), req.syms


def test_gelu_epilogue_in_the_negative_tail():
    # pre-activations between -4.25 and -3, where GELU is small enough for bf16 to show the fit: per bin, rms error within what
    # bf16 rounding gives (ulp / sqrt 12) and 2.2e-5: the fit's own error is at most 2.0e-5 there, the hardware tanh adds little
    from math import erf
    M = 2048
    ir = "sym M 1 4096\ninput x bf16 [1,M,64]\nconst W bf16 [64,64]\nnode MatMul x W -> t\nnode Gelu t -> y\noutput y\n"
    W = np.zeros((64, 64), np.float32)
    W[0], W[1] = 1.0, np.arange(64) * 2.0 ** -12
    x = np.zeros((1, M, 64), np.float32)
    x[0, :, 0], x[0, :, 1] = bf16_round(np.linspace(-4.25, -3.0, M).astype(np.float32)), 1.0
    wl = WL.Workload("gelu_tail", "bf16", ir, {"W": bf16_round(W)}, ["M"], ["y"], {"batch_fn": lambda j: []})
    _, _, outs = run_batch(wl, [Request({"M": M}, {"x": x})])
    pre = x[0, :, :1].astype(np.float64) + bf16_round(W)[1]
    want = np.array([0.5 * v * (1 + erf(v / np.sqrt(2))) for v in pre.ravel()])
    err = outs[0]["y"][0].astype(np.float64).ravel() - want
    ulp = 2.0 ** (np.floor(np.log2(np.abs(want))) - 7)
    for lo in np.arange(-4.25, -3.0, 0.25):
        m = (pre.ravel() >= lo) & (pre.ravel() < lo + 0.25)
        rms, rounding = np.sqrt((err[m] ** 2).mean()), np.sqrt((ulp[m] ** 2 / 12).mean())
        assert rms <= np.hypot(rounding, 2.2e-5), (lo, rms, rounding)


def _attention_alone(D, H):
    """softmax(Q K^T / 8) V out of a packed [L, 3 D] input, behind it a product with the identity (exact in bf16)."""
    ir = WL._IR()
    ir.add("sym L 1 1024")
    ir.add(f"input x bf16 [1,L,{3 * D}]")
    WL._attn_iconsts(ir, D, H)
    ir.add(f"const I bf16 [{D},{D}]")
    xs = ir.node("Shape", ["x"], ir.tmp())
    bl = ir.node("Gather", [xs, "i_01"], ir.tmp(), axis=0)
    s4, s3 = (ir.node("Concat", [bl, c], ir.tmp(), axis=0) for c in ("i_heads", "i_D"))
    qkv = []
    for i, perm in enumerate(("0,2,1,3", "0,2,3,1", "0,2,1,3")):
        sl = ir.node("Slice", ["x", f"i_st{i}", f"i_en{i}", "i_ax2"], ir.tmp())
        qkv.append(ir.node("Transpose", [ir.node("Reshape", [sl, s4], ir.tmp())], ir.tmp(), perm=perm))
    s1 = ir.node("Mul", [ir.node("MatMul", qkv[:2], ir.tmp()), "f_scale"], ir.tmp())
    o = ir.node("MatMul", [ir.node("Softmax", [s1], ir.tmp(), axis=-1), qkv[2]], ir.tmp())
    y0 = ir.node("Reshape", [ir.node("Transpose", [o], ir.tmp(), perm="0,2,1,3"), s3], ir.tmp())
    ir.node("MatMul", [y0, "I"], "y")
    ir.add("output y")
    return WL.Workload("attention_alone", "bf16", ir.text(), {"I": np.eye(D, dtype=np.float32)}, ["L"], ["y"], {"batch_fn": lambda j: []})


def _softmax64(x, H):
    L = x.shape[1]
    q, k, v = x.astype(np.float64).reshape(L, 3, H, 64).transpose(1, 2, 0, 3)
    s = q @ k.transpose(0, 2, 1) / 8
    p = np.exp(s - s.max(-1, keepdims=True))
    return ((p / p.sum(-1, keepdims=True)) @ v).transpose(1, 0, 2).reshape(L, H * 64)


@pytest.mark.parametrize("L,top,base", [(128, 100, 10), (65, 64, 0), (300, 127, 63), (400, 384, 200), (300, 200, 130)])
def test_attention_rows_dominated_by_one_key(L, top, base):
    # every row has one heavy key, the next one powers of two below it: where the heavy key is among the first 128 (or moves
    # the reference later on), its weight is exactly 1 and what is left is the output's rounding (1.66e-3 rms over normal values)
    # and that of weights of a fifth or less; a heavy weight that is rounded to bf16 as well makes it 2.2e-3
    H = 6
    wl = _attention_alone(64 * H, H)
    rng = np.random.default_rng(71)
    x = np.zeros((1, L, 3, H, 64), np.float32)
    # past the first 128 keys the gap is more than 2^8, so that the reference moves
    x[0, :, 0, :, 0] = rng.uniform(*((24, 86) if top < 128 else (100, 400)), (L, H))
    x[0, :, 1, :, 0] = -3.0
    x[0, base, 1, :, 0], x[0, top, 1, :, 0] = 0.5, 1.0
    x[0, :, 2] = rng.standard_normal((L, H, 64))
    x = bf16_round(x.reshape(1, L, -1))
    _, _, outs = run_batch(wl, [Request({"L": L}, {"x": x}), Request({"L": L}, {"x": x})])
    want = _softmax64(x, H)
    for o in outs:
        err = o["y"][0].astype(np.float64) - want
        assert np.linalg.norm(err) / np.linalg.norm(want) <= 1.85e-3


def test_exact_staging_with_a_folded_layernorm_across_stages():
    # the GEMM that writes the row statistics of a folded LayerNorm runs in the first stage, the one that reads them (as its
    # residual; its own operand is the gated network's pooled output) in the last: same bits as the bounded run
    wl = WL.cfg5(B=6, side=32, widths=(64,), per_stage=2)
    lines = wl.ir.splitlines()
    head = [ln for ln in lines if not ln.startswith(("node", "output"))]
    nodes = [ln for ln in lines if ln.startswith("node")]
    rng = np.random.default_rng(73)
    consts = {"W0": (64, 64), "b0": (64,), "g": (64,), "be": (64,), "W1": (64, 64), "b1": (64,)}
    head += ["input z bf16 [1,6,64]", "iconst i_r3 i64 [3] = 1 6 64"] + [f"const lf.{n} bf16 [{','.join(map(str, s))}]" for n, s in consts.items()]
    first = ["node MatMul z lf.W0 -> lf0", "node Add lf0 lf.b0 -> lf1", "node Add lf1 z -> lf2",
             "node LayerNormalization lf2 lf.g lf.be -> lf3 {axis=-1 epsilon=1e-5}"]
    last = ["node Reshape gap i_r3 -> gr", "node MatMul gr lf.W1 -> lf4", "node Add lf4 lf.b1 -> lf5", "node Add lf5 lf3 -> lfy"]
    ir = "\n".join(head + first + nodes + last + [ln for ln in lines if ln.startswith("output")] + ["output lfy"]) + "\n"
    wl2 = WL.Workload("gated_ln_fold", "bf16", ir, {**wl.consts, **{"lf." + n: bf16_round((rng.standard_normal(s) / 8).astype(np.float32)) for n, s in consts.items()}},
                      wl.sym_names, wl.outputs + ["lfy"], wl.meta)
    req = wl.batch(0)[0]
    req = Request(req.syms, {**req.inputs, "z": bf16_round(rng.standard_normal((1, 6, 64)).astype(np.float32))})
    s, p, ref = run_batch(wl2, [req], opt_flags=B.OPT_LN_FOLD)
    kinds = [s.graph.group_info(i)["kind"] for i in range(s.graph.num_groups())]
    assert "layernorm" not in kinds and kinds[0] == "gemm" and kinds.index("gate") < len(kinds) - 1 - kinds[::-1].index("gemm")
    assert p.run_exact().reserved[2] == 3
    p.check_device_status()
    got = p.outputs()
    for name in ref[0]:
        assert np.array_equal(ref[0][name], got[0][name]), name


def test_plan_dropped_inside_a_callers_capture():
    # the second stream of a plan that a caller has captured and dropped belongs to the capture until it ends: another plan that
    # wants a second stream meanwhile, on another stream, gets one of its own; both give the eager run's bits
    wl = WL.cfg4(blocks=1)
    rng = np.random.default_rng(79)
    reqs = [Request({"H": 24, "W": 70}, {"x": bf16_round(rng.uniform(-1, 1, (1, 64, 24, 70)).astype(np.float32))})]
    s, p, ref = run_batch(wl, reqs)
    assert any(p.plan.group_on_side_stream(i) for i in range(s.graph.num_groups()))
    args = [t.data_ptr() for t in p.in_dev], [t.data_ptr() for t in p.out_dev], p.arena.data_ptr(), p.arena.numel()
    q = s.prepare(reqs)
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(mine):
        graph.capture_begin(capture_error_mode="relaxed")
        plan = s.graph.bind_dims(wl.sym_names, [[24, 70]]).plan()
        plan.run(*args, mine.cuda_stream)
        del plan
        q.plan.run([t.data_ptr() for t in q.in_dev], [t.data_ptr() for t in q.out_dev], q.arena.data_ptr(), q.arena.numel(), other.cuda_stream)
        graph.capture_end()
    torch.cuda.synchronize()
    got = q.outputs()
    for t in p.out_dev:
        t.zero_()
    graph.replay()
    torch.cuda.synchronize()
    again = p.outputs()
    for name in ref[0]:
        assert np.array_equal(got[0][name], ref[0][name]) and np.array_equal(again[0][name], ref[0][name])


def test_counts_are_those_of_the_last_run():
    # the counts behind an output shape are read once per run, and must not outlive it: a shape asked for through another
    # stream while the run is still waiting, several threads asking at once, replays of a caller's graph that holds the run
    import threading
    ir = "sym A 0 100000\ninput x f32 [A]\nnode NonZero x -> nz\noutput nz\n"
    wl = WL.Workload("counts", "f32", ir, {}, ["A"], ["nz"], {"batch_fn": lambda j: []})
    reqs = [Request({"A": n}, {"x": np.ones(n, np.float32)}) for n in (1000, 5000)]
    s, p, _ = run_batch(wl, reqs)
    args = [t.data_ptr() for t in p.in_dev], [t.data_ptr() for t in p.out_dev], p.arena.data_ptr(), p.arena.numel()
    shapes = lambda stream: [p.plan.output_shape(p.arena.data_ptr(), stream, r, 0) for r in range(2)]
    full, none = [[1, 1000], [1, 5000]], [[1, 0], [1, 0]]
    # another stream asks while the run waits behind a long kernel
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    p.in_dev[0].zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(mine):
        torch.cuda._sleep(200_000_000)
    p.plan.run(*args, mine.cuda_stream)
    shapes(other.cuda_stream)                            # whatever it is, it is not kept
    mine.synchronize()
    assert shapes(mine.cuda_stream) == none and shapes(other.cuda_stream) == none
    # threads
    p.in_dev[0].copy_(torch.from_numpy(p.in_host[0]))
    torch.cuda.synchronize()
    p.plan.run(*args, mine.cuda_stream)
    bad = []
    threads = [threading.Thread(target=lambda: bad.extend(i for i in range(200) if shapes(mine.cuda_stream) != full)) for _ in range(4)]
    for t in threads: t.start()
    for t in threads: t.join()
    assert not bad
    # a run inside a graph of the caller's
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(mine):
        graph.capture_begin(capture_error_mode="relaxed")
        p.plan.run(*args, mine.cuda_stream)
        graph.capture_end()
        for data, want in ((p.in_host[0], full), (np.zeros_like(p.in_host[0]), none), (p.in_host[0], full)):
            p.in_dev[0].copy_(torch.from_numpy(data))
            graph.replay()
            assert shapes(mine.cuda_stream) == want


def _relu_chain():
    return B.Graph("sym A 1 4000000000\ninput x bf16 [A]\nnode Relu x -> y\noutput y\n", 0)


def _run_relu(x, out):
    g = _relu_chain()
    plan = g.bind_dims(["A"], [[x.numel()]]).plan()
    arena = torch.empty(max(plan.arena_bytes, 256), dtype=torch.uint8, device="cuda")
    plan.run([x.data_ptr()], [out.data_ptr()], arena.data_ptr(), arena.numel(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()


@pytest.mark.parametrize("n", [2 ** 31 - 1, 2 ** 31 - 8192])
def test_chain_up_to_the_last_32_bit_index(n):
    # the largest requests that 32-bit flat indices hold, whose last tile reaches past them; the words behind stay as they are
    x = torch.empty(n + 9, dtype=torch.bfloat16, device="cuda")[:n]
    x.normal_()
    buf = torch.full((n + 9,), 7.0, dtype=torch.bfloat16, device="cuda")
    _run_relu(x, buf[:n])
    for lo in range(0, n, 1 << 28):
        hi = min(n, lo + (1 << 28))
        assert torch.equal(buf[lo:hi], torch.relu(x[lo:hi]))
    assert bool((buf[n:] == 7.0).all())


@pytest.mark.parametrize("n,dx,dy", [(100003, 1, 0), (8192, 0, 1), (8193, 3, 5), (5, 1, 1)])
def test_chain_buffers_off_16_bytes(n, dx, dy):
    # a caller's buffers that start on an odd element are read and written one element at a time
    x = torch.randn(n + 8, device="cuda").to(torch.bfloat16)[dx:dx + n]
    buf = torch.full((n + 16,), 7.0, dtype=torch.bfloat16, device="cuda")
    _run_relu(x, buf[dy:dy + n])
    assert torch.equal(buf[dy:dy + n], torch.relu(x))
    assert bool((buf[:dy] == 7.0).all()) and bool((buf[dy + n:] == 7.0).all())


def _nonzero(x, dims, out):
    """NonZero of a tensor on the GPU into `out`; returns the number of elements found."""
    names = ["A", "B", "C", "D"][:len(dims)]
    ir = "".join(f"sym {n} 0 8000000000\n" for n in names) + f"input x {'bf16' if x.dtype == torch.bfloat16 else 'f32'} [{','.join(names)}]\nnode NonZero x -> nz\noutput nz\n"
    plan = B.Graph(ir, 0).bind_dims(names, [list(dims)]).plan()
    arena = torch.empty(max(plan.arena_bytes, 256), dtype=torch.uint8, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    plan.run([x.data_ptr()], [out.data_ptr()], arena.data_ptr(), arena.numel(), stream)
    return plan.output_shape(arena.data_ptr(), stream, 0, 0)[1]


def test_nonzero_finds_more_than_32_bits_count():
    # every element non-zero, more of them than an int holds: offsets and the count itself
    n = 2 ** 31 + 4099
    x = torch.ones(n, dtype=torch.bfloat16, device="cuda")
    out = torch.empty(n, dtype=torch.int64, device="cuda")
    assert _nonzero(x, (n,), out) == n
    for lo in range(0, n, 1 << 28):
        hi = min(n, lo + (1 << 28))
        assert torch.equal(out[lo:hi], torch.arange(lo, hi, device="cuda"))


@pytest.mark.parametrize("rows,cols", [(4099, 4097), (2 ** 20 + 1, 4097)])
def test_nonzero_chunks_of_several_pieces(rows, cols):
    # above 2048 x 8192 elements a chunk has several pieces, above 2^32 the coordinates are worked out in 64 bits
    n = rows * cols
    x = torch.zeros(n, dtype=torch.bfloat16, device="cuda")
    at = torch.tensor(sorted({0, 1, 8191, 8192, cols - 1, cols, n // 2, n // 2 + 1, n - cols, n - 8193, n - 2, n - 1}), device="cuda")
    x[at] = 1.0
    k = at.numel()
    out = torch.full((2 * k,), -1, dtype=torch.int64, device="cuda")
    assert _nonzero(x, (rows, cols), out) == k
    assert torch.equal(out[:k], at // cols) and torch.equal(out[k:], at % cols)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n", [5, 8193, 40001])
def test_nonzero_of_a_buffer_off_16_bytes(dtype, n):
    x = (torch.randn(n + 1, device="cuda") * (torch.rand(n + 1, device="cuda") < 0.5)).to(dtype)[1:]
    want = torch.nonzero(x).flatten()
    out = torch.empty(n, dtype=torch.int64, device="cuda")
    assert _nonzero(x, (n,), out) == want.numel()
    assert torch.equal(out[:want.numel()], want)
