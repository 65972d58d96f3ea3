"""Kernel edges on the GPU: sizes at the ends of tiles, items and dispatch rules, against the oracle."""
import numpy as np
import pytest

from oracle import interp as O
from paper_2403_00176_b200 import workloads as WL
from paper_2403_00176_b200.workloads import Request, bf16_round
from tests.gpu_harness import run_batch

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
