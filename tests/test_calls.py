"""Arguments of the per-batch calls: what is refused before anything reaches the GPU."""
import ctypes as C

import pytest

from paper_2403_00176_b200 import binding as B

IR = "sym A 1 100\ninput x f32 [A]\ninput z f32 [A]\nnode Add x z -> y\noutput y\n"


def _plan(ir=IR, names=("A",), values=((5,),)):
    return B.Graph(ir, 0).bind_dims(list(names), [list(v) for v in values]).plan()


@pytest.mark.parametrize("ins,outs", [([], [256]), ([256], [256]), ([256, None], [256]), ([256, 512], []), ([256, 512], [None]), ([256, 0], [256]),
                                      ([C.c_void_p(256), C.c_void_p(None)], [256])])
@pytest.mark.parametrize("how", ["run", "run_graph", "run_exact"])
def test_missing_and_null_buffers_are_refused(how, ins, outs):
    # a list that lacks a buffer is a list with a null buffer, whatever the stack holds behind it
    p = _plan()
    for filler in (1 << 20, 3 << 20):
        # a call that is refused for its arena leaves the stack full of addresses
        with pytest.raises(B.Sod2Error, match="ARENA_TOO_SMALL"):
            p.run([filler] * 64, [filler] * 64, 256, 0, 0)
        with pytest.raises(B.Sod2Error, match="INVALID_ARG"):
            getattr(p, how)(ins, outs, 1 << 30, 1 << 20, 0)


def test_entries_may_be_ctypes_pointers():
    # (refused for the arena, that is after the lists have been read)
    p = _plan()
    with pytest.raises(B.Sod2Error, match="ARENA_TOO_SMALL"):
        p.run([C.c_void_p(256), 512], (C.c_void_p(256),), 256, 0, 0)
    with pytest.raises(TypeError):
        p.run(["x", 512], [256], 256, 0, 0)


def test_more_buffers_than_the_call_keeps_on_the_stack():
    n = 70
    ir = "".join(f"input x{i} f32 [3]\n" for i in range(n)) + "".join(f"node Relu x{i} -> y{i}\noutput y{i}\n" for i in range(n))
    p = _plan(ir, (), ((),))
    with pytest.raises(B.Sod2Error, match="INVALID_ARG"):
        p.run([256] * (n - 1), [256] * n, 1 << 30, 1 << 20, 0)
    with pytest.raises(B.Sod2Error, match="ARENA_TOO_SMALL"):
        p.run([256] * (n + 3), [256] * n, 256, 0, 0)
