"""Small outputs stored to the host by one launch: sizes of one element up to the largest copied
this way and just above it, sixty at a time, binary64 scalars, and an output bound to the
caller's array, each the host loops' bits on the first, the captured and the replayed run."""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gao():
    from paper_1806_01430_gb300 import _build
    _build.build()
    import paper_1806_01430_gb300 as g
    return g


def spoil(gao, p, b, nbytes):
    """Fill buffer b's mirror with something that no run writes."""
    ptr = ctypes.c_void_p(None)
    assert gao.lib().prog_output(p.handle, b, ctypes.byref(ptr), None) == gao.GAO_OK
    ctypes.memset(ptr.value, 0xA5, nbytes)


def check(gao, bufs, loops, bound=None):
    p = gao.prog_create(bufs, loops, seed=11)
    keep = np.zeros((bufs[bound].rows, bufs[bound].cols), np.float32) if bound is not None else None
    if bound is not None:
        gao.prog_bind_host(p, bound, keep)
    outs = [b for b in range(len(bufs)) if bufs[b].role == W.OUTPUT and b != bound]
    gao.prog_run(p, 0)
    want = {b: gao.prog_output(p, b).copy() for b in outs}
    want_bound = keep.copy() if bound is not None else None
    for _ in range(3):
        for b in outs:
            spoil(gao, p, b, want[b].nbytes)
        if bound is not None:
            keep[...] = -7.0
        gao.prog_run(p, (1 << len(loops)) - 1)
        for b in outs:
            got = gao.prog_output(p, b)
            if got.dtype == np.float32:
                assert np.array_equal(got.view(np.uint32), want[b].view(np.uint32)), b
            else:
                # partials of up to four of the 131040 values in [-1, 1] are rounded to binary32 twice
                assert abs(got[0, 0] - want[b][0, 0]) <= 4 * 2.0 ** -24 * 131040, b
        if bound is not None:
            assert np.array_equal(keep.view(np.uint32), want_bound.view(np.uint32))
    gao.prog_destroy(p)


def test_sizes(gao):
    shapes = [(1, 1), (3, 1), (1, 4), (1, 5), (7, 1), (255, 4), (1024, 4), (1, 1025), (360, 364), (256, 512),
              (131073, 1), (300, 700)]  # (256, 512): 512 KiB
    bufs = [W.Buffer(f"o{i}", r, c, role=W.OUTPUT) for i, (r, c) in enumerate(shapes)]
    n = len(shapes)
    loops = [W.Loop(W.INIT, [], list(range(i, min(i + 4, n)))) for i in range(0, n, 4)]
    bufs += [W.Buffer("s", 1, 1, W.F64, W.OUTPUT), W.Buffer("f", 1, 1, W.F64, W.OUTPUT)]
    loops += [W.Loop(W.SUM, [8], [n]), W.Loop(W.FROBENIUS, [5], [n + 1])]
    check(gao, bufs, loops)
    check(gao, bufs, loops, bound=5)


def test_many_outputs(gao):
    bufs = [W.Buffer(f"o{i}", 1 + i % 5, 1 + (i % 12) * 7, role=W.OUTPUT) for i in range(12)]
    loops = [W.Loop(W.INIT, [], list(range(i, i + 4))) for i in range(0, 12, 4)]
    for i in range(48):
        bufs.append(W.Buffer(f"r{i}", bufs[i % 12].rows, bufs[i % 12].cols, role=W.OUTPUT))
        loops.append(W.Loop(W.RELU, [i % 12], [12 + i]))
    check(gao, bufs, loops)
