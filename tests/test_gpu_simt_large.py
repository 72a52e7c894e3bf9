"""FP32 SIMT GEMM on its large tiles with rows of any alignment: operands read a word at a time, K of a
step or less up to several chunks, whole and split over a cluster, C0 in a buffer of its own and
in C's: the bits of the host loop."""
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


@pytest.mark.parametrize("own", [False, True])
@pytest.mark.parametrize("M,N,K", [(2049, 2051, 1), (2049, 2051, 33), (2048, 2052, 33), (2050, 2049, 256), (2049, 2050, 273),
                                   (202, 1415, 1040), (1442, 205, 1044)])
def test_large_tiles_of_any_alignment(gao, M, N, K, own):
    c0 = 3 if own else 2
    bufs = [W.Buffer("A", M, K), W.Buffer("B", K, N), W.Buffer("C", M, N, role=W.OUTPUT)] + [W.Buffer("C0", M, N)] * own
    loops = [W.Loop(W.INIT, [], [0, 1, c0]), W.Loop(W.GEMM, [0, 1, c0], [2], 1.5, 0.5)]
    out = {}
    p = gao.prog_create(bufs, loops, seed=M + N + K)
    for mask in (0b01, 0b11):
        gao.prog_run(p, mask)
        out[mask] = gao.prog_output(p, 2).copy()
    gao.prog_destroy(p)
    assert np.array_equal(out[0b01].view(np.uint32), out[0b11].view(np.uint32))
