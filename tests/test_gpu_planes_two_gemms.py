"""Two GEMM loops share one room for bfloat16 planes, so neither's operands are formed there by the
INIT loop: both results carry the bits of the program whose operands are kept as binary32, and
of each GEMM alone on the GPU."""
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


@pytest.mark.parametrize("prec", [1, 2, 3])
def test_two_gemms(gao, prec):
    n = 200
    got = []
    for keep in (False, True):
        role = W.OUTPUT if keep else W.TEMP
        bufs = [W.Buffer(nm, n, n, role=role) for nm in ("A", "B", "A2", "B2")]
        bufs += [W.Buffer("C0", n, n), W.Buffer("C", n, n, role=W.OUTPUT), W.Buffer("C2", n, n, role=W.OUTPUT)]
        loops = [W.Loop(W.INIT, [], [0, 1, 2, 3]), W.Loop(W.INIT, [], [4]), W.Loop(W.GEMM, [0, 1, 4], [5], 1.5, 0.5),
                 W.Loop(W.GEMM, [2, 3, 4], [6], 1.5, 0.5)]
        p = gao.prog_create(bufs, loops, seed=8, gemm_prec=prec)
        for _ in range(3):
            gao.prog_run(p, 0b1111)
            got.append((gao.prog_output(p, 5), gao.prog_output(p, 6)))
            assert gao.prog_planes_for(p, 0) == -1 and gao.prog_planes_for(p, 3) == -1
        gao.prog_run(p, 0b0111)
        assert np.array_equal(gao.prog_output(p, 5).view(np.uint32), got[-1][0].view(np.uint32))
        assert gao.prog_planes_for(p, 0) == (-1 if keep else 2)
        gao.prog_destroy(p)
    for c, c2 in got:
        assert np.array_equal(c.view(np.uint32), got[-1][0].view(np.uint32))
        assert np.array_equal(c2.view(np.uint32), got[-1][1].view(np.uint32))
