"""A replayed run leaves the operands that it formed as a GEMM's planes known as such, whatever
gene ran between: the residual check and the device pointer still form their values."""
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


@pytest.mark.parametrize("between", [0b00, 0b01, 0b10])
def test_planes_after_a_replay(gao, between):
    n = 200
    bufs = [W.Buffer(nm, n, n) for nm in ("A", "B", "C0")] + [W.Buffer("C", n, n, role=W.OUTPUT)]
    p = gao.prog_create(bufs, [W.Loop(W.INIT, [], [0, 1, 2]), W.Loop(W.GEMM, [0, 1, 2], [3], 1.5, 0.5)], seed=9, gemm_prec=3)
    rng = np.random.default_rng(1)
    x, y = rng.choice([-1.0, 1.0], n), rng.choice([-1.0, 1.0], n)
    for gene in (0b11, 0b11, between):
        gao.prog_run(p, gene)
    for _ in range(2):
        gao.prog_run(p, 0b11)  # replayed
        assert [gao.prog_planes_for(p, b) for b in (0, 1)] == [1, 1]
        r = gao.prog_gemm_residual(p, 1, x, y)
        assert max(r["right"], r["left"]) <= 1e-6
        assert [gao.prog_planes_for(p, b) for b in (0, 1)] == [-1, -1]
    gao.prog_destroy(p)
