"""An operand formed as a GEMM's planes beside an A that is on the host when the GEMM runs -- an
INPUT, or rewritten by a host loop after the INIT loop -- on both sides of the size from which
such an A is copied in row blocks: the bits of the program whose B is kept as binary32, with the
chain fused and apart, on the first, the captured and the replayed run."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
N, SEED = 2080, 12


@pytest.fixture(scope="module")
def gao():
    from paper_1806_01430_gb300 import _build
    _build.build()
    import paper_1806_01430_gb300 as g
    return g


def program(kind, m, k, keep):
    o, L = W.OUTPUT, W.Loop
    bufs = [W.Buffer("A", m, k, role=W.INPUT if kind == "input" else W.TEMP), W.Buffer("B", k, N, role=o if keep else W.TEMP),
            W.Buffer("C0", m, N), W.Buffer("C", m, N, role=o), W.Buffer("S", m, N), W.Buffer("D", m, N),
            W.Buffer("E", N, m, role=o)]
    loops = [L(W.INIT, [], [1, 2, 4] if kind == "input" else [0, 1, 2, 4])]
    if kind != "input":
        loops.append(L(W.RELU, [0], [0]))
    return bufs, loops + [L(W.GEMM, [0, 1, 2], [3], 1.5, 0.5), L(W.AXPY, [3, 4], [5], 2.0), L(W.TRANSPOSE, [5], [6])]


@pytest.mark.parametrize("prec", [1, 2, 3, 4])
@pytest.mark.parametrize("fuse", [0, 1])
@pytest.mark.parametrize("kind,gene", [("input", 0b1111), ("rewritten", 0b11101), ("rewritten", 0b11111)])
@pytest.mark.parametrize("m,k", [(2304, 2048), (300, 2048)])
def test_planes_beside_a_host_operand(gao, prec, fuse, kind, gene, m, k):
    rng = np.random.default_rng(m)
    A = rng.standard_normal((m, k)).astype(np.float32)
    got = []
    for keep in (False, True):
        bufs, loops = program(kind, m, k, keep)
        p = gao.prog_create(bufs, loops, seed=SEED, gemm_prec=prec, fuse_chains=fuse)
        if kind == "input":
            gao.prog_set_input(p, 0, A)
        for _ in range(3):
            gao.prog_run(p, gene)
            got.append([gao.prog_output(p, b).copy() for b in (3, 6)])
        gao.prog_destroy(p)
    for g in got[:-1]:
        for a, b in zip(g, got[-1]):
            assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
