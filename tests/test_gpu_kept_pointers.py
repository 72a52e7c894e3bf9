"""A device pointer taken once and read after every run: operands that INIT would form as a
GEMM's planes or codes and the last value of a reduced element-wise chain, each spoiled between
runs, carry the unfused binary32 program's bits -- taken before the first run, or after the run
was captured."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
BF16X3, BF16X6, FP8 = 2, 3, 4


@pytest.fixture(scope="module")
def gao():
    from paper_1806_01430_gb300 import _build
    _build.build()
    import paper_1806_01430_gb300 as g
    return g


def gemm(m, k, n):
    bufs = [W.Buffer("A", m, k), W.Buffer("B", k, n), W.Buffer("C0", m, n), W.Buffer("C", m, n, role=W.OUTPUT)]
    return bufs, [W.Loop(W.INIT, [], [0, 1, 2], flags=1), W.Loop(W.GEMM, [0, 1, 2], [3], 1.5, 0.5)]


def chain(n):
    o, L = W.OUTPUT, W.Loop
    bufs = [W.Buffer(nm, n, n) for nm in ("A", "B", "C", "S", "D", "E", "P")] + [W.Buffer("s", 1, 1, W.F64, o)]
    return bufs, [L(W.INIT, [], [0, 1, 2, 3]), L(W.GEMM, [0, 1, 2], [2], 1.5, 0.5), L(W.AXPY, [2, 3], [4], 2.0),
                  L(W.TRANSPOSE, [4], [5]), L(W.SQUARE, [5], [6]), L(W.SUM, [6], [7])]


CASES = {"gemm_x6": (gemm(300, 129, 200), BF16X6, 0, (0, 1)), "gemm_fp8": (gemm(300, 129, 201), FP8, 0, (0, 1)),
         "chain_x3": (chain(2052), BF16X3, 1, (0, 1, 6))}


@pytest.mark.parametrize("before", [0, 3])
@pytest.mark.parametrize("case", sorted(CASES))
def test_kept_pointer_sees_every_run(gao, case, before):
    torch = pytest.importorskip("torch")
    (bufs, loops), prec, fuse, kept = CASES[case]
    nbytes = gao.prog_device_bytes(bufs, loops, gemm_prec=prec)
    gene = (1 << len(loops)) - 1

    def make(fuse_chains):
        raw = torch.empty(nbytes + 1024, dtype=torch.uint8, device="cuda")
        arena = raw[-raw.data_ptr() % 1024:][:nbytes]
        torch.cuda.synchronize()
        p = gao.prog_create(bufs, loops, seed=5, gemm_prec=prec, fuse_chains=fuse_chains, arena=arena)

        def view(b):
            off = gao.prog_device_ptr(p, b) - arena.data_ptr()
            return arena[off:off + 4 * bufs[b].rows * bufs[b].cols].view(torch.int32)
        return p, view

    p, view = make(0)
    gao.prog_run(p, gene)
    want = {b: view(b).clone() for b in kept}
    gao.prog_destroy(p)
    p, view = make(fuse)
    for _ in range(before):
        gao.prog_run(p, gene)
    held = {b: view(b) for b in kept}
    if before:
        for b in kept:
            assert torch.equal(held[b], want[b]), b
    for _ in range(4):
        for b in kept:
            held[b].fill_(0x7FC00000)
        torch.cuda.synchronize()
        gao.prog_run(p, gene)
        for b in kept:
            assert torch.equal(held[b], want[b]), b
            assert gao.prog_planes_for(p, b) == -1
    gao.prog_destroy(p)


def test_batch_run_ends_the_planes_of_a_run_alone(gao):
    """A batch writes binary32 operands: what an earlier run of the program formed as planes is
    not reported, or formed again, after it."""
    bufs, loops = gemm(200, 129, 300)
    p = gao.prog_create(bufs, loops, seed=7, gemm_prec=BF16X3)
    gao.prog_run(p, 0b11)
    assert [gao.prog_planes_for(p, b) for b in (0, 1)] == [1, 1]
    b = gao.batch_create([p])
    gao.batch_evaluate(b, [0b11])
    assert [gao.prog_planes_for(p, i) for i in (0, 1)] == [-1, -1]
    gao.batch_destroy(b)
    gao.prog_destroy(p)
