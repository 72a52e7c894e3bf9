"""Column maxima on both sides of the sizes where strips (one launch) give way to keys in global
memory (two): the route taken, torch's maxima, and no key of an earlier call left in a later
one whose maxima are all smaller.  A chain with the sum and column maxima of its last value
keeps separate passes for tall inputs of few columns."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gao():
    from paper_1806_01430_gb300 import _build
    _build.build()
    import paper_1806_01430_gb300 as g
    return g


@pytest.mark.parametrize("rows,cols,launches", [
    (8192, 16, 1), (8193, 16, 2), (16384, 17, 1), (16385, 17, 2), (16384, 288, 1), (16385, 288, 2), (65536, 292, 1),
    (65537, 292, 2), (65537, 293, 1), (8192, 8192, 1), (8193, 8192, 2), (8193, 8191, 1),
    (10240, 4900, 1), (10280, 4900, 2)])
def test_route_and_maxima(gao, rows, cols, launches):
    torch = pytest.importorskip("torch")
    p = gao.prog_create([W.Buffer("X", rows, cols), W.Buffer("q", 1, cols, role=W.OUTPUT)],
                        [W.Loop(W.INIT, [], [0]), W.Loop(W.COLMAX, [0], [1])], seed=3)
    gao.prog_run(p, 0b11)
    assert gao.prog_stats(p)[1]["launches"] == launches
    gao.prog_destroy(p)
    X = torch.randn(rows, cols, device="cuda", generator=torch.Generator("cuda").manual_seed(rows + cols))
    out = torch.empty(cols, device="cuda")
    for _ in range(2):
        assert gao.gao_colmax_noalloc(X.data_ptr(), rows, cols, out.data_ptr(), torch.cuda.current_stream()) == gao.GAO_OK
        assert torch.equal(out, X.amax(0))
        X -= 100.0


@pytest.mark.parametrize("rows,cols,fused", [(131072, 300, True), (131073, 300, False), (131073, 353, True)])
def test_route_of_a_reduced_chain(gao, rows, cols, fused):
    L = W.Loop
    bufs = [W.Buffer("X", rows, cols), W.Buffer("P", rows, cols), W.Buffer("q", 1, cols, role=W.OUTPUT)]
    got = []
    for fuse in (1, 0):
        p = gao.prog_create(bufs, [L(W.INIT, [], [0]), L(W.SQUARE, [0], [1]), L(W.COLMAX, [1], [2])], seed=4, fuse_chains=fuse)
        gao.prog_run(p, 0b111)
        got.append((gao.prog_output(p, 2).copy(), gao.prog_stats(p)[2]["placement"]))
        gao.prog_destroy(p)
    assert got[0][1] == (2 if fused else 1)
    assert (got[0][0] == got[1][0]).all()
