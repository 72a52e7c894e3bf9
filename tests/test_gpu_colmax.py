"""Column maxima at the edges of the column strips (32, 64 or 128 columns), of the clusters (1 to 8
blocks of rows) and of the fallback for tall inputs of few columns: equal to numpy's maxima,
for any row alignment, with infinities, -0 and NaNs of either sign ordered as the host loop
orders them (a NaN with a clear sign above everything, one with a set sign below)."""
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


@pytest.mark.parametrize("rows,cols", [
    (1, 1), (1, 5), (2, 33), (31, 32), (129, 31), (257, 64), (511, 65), (513, 128), (1080, 1921), (64, 4864), (70, 9729),
    (1000, 19456), (16384, 4), (16385, 4), (40000, 3), (20000, 300)])
def test_column_maxima(gao, rows, cols):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(rows + cols)
    X = rng.standard_normal((rows, cols)).astype(np.float32)
    special = {0: 0x7F800000, 1: 0x7FC00001, 2: 0xFFC00000, 3: 0x80000000}  # +inf, NaN, -NaN, -0 per column
    for c, bits in special.items():
        if c < cols:
            X.view(np.uint32)[rng.integers(rows), c] = bits
    # the order of the values as unsigned integers: all bits flipped below zero, the sign bit above
    u = X.view(np.uint32)
    key = np.where(u >> 31, ~u, u | np.uint32(0x80000000)).max(axis=0)
    want = np.where(key >> 31, key & np.uint32(0x7FFFFFFF), ~key).view(np.float32)
    if cols > 4:
        assert np.array_equal(want[4:], X[:, 4:].max(axis=0))
    d = torch.from_numpy(X).cuda()
    out = torch.empty(cols, device="cuda")
    assert gao.gao_colmax_noalloc(d.data_ptr(), rows, cols, out.data_ptr()) == gao.GAO_OK
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.array_equal(got.view(np.uint32), want.view(np.uint32))
    # the COLMAX loop of a program, on the GPU and on the host
    bufs = [W.Buffer("X", rows, cols, role=W.INPUT), W.Buffer("q", 1, cols, role=W.OUTPUT)]
    p = gao.prog_create(bufs, [W.Loop(W.COLMAX, [0], [1])])
    gao.prog_set_input(p, 0, X)
    for mask in (1, 0):
        gao.prog_run(p, mask)
        assert np.array_equal(gao.prog_output(p, 1).ravel().view(np.uint32), want.view(np.uint32)), mask
    gao.prog_destroy(p)
