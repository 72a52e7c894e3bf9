"""SUM and COLMAX of an element-wise chain's last value formed in the chain's pass: at the edges
of the column strips and of their clusters, for chains of one operation and more over one, two
and three arrays, the column maxima carry the bits of the separate loops and the sum is within
its rounding of them.  Asking for the unwritten value's device pointer forms it."""
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


def chain(kind):
    """Loops over X, Y, Z (0, 1, 2) and temporaries 3, 4, 5; the last output."""
    L = W.Loop
    return {"one": ([L(W.SQUARE, [0], [3])], 3),
            "self": ([L(W.AXPY, [0, 0], [3], -0.5), L(W.AXPY, [3, 3], [4], 0.25)], 4),
            "two": ([L(W.RELU, [0], [3]), L(W.AXPY, [0, 3], [4], -0.75), L(W.AXPY, [4, 1], [5], 2.0)], 5),
            "three": ([L(W.AXPY, [0, 1], [3], 3.0), L(W.SQUARE, [3], [4]), L(W.AXPY, [2, 4], [5], -1.5)], 5)}[kind]


@pytest.mark.parametrize("rows,cols", [(1, 1), (3, 5), (31, 32), (129, 66), (512, 128), (300, 1001), (1025, 4864),
                                       (40000, 3), (2000, 3000)])
@pytest.mark.parametrize("kind,reduce", [("one", "both"), ("self", "sum"), ("two", "both"), ("two", "colmax"),
                                         ("three", "both")])
def test_reductions_in_the_chain(gao, rows, cols, kind, reduce):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(rows * 7 + cols)
    ops, last = chain(kind)
    bufs = [W.Buffer(n, rows, cols, role=W.INPUT) for n in "XYZ"] + [W.Buffer(n, rows, cols) for n in "PQR"]
    bufs += [W.Buffer("s", 1, 1, W.F64, W.TEMP if reduce == "colmax" else W.OUTPUT),
             W.Buffer("q", 1, cols, role=W.TEMP if reduce == "sum" else W.OUTPUT)]
    loops = ops + ([W.Loop(W.SUM, [last], [6])] if reduce != "colmax" else [])
    loops += [W.Loop(W.COLMAX, [last], [7])] if reduce != "sum" else []
    data = [rng.standard_normal((rows, cols)).astype(np.float32) for _ in range(3)]
    nbytes = gao.prog_device_bytes(bufs, loops)
    got = {}
    for fuse in (0, 1):
        raw = torch.empty(nbytes + 1024, dtype=torch.uint8, device="cuda")
        arena = raw[-raw.data_ptr() % 1024:][:nbytes]
        torch.cuda.synchronize()
        p = gao.prog_create(bufs, loops, fuse_chains=fuse, arena=arena)
        for i in range(3):
            gao.prog_set_input(p, i, data[i])
        for _ in range(3):  # the second run is captured, the third replayed
            gao.prog_run(p, (1 << len(loops)) - 1)
        placed = [s["placement"] for s in gao.prog_stats(p)]
        fits = rows < 16384  # taller inputs of few columns keep the separate reductions
        assert placed[len(ops):] == [2 if fuse and fits else 1] * (len(loops) - len(ops)), placed
        out = {6: gao.prog_output(p, 6).copy() if reduce != "colmax" else None,
               7: gao.prog_output(p, 7).copy() if reduce != "sum" else None}
        off = gao.prog_device_ptr(p, last) - arena.data_ptr()
        out[3] = arena[off:off + rows * cols * 4].cpu().numpy().view(np.uint32).reshape(rows, cols)
        got[fuse] = out
        gao.prog_destroy(p)
    assert np.array_equal(got[0][3], got[1][3])
    v = got[1][3].view(np.float32).astype(np.float64)
    if reduce != "sum":
        assert np.array_equal(got[0][7].view(np.uint32), got[1][7].view(np.uint32))
        assert np.array_equal(got[1][7].ravel(), v.max(axis=0).astype(np.float32))
    if reduce != "colmax":
        # partials of four columns are rounded to binary32 twice, what is added to them is compensated
        bound = 4 * 2.0 ** -24 * np.abs(v).sum() + 1e-300
        for fuse in (0, 1):
            assert abs(float(got[fuse][6][0, 0]) - v.sum()) <= bound
