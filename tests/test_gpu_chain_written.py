"""An element-wise chain in one pass with one, some or all of its values written, over one, two and
three arrays (one written value and at most two arrays: loaded before the first operation), at
the edges of its quadruples: the bits of the separate loops."""
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


L = W.Loop
CHAINS = {"one": (1, [L(W.RELU, [0], [3]), L(W.SQUARE, [3], [4]), L(W.AXPY, [4, 4], [5], -0.5)]),
          "two": (2, [L(W.RELU, [0], [3]), L(W.AXPY, [0, 3], [4], -0.5), L(W.SQUARE, [4], [5]), L(W.AXPY, [5, 1], [6], 0.25)]),
          "twice": (2, [L(W.RELU, [0], [3]), L(W.SQUARE, [3], [4]), L(W.AXPY, [4, 0], [3], 1.0), L(W.AXPY, [3, 1], [5], 2.0)]),
          "three": (3, [L(W.AXPY, [0, 1], [3], 3.0), L(W.SQUARE, [3], [4]), L(W.AXPY, [2, 4], [5], -1.5)])}


@pytest.mark.parametrize("rows,cols", [(1, 1), (3, 5), (129, 66), (1025, 1024)])
@pytest.mark.parametrize("written", [1, 2, 4])
@pytest.mark.parametrize("kind", sorted(CHAINS))
def test_chain_with_values_written(gao, kind, written, rows, cols):
    ext, ops = CHAINS[kind]
    bufs = [W.Buffer(f"b{i}", rows, cols) for i in range(7)]
    outs = sorted({op.outs[0] for op in ops[-written:]})
    for b in outs:
        bufs[b].role = W.OUTPUT
    loops = [L(W.INIT, [], list(range(ext)))] + ops
    got = []
    for fuse in (0, 1):
        p = gao.prog_create(bufs, loops, seed=rows + cols, fuse_chains=fuse)
        gao.prog_run(p, (1 << len(loops)) - 1)
        got.append([gao.prog_output(p, b).copy().view(np.uint32) for b in outs])
        assert [s["placement"] for s in gao.prog_stats(p)][2:] == [2 if fuse else 1] * (len(ops) - 1)
        gao.prog_destroy(p)
    for a, b in zip(*got):
        assert np.array_equal(a, b)
