"""The fused image pass with every intermediate map written, at the edges of a lane's eight, a warp's
240 and a block's 960 columns and of the three-row steps, rows of any alignment: the bits of the
separate loops, the edge energy within its rounding, equal column maxima."""
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


@pytest.mark.parametrize("presets", [(0, 2, 3), (1, 3, 0)])
@pytest.mark.parametrize("rows,cols", [(1, 1), (2, 7), (5, 9), (17, 63), (50, 239), (18, 240), (33, 241), (49, 249), (20, 481),
                                       (19, 959), (21, 964), (35, 1201), (200, 1923)])
def test_every_map_written(gao, rows, cols, presets):
    L, o = W.Loop, W.OUTPUT
    bufs = [W.Buffer("X", rows, cols)] + [W.Buffer(n, rows, cols, role=o) for n in ("B", "gx", "gy", "sx", "sy", "M")]
    bufs += [W.Buffer("e", 1, 1, W.F64, o), W.Buffer("q", 1, cols, role=o)]
    loops = [L(W.INIT, [], [0]), L(W.STENCIL3, [0], [1], flags=presets[0]), L(W.STENCIL3, [1], [2], flags=presets[1]),
             L(W.STENCIL3, [1], [3], flags=presets[2]), L(W.SQUARE, [2], [4]), L(W.SQUARE, [3], [5]),
             L(W.AXPY, [4, 5], [6], 1.0), L(W.SUM, [6], [7]), L(W.COLMAX, [6], [8])]
    got = []
    for fuse in (0, 1):
        p = gao.prog_create(bufs, loops, seed=rows * cols, fuse_chains=fuse)
        gao.prog_run(p, (1 << len(loops)) - 1)
        got.append([gao.prog_output(p, b).copy() for b in range(1, 9)])
        placed = [s["placement"] for s in gao.prog_stats(p)]
        gao.prog_destroy(p)
    assert placed == [1, 1] + [2] * 7
    for b in (0, 1, 2, 3, 4, 5, 7):
        assert np.array_equal(got[0][b].view(np.uint32), got[1][b].view(np.uint32)), b
    # partials of up to eight values are rounded to binary32 three times
    M = got[0][5].astype(np.float64)
    for g in got:
        assert abs(g[6][0, 0] - M.sum()) <= 6 * 2.0 ** -24 * M.sum()
