"""Split GEMMs on rows of any alignment with eight and with sixteen epilogue warps: on both sides of
the inner dimensions where the number changes, the bits of the same columns in a product with
16-byte aligned rows."""
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


@pytest.mark.parametrize("prec,kchunk", [(2, 0), (2, 4096), (3, 0), (3, 4096)])
@pytest.mark.parametrize("below", [0, 1])
def test_unaligned_rows_behind_a_long_inner_dimension(gao, prec, kchunk, below):
    m, n, k = 3201, 3203, 1000 * prec - below  # 26 x 26 tiles: more than four an SM
    rng = np.random.default_rng(k)
    A, B, C0 = (rng.standard_normal(s).astype(np.float32) for s in ((m, k), (k, n), (m, n)))
    out = []
    for w in (n, n + 1):
        pad = lambda x: np.pad(x, ((0, 0), (0, w - n)))
        bufs = [W.Buffer("X", m, k, role=W.INPUT), W.Buffer("B", k, w, role=W.INPUT), W.Buffer("C0", m, w, role=W.INPUT),
                W.Buffer("C", m, w, role=W.OUTPUT), W.Buffer("A", m, k)]
        # A on the device when the GEMM runs: one launch, not row blocks
        loops = [W.Loop(W.RELU, [0], [4]), W.Loop(W.GEMM, [4, 1, 2], [3], 1.5, 0.5)]
        p = gao.prog_create(bufs, loops, gemm_prec=prec, kchunk=kchunk)
        for i, x in enumerate((A, pad(B), pad(C0))):
            gao.prog_set_input(p, i, x)
        gao.prog_run(p, 0b11)
        out.append(gao.prog_output(p, 3)[:, :n].copy())
        gao.prog_destroy(p)
    assert np.array_equal(out[0].view(np.uint32), out[1].view(np.uint32))
