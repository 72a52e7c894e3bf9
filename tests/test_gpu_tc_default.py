"""The epilogue that the tensor-core precisions choose for rows that are not 16-byte aligned
carries the bits of the same columns in a product with aligned rows."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
PREC = {"bf16": 1, "bf16x3": 2, "bf16x6": 3, "fp8": 4}


@pytest.fixture(scope="module")
def gao():
    from paper_1806_01430_gb300 import _build
    _build.build()
    import paper_1806_01430_gb300 as g
    return g


@pytest.mark.parametrize("prec", ["bf16", "bf16x3", "bf16x6", "fp8"])
@pytest.mark.parametrize("m,k,n", [(1, 1, 1), (33, 70, 31), (129, 300, 257), (500, 129, 1023)])
def test_unaligned_rows_carry_the_aligned_bits(gao, prec, m, k, n):
    rng = np.random.default_rng(m + k + n)
    A, B, C0 = (rng.standard_normal(s).astype(np.float32) for s in ((m, k), (k, n), (m, n)))
    wide = -(-n // 4) * 4 + (4 if n % 4 == 0 else 0)
    out = []
    for w in (n, wide):
        pad = lambda x: np.pad(x, ((0, 0), (0, w - n)))
        bufs = [W.Buffer("A", m, k, role=W.INPUT), W.Buffer("B", k, w, role=W.INPUT),
                W.Buffer("C0", m, w, role=W.INPUT), W.Buffer("C", m, w, role=W.OUTPUT)]
        p = gao.prog_create(bufs, [W.Loop(W.GEMM, [0, 1, 2], [3], 1.5, 0.5)], gemm_prec=PREC[prec])
        for i, x in enumerate((A, pad(B), pad(C0))):
            gao.prog_set_input(p, i, x)
        gao.prog_run(p, 1)
        out.append(gao.prog_output(p, 3)[:, :n].copy())
        gao.prog_destroy(p)
    assert np.array_equal(out[0].view(np.uint32), out[1].view(np.uint32))
