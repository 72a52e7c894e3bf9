"""The tile shapes and epilogues that the split precisions choose by size, alignment and chain: the
default carries the bits of the one-CTA tiles (and of the same columns in a product with
16-byte aligned rows), on both sides of the sizes where it changes."""
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


def chain_program(m, k, n, keep):
    o = W.OUTPUT
    ab = o if keep else W.TEMP  # kept: split by the GEMM; else formed as planes where large enough
    bufs = [W.Buffer("A", m, k, role=ab), W.Buffer("B", k, n, role=ab), W.Buffer("C", m, n, role=o), W.Buffer("S", m, n),
            W.Buffer("D", m, n), W.Buffer("E", n, m, role=o), W.Buffer("r", n, 1, role=o),
            W.Buffer("f", 1, 1, W.F64, o)]
    L = W.Loop
    return bufs, [L(W.INIT, [], [0, 1, 2, 3]), L(W.GEMM, [0, 1, 2], [2], 1.5, 0.5), L(W.AXPY, [2, 3], [4], 2.0),
                  L(W.TRANSPOSE, [4], [5]), L(W.ROWSUM, [5], [6]), L(W.FROBENIUS, [5], [7])]


@pytest.mark.parametrize("prec", ["bf16x3", "bf16x6"])
@pytest.mark.parametrize("m,k,n", [(3968, 1500, 3840), (3968, 1499, 3840), (3841, 1600, 3969), (3840, 1500, 3712),
                                   (2433, 1500, 3072)])
def test_chain_default_against_one_cta(gao, prec, m, k, n):
    got = []
    for cfg, keep in ((0, False), (0, True), (1, False), (9, True), (13, False)):
        bufs, loops = chain_program(m, k, n, keep)
        p = gao.prog_create(bufs, loops, seed=3, gemm_prec=PREC[prec], tile_cfg=cfg, fuse_chains=1)
        gao.prog_run(p, 0b111111)
        got.append([gao.prog_output(p, b).copy() for b in (2, 5, 6, 7)])
        planes = [not keep and 4 * x >= 1 << 24 for x in (m * k, k * n)]
        assert [gao.prog_planes_for(p, b) == 1 for b in (0, 1)] == planes
        assert gao.prog_stats(p)[1]["launches"] == 5 - sum(planes)
        gao.prog_destroy(p)
    for g in got[1:]:
        for a, b in zip(got[0][:3], g[:3]):
            assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
        # the norm: binary64 partials of the same squares, added in another order
        assert abs(got[0][3][0, 0] - g[3][0, 0]) <= 1e-12 * abs(g[3][0, 0])


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
