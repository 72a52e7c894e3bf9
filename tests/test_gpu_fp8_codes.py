"""FP8 quantisation at the edges of its 128-element blocks, 64-column groups and 128-row tiles:
multiplied by the identity, each operand comes back as the e4m3 codes of its blocks' scaling
formed here in numpy, exactly -- ragged rows and columns, empty blocks, values that
round to even, flush to zero or lie above the largest significand."""
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


def e4m3(X):
    """Rows of X in 128-element blocks, each scaled by the power of two that puts its largest
    magnitude at 448 or less, rounded to e4m3."""
    M, K = X.shape
    P = np.zeros((M, -(-K // 128) * 128))
    P[:, :K] = X
    blk = P.reshape(M, -1, 128)
    amax = np.abs(blk).max(axis=2, keepdims=True)
    f, e = np.frexp(np.where(amax > 0, amax, 1.0))  # amax = f 2^e, f in [0.5, 1)
    e = e - 1 - 8 + (2 * f > 1.75)
    y = np.ldexp(blk, -e)
    step = np.ldexp(1.0, np.maximum(np.frexp(y)[1] - 1, -6) - 3)
    q = np.clip(np.round(y / step) * step, -448, 448)
    return np.where(amax > 0, np.ldexp(q, e), 0.0).reshape(M, -1)[:, :K]


@pytest.mark.parametrize("m,k", [(1, 1), (5, 129), (130, 64), (129, 200), (300, 385), (257, 512), (1000, 127), (63, 1028)])
def test_codes_of_both_operands(gao, m, k):
    rng = np.random.default_rng(m * 31 + k)
    X = np.ldexp(rng.standard_normal((m, k)), rng.integers(-12, 3, (m, k)))
    X *= np.ldexp(1.0, rng.integers(-20, 21, (m, 1)))
    X[rng.random((m, k)) < 0.1] = 0.0
    X[m // 2, : min(k, 128)] = 0.0                                   # an empty block
    X[0, 0] = 448.0                                                 # the largest code, then halfway cases
    if k > 3:
        X[0, 1:4] = [17.0, 19.0, 2.0 ** -10]
    if m > 2:
        X[2, 0] = np.float32(np.abs(X[2]).max() * 1.9 + 1e-3)        # a significand above 1.75
    X = X.astype(np.float32)
    want = e4m3(X.astype(np.float64)).astype(np.float32)
    for A, B in ((X, np.eye(k, dtype=np.float32)), (np.eye(k, dtype=np.float32), np.ascontiguousarray(X.T))):
        (M, K), N = A.shape, B.shape[1]
        bufs = [W.Buffer("A", M, K, role=W.INPUT), W.Buffer("B", K, N, role=W.INPUT),
                W.Buffer("C0", M, N, role=W.INPUT), W.Buffer("C", M, N, role=W.OUTPUT)]
        p = gao.prog_create(bufs, [W.Loop(W.GEMM, [0, 1, 2], [3], 1.0, 1.0)], gemm_prec=gao.FP8)
        for i, x in enumerate((A, B, np.zeros((M, N), np.float32))):
            gao.prog_set_input(p, i, x)
        gao.prog_run(p, 1)
        C = gao.prog_output(p, 3)
        assert np.array_equal(C if A is X else C.T, want)
        gao.prog_destroy(p)


@pytest.mark.parametrize("rowscale", [0, 3])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (5, 63, 129), (130, 64, 127), (129, 201, 256), (300, 65, 385), (257, 1001, 1030)])
def test_codes_formed_by_the_init_loop(gao, m, n, k, rowscale):
    """A and B formed straight as codes (TEMP) against INIT then quantisation (kept as OUTPUT), with
    and without rows scaled: the same bits of C."""
    got = []
    for keep in (False, True):
        role = W.OUTPUT if keep else W.TEMP
        bufs = [W.Buffer("A", m, k, role=role), W.Buffer("B", k, n, role=role), W.Buffer("C0", m, n),
                W.Buffer("C", m, n, role=W.OUTPUT)]
        loops = [W.Loop(W.INIT, [], [0, 1, 2], flags=rowscale), W.Loop(W.GEMM, [0, 1, 2], [3], 1.5, 0.5)]
        p = gao.prog_create(bufs, loops, seed=m + n + k, gemm_prec=gao.FP8)
        for _ in range(3):  # plain, captured, replayed
            gao.prog_run(p, 0b11)
            got.append(gao.prog_output(p, 3))
            assert [gao.prog_planes_for(p, b) for b in (0, 1)] == ([-1, -1] if keep else [1, 1])
            assert gao.prog_stats(p)[1]["launches"] == (3 if keep else 1)
        gao.prog_destroy(p)
    for c in got:
        assert np.array_equal(c.view(np.uint32), got[-1].view(np.uint32))
