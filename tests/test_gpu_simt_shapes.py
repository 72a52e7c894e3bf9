"""FP32 SIMT GEMM at the edges of its block tiles (128, 64, 32), of its K steps and chunks, and of
the splits over a cluster: the same bits as the host loop, which sums in the same chunks and
order, for 16-byte aligned rows and any others, and for kchunk values that leave one chunk,
two to eight (split) or more.  The GPU kernel rounds kchunk up to a multiple of 16 (gao_opts),
so the host loop it is compared with is given that multiple."""
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


@pytest.mark.parametrize("M,N,K,kchunk", [
    (1, 1, 1, 0), (32, 32, 32, 0), (33, 31, 30, 0), (64, 96, 255, 0), (256, 256, 256, 0), (257, 260, 264, 0),
    (129, 127, 513, 0), (300, 520, 1000, 0), (513, 640, 1284, 0), (1000, 1000, 1000, 0), (1200, 1001, 777, 0),
    (1300, 1408, 2048, 0), (900, 70, 2305, 0), (40, 2000, 300, 16), (128, 128, 128, 48), (700, 500, 1300, 100),
    (2100, 2050, 320, 0)])
def test_simt_gemm_bits_of_the_host_loop(gao, M, N, K, kchunk):
    bufs = [W.Buffer("A", M, K), W.Buffer("B", K, N), W.Buffer("C0", M, N), W.Buffer("C", M, N, role=W.OUTPUT)]
    loops = [W.Loop(W.INIT, [], [0, 1, 2]), W.Loop(W.GEMM, [0, 1, 2], [3], 1.5, 0.5)]
    out = {}
    for mask, kc in ((0b01, -(-kchunk // 16) * 16), (0b11, kchunk)):
        p = gao.prog_from_workload(W.Program("simt", bufs, loops, M + N + K), kchunk=kc)
        gao.prog_run(p, mask)
        out[mask] = gao.prog_output(p, 3)
        gao.prog_destroy(p)
    assert np.array_equal(out[0b01].view(np.uint32), out[0b11].view(np.uint32))
