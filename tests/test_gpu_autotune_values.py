"""The autotuner's timed launches run the GEMM into C again (adding beta C0 each time where C0 is
C) and, with the chain, D and E: a value that the run before them only reduced still has the
values that its sum and column maxima were formed from."""
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


@pytest.mark.parametrize("prec", [1, 2, 3])
def test_reduced_value_after_autotuning(gao, prec):
    torch = pytest.importorskip("torch")
    n, o, L = 300, W.OUTPUT, W.Loop
    bufs = [W.Buffer(nm, n, n) for nm in ("A", "B", "C", "S", "D", "E", "P")]
    bufs += [W.Buffer("q", 1, n, role=o), W.Buffer("s", 1, 1, W.F64, o)]
    loops = [L(W.INIT, [], [0, 1, 2, 3]), L(W.GEMM, [0, 1, 2], [2], 1.5, 0.5), L(W.AXPY, [2, 3], [4], 2.0),
             L(W.TRANSPOSE, [4], [5]), L(W.SQUARE, [5], [6]), L(W.COLMAX, [6], [7]), L(W.SUM, [6], [8])]
    nbytes = gao.prog_device_bytes(bufs, loops, gemm_prec=prec)
    raw = torch.empty(nbytes + 1024, dtype=torch.uint8, device="cuda")
    arena = raw[-raw.data_ptr() % 1024:][:nbytes]
    torch.cuda.synchronize()
    p = gao.prog_create(bufs, loops, seed=6, gemm_prec=prec, fuse_chains=1, arena=arena)
    gao.prog_run(p, 0b1111111)
    q = gao.prog_output(p, 7).copy()
    gao.prog_autotune(p, pop=2, generations=1)
    off = gao.prog_device_ptr(p, 6) - arena.data_ptr()
    P = arena[off:off + 4 * n * n].view(torch.float32).view(n, n).cpu().numpy()
    assert np.array_equal(P.max(axis=0).view(np.uint32), q.ravel().view(np.uint32))
    gao.prog_destroy(p)
