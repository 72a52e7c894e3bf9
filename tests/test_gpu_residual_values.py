"""The residual check's binary64 values of the operands, whatever the operand's kind: zeros of
either sign, subnormal and normal numbers at the ends of the range, infinities and NaNs.  With
K = 0 the residual of an M x N matrix C against C0 = null is r = C x and s = y^T C, which numpy
gives exactly when every row (and column) of C has a single nonzero term."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gao():
    from paper_1806_01430_gb300 import _build
    _build.build()
    import paper_1806_01430_gb300 as g
    return g


@pytest.mark.parametrize("n", [5, 64, 259, 1028])
@pytest.mark.parametrize("bits", [0x00000000, 0x80000000, 0x00000001, 0x807FFFFF, 0x00400000, 0x00800000, 0x3F800001,
                                  0xFF7FFFFF, 0x7F800000, 0xFF800000, 0x7FC00000])
def test_operand_values(gao, n, bits):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n)
    C = np.zeros((n, n), dtype=np.float32)
    C[np.arange(n), rng.permutation(n)] = np.array([bits], dtype=np.uint32).view(np.float32)[0]
    x, y = 1.0 + rng.random(n), 1.0 + rng.random(n)
    d = [torch.from_numpy(v).cuda() for v in (C, x, y)]
    scratch = torch.empty(gao.gao_gemm_residual_scratch(n, n, 0), dtype=torch.uint8, device="cuda")
    r, s = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    out = gao.gao_gemm_residual(0, 0, 0, d[0].data_ptr(), n, n, 0, 1.0, 0.0, d[1].data_ptr(), d[2].data_ptr(),
                                scratch.data_ptr(), scratch.numel(), r.data_ptr(), s.data_ptr())
    with np.errstate(invalid="ignore"):
        C64 = C.astype(np.float64)
        want_r, want_s = (C64 * x).sum(axis=1), (C64 * y[:, None]).sum(axis=0)
    assert np.array_equal(r.cpu().numpy(), want_r, equal_nan=True)
    assert np.array_equal(s.cpu().numpy(), want_s, equal_nan=True)
    if np.isfinite(want_r).all():
        assert out["right_argmax"] == int(np.abs(want_r).argmax())
        assert out["left_argmax"] == int(np.abs(want_s).argmax())
