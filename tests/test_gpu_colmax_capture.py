"""gao_colmax_noalloc captured after one first call of another shape: every kernel that a shape can
take (strips of three widths, aligned and not, and the keys) runs in the capture and replays, in
a process of its own so that nothing else has loaded them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import torch
import paper_1806_01430_gb300 as gao
X = torch.randn(1 << 22, device="cuda")
q = torch.empty(8192, device="cuda")
s = torch.cuda.Stream()
torch.cuda.synchronize()
assert gao.gao_colmax_noalloc(X.data_ptr(), 64, 64, q.data_ptr(), s) == gao.GAO_OK
s.synchronize()
for r, c in ((65, 63), (300, 2500), (300, 2501), (300, 5000), (300, 5001), (40000, 3)):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="global"):
        assert gao.gao_colmax_noalloc(X.data_ptr(), r, c, q.data_ptr(), s) == gao.GAO_OK
    for _ in range(2):
        q.fill_(-1e9)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(q[:c], X[:r * c].view(r, c).amax(0)), (r, c)
print("captured")
"""


def test_capture_of_other_shapes():
    pytest.importorskip("torch")
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env={**os.environ, "CUDA_MODULE_LOADING": "LAZY", "PYTHONPATH": ROOT})
    assert r.returncode == 0 and "captured" in r.stdout, r.stderr[-2000:]
