"""lrs_orthonormalize (the QR step of Algorithm 1) against numpy's Householder
QR with the signs of diag(R) made positive."""
import numpy as np
import pytest

import oracle.altgdmin_lrs as O
from tests.gpu_helpers import gpu_available

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r", [(1000, 5), (4096, 10), (17, 16), (300, 1)])
def test_orthonormalize_matches_positive_qr(n, r):
    if not gpu_available():
        pytest.skip("no CUDA device")
    import torch
    from paper_2311_03824_gb300 import lrs as L
    Z = np.random.default_rng(n + r).standard_normal((n, r)).astype(np.float32)
    Zd = torch.from_numpy(Z).cuda()
    Qd = torch.empty_like(Zd)
    L.lrs_orthonormalize(Zd, Qd)
    Q = Qd.cpu().numpy().astype(np.float64)
    Qo, _ = O.qr_positive(Z.astype(np.float64))
    assert np.abs(Q - Qo).max() < 2e-5
    assert np.abs(Q.T @ Q - np.eye(r)).max() < 1e-5


# The cluster kernel's static and dynamic shared memory together pass 48 KB at
# these sizes, the dynamic part alone does not (one size per compiled width).
LIMIT_SIZES = [(47300, 2), (23000, 4), (18000, 5), (11000, 8), (7500, 12), (5500, 16)]


def test_shared_memory_limit_in_a_fresh_process():
    """The limit is a state of the process: no larger call has been before."""
    if not gpu_available():
        pytest.skip("no CUDA device")
    import os
    import subprocess
    import sys
    code = (
        "import torch\n"
        "from paper_2311_03824_gb300 import lrs as L\n"
        f"for n, r in {LIMIT_SIZES}:\n"
        "    g = torch.Generator(device='cuda').manual_seed(n)\n"
        "    Z = torch.randn(n, r, generator=g, device='cuda')\n"
        "    Q = torch.empty_like(Z)\n"
        "    L.lrs_orthonormalize(Z, Q)\n"
        "    Qo, R = torch.linalg.qr(Z.double())\n"
        "    Qo = Qo * torch.diagonal(R).sign()\n"
        "    assert (Q.double() - Qo).abs().max() < 2e-5, (n, r)\n")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    res = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stderr[-2000:]
