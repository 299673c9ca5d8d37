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


def _qr(Z):
    import torch
    from paper_2311_03824_gb300 import lrs as L
    Zd = torch.from_numpy(np.ascontiguousarray(Z, np.float32)).cuda()
    Qd = torch.empty_like(Zd)
    L.lrs_orthonormalize(Zd, Qd)
    return Qd.cpu().numpy().astype(np.float64)


# n below, at and above the cluster kernel's rows and its size (n r = 409600),
# beyond which the separate kernels run; n < 8 r
@pytest.mark.parametrize("cond", [1.0, 20.0, 1e3, 1e5])
@pytest.mark.parametrize("n,r", [(17, 16), (40, 6), (1000, 5), (25600, 16), (25700, 16), (70000, 7)], ids=str)
def test_kernels_and_factors_of_any_condition(n, r, cond):
    """The rows take r float32 products with entries of R^-1 in each pass:
    ||Q - Q_exact||_F <= (r + 2) 2^-24 cond ||Q_exact||_F; Q^T Q - I, which the
    second pass mends, is that of cond = 1."""
    if not gpu_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(n + r)
    Q0, _ = np.linalg.qr(rng.standard_normal((n, r)))
    V, _ = np.linalg.qr(rng.standard_normal((r, r)))
    Z = ((Q0 * np.geomspace(1.0, 1.0 / cond, r)) @ V.T).astype(np.float32)
    Q = _qr(Z)
    Qo, _ = O.qr_positive(Z.astype(np.float64))
    assert np.linalg.norm(Q - Qo) <= (r + 2) * 2.0 ** -24 * cond * np.sqrt(r)
    assert np.abs(Q.T @ Q - np.eye(r)).max() <= (r + 2) * 2.0 ** -24


@pytest.mark.parametrize("e", [-70, 62])
@pytest.mark.parametrize("n,r", [(1000, 5), (300, 16), (70000, 7)], ids=str)
def test_matrices_of_any_scale(n, r, e):
    """Z times 2^e (the Gram's entries leave float32's range) and columns of
    different scales: the same Q."""
    if not gpu_available():
        pytest.skip("no CUDA device")
    Z = np.random.default_rng(n + r).standard_normal((n, r)).astype(np.float32)
    Qo, _ = O.qr_positive(Z.astype(np.float64))
    for Zs in (np.ldexp(Z, e), Z * np.exp2(np.linspace(0, e, r).round()).astype(np.float32)):
        assert np.linalg.norm(_qr(Zs) - Qo) <= 3 * 2.0 ** -24 * np.linalg.norm(Qo)


@pytest.mark.parametrize("n,r", [(1000, 5), (4096, 10), (20000, 3), (50000, 8), (2000, 16)], ids=str)
def test_well_conditioned_rows_are_rounded_once(n, r):
    """A rounding to float32 of entries with log-uniform mantissas is 2^-23 / sqrt(12)
    * 0.74 = 2.5e-8 in the mean square; 10 % for the sample of n r entries."""
    if not gpu_available():
        pytest.skip("no CUDA device")
    Z = np.random.default_rng(n + r).standard_normal((n, r)).astype(np.float32)
    Qo, _ = O.qr_positive(Z.astype(np.float64))
    assert np.linalg.norm(_qr(Z) - Qo) <= 1.1 * 2.0 ** -23 / np.sqrt(12) * 0.74 * np.sqrt(r)
