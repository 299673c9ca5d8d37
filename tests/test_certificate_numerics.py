"""The bound that lets a Gaussian IHT sweep keep its support without a pass over
A_k, checked on the CPU in numpy (no GPU): after a pass at u_ref the float32 sums
g_j = a_j^T u_ref may be off by their own rounding, at most (m + 4) 2^-24 ||a_j||
||u_ref||, which is no share of |g_j|.  Every row group's large term swallows the
small ones that follow and the large ones cancel, so that float32 returns g_j = 0
where it is about 1e-4 ||a_j|| ||u_ref||."""
import numpy as np
import pytest


def pass_sum(a, u):
    """a^T u as the pass sums it: row group o (rows 4 o + s of every 16) in one
    chain of fused multiply-adds, the four groups in two shuffles."""
    acc = np.zeros(4, np.float32)
    for t in range(0, len(a), 16):
        for s in range(4):
            i = t + 4 * np.arange(4) + s
            acc = (acc.astype(np.float64) + a[i].astype(np.float64) * u[i].astype(np.float64)).astype(np.float32)
    acc = acc[[0, 1]] + acc[[2, 3]]
    return np.float32(acc[0] + acc[1])


@pytest.mark.parametrize("m", [160, 2048, 8192])
def test_bound_after_a_pass_holds_where_its_sums_cancel(m):
    a = np.full(m, 2.0 ** -13, np.float32)
    u = a.copy()
    a[[0, 4, 8, 12]] = 1
    u[[0, 4, 8, 12]] = [1, 1, -1, -1]
    exact = abs(float(a.astype(np.float64) @ u.astype(np.float64)))
    g = abs(float(pass_sum(a, u)))
    na, nu = float(np.linalg.norm(a)), float(np.linalg.norm(u))
    assert 1.001 * g < exact                             # the pass's value is no bound
    assert 1.001 * (g + na * (m + 4) * 2.0 ** -24 * nu) >= exact
