"""The DFT sweep's branches against the FP64 oracle: supports by columns and term
by term, projections with the basis in its own shared memory, in the frame's
place or in global memory, every rank width, and given supports in any order.

Bars are those of the other parity tests (one GDmin step from the oracle's
iterates).  The order test compares two runs that differ in the order of
float32 sums over the support alone: 1e-5 relative."""
import numpy as np
import pytest

import oracle.altgdmin_lrs as O
from lrsgen import FourierInstance
from tests.gpu_helpers import Problem, check_records, gpu_available, new_fourier_solver, one_step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not gpu_available():
        pytest.skip("no CUDA device")
    from paper_2311_03824_gb300 import build
    build.build()


# fewer samples than two per row; runs of more than four adjacent columns in a
# 256-thread frame; a rank below its width; the basis in the frame's place; in
# global memory (r m pixels do not fit the frame); the widest ranks; tall frames
# that leave no room for the tables
@pytest.mark.parametrize("nx,ny,q,r,m,rho,T", [
    (64, 4, 8, 2, 100, 3, 12), (32, 32, 10, 3, 400, 40, 12), (64, 64, 6, 5, 1300, 20, 12),
    (128, 128, 9, 7, 2300, 60, 4), (128, 128, 10, 8, 3000, 60, 4), (16, 16, 16, 9, 160, 3, 6),
    (20, 20, 24, 13, 260, 3, 6), (2048, 8, 4, 2, 4200, 6, 2), (2048, 8, 4, 3, 4200, 6, 2)])
def test_sweep_one_step(nx, ny, q, r, m, rho, T):
    inst = FourierInstance(nx=nx, ny=ny, q=q, r=r, m=m, rho=rho, seed=50 + nx + r,
                           mask_law="uniform", b_law="gauss")
    _, log = O.run_alg1(O.FourierOperator(inst.masks, nx, ny), inst.Y, r, rho, T,
                        keep=tuple(range(T + 1)), Xstar=inst.Xstar)
    s = new_fourier_solver(inst)
    try:
        recs = one_step(Problem.fourier(inst), s, log, range(T))
    finally:
        s.close()
    check_records(recs, min_whole=T // 2)


@pytest.mark.parametrize("repeat", [False, True])
def test_support_in_any_order(repeat):
    """A state's support may come unsorted, or with a pixel twice (value zero)."""
    inst = FourierInstance(nx=32, ny=32, q=6, r=2, m=400, rho=8, seed=61)
    rng = np.random.default_rng(3)
    outs = []
    for order in (False, True):
        s = new_fourier_solver(inst)
        try:
            s.init()
            s.iterate(3)
            U, B, Si, Sv = s.get()
            Si, Sv = Si.copy(), Sv.copy()
            if repeat:
                Si[:, 1], Sv[:, 1] = Si[:, 0], Sv[:, 0]
            if order:
                for k in range(len(Si)):
                    p = rng.permutation(Si.shape[1])
                    Si[k], Sv[k] = Si[k, p], Sv[k, p]
            from paper_2311_03824_gb300 import lrs as L
            L.lrs_set_state(s.h, np.ascontiguousarray(U.T), np.ascontiguousarray(B.T), Si, Sv, 3,
                            s.progress()[0])
            s.iterate(2)
            outs.append(s.X())
            got = s.get()[2]
            assert (np.diff(got, axis=1) > 0).all()
        finally:
            s.close()
    if not repeat:
        rel = np.linalg.norm(outs[0] - outs[1]) / np.linalg.norm(outs[0])
        assert rel <= 1e-5, rel


@pytest.mark.parametrize("nx,ny,m", [(32, 32, 400), (20, 12, 140), (64, 4, 100)])
def test_given_support_with_repeats_and_entries_outside(nx, ny, m):
    from tests.test_gpu_stream import given_support_steps
    inst = FourierInstance(nx=nx, ny=ny, q=6, r=2, m=m, rho=8, seed=61, mask_law="uniform", b_law="gauss")
    _, log = O.run_alg1(O.FourierOperator(inst.masks, nx, ny), inst.Y, 2, 8, 4, keep=tuple(range(5)), Xstar=inst.Xstar)
    s = new_fourier_solver(inst)
    try:
        recs = given_support_steps(Problem.fourier(inst), s, log, range(1, 4), [-1, nx * ny, 2 ** 31 - 1, -2 ** 31])
    finally:
        s.close()
    check_records(recs, min_whole=2, max_excluded=0.1)

@pytest.mark.parametrize("e", [-40, 40])
def test_measurements_of_any_scale(e):
    """y scaled by a power of two scales B and S and leaves U, whether or not the
    Grams of the initialisation (fourth powers of y) leave float32's range."""
    inst = FourierInstance(nx=16, ny=16, q=24, r=2, m=140, rho=3, seed=63)
    X = []
    for k in (0, e):
        s = new_fourier_solver(inst)
        try:
            f = np.float32(2.0 ** k)
            s.set_measurements(np.ascontiguousarray(inst.Y, np.complex64) * f, np.ascontiguousarray(inst.masks, np.int32))
            s.init()
            s.iterate(10)
            X.append(s.X() / f)
        finally:
            s.close()
    assert np.linalg.norm(X[1] - X[0]) <= 1e-5 * np.linalg.norm(X[0])


def test_cooperative_qr():
    """128 x 128 frames at r = 12: the matrix does not fit one cluster."""
    inst = FourierInstance(nx=128, ny=128, q=14, r=12, m=2500, rho=8, seed=64, mask_law="uniform", b_law="gauss")
    _, log = O.run_alg1(O.FourierOperator(inst.masks, 128, 128), inst.Y, 12, 8, 2, keep=(0, 1, 2), Xstar=inst.Xstar)
    s = new_fourier_solver(inst)
    try:
        recs = one_step(Problem.fourier(inst), s, log, range(2))
    finally:
        s.close()
    check_records(recs, min_whole=1)


@pytest.mark.parametrize("cond", [1.0, 30.0, 1e3, 1e4])
@pytest.mark.parametrize("nx,ny,r", [(20, 20, 4), (64, 64, 6), (64, 64, 16), (4, 4, 7)], ids=str)
def test_rows_of_the_step_are_rounded_once_a_pass(nx, ny, r, cond):
    """A step of length zero is the QR of the state's own U.  One or two passes,
    exact products and at least 45-bit factors leave a rounding to float32 each
    (2^-24 relative per entry, the first one doubled at most by the second
    factor): ||U1 - Q||_F <= 3 * 2^-24 ||Q||_F at any condition whose square the
    factors resolve."""
    from paper_2311_03824_gb300 import lrs as L
    n = nx * ny
    inst = FourierInstance(nx=nx, ny=ny, q=3, r=r, m=n - n // 4, rho=2, seed=65, mask_law="uniform", b_law="gauss")
    rng = np.random.default_rng(r)
    Q0, _ = np.linalg.qr(rng.standard_normal((n, r)) + 1j * rng.standard_normal((n, r)))
    V, _ = np.linalg.qr(rng.standard_normal((r, r)) + 1j * rng.standard_normal((r, r)))
    U = ((Q0 * np.geomspace(1.0, 1.0 / cond, r)) @ V.conj().T).astype(np.complex64)
    s = new_fourier_solver(inst)
    try:
        L.lrs_set_state(s.h, np.ascontiguousarray(U.T), np.zeros((3, r), np.complex64),
                        np.tile(np.arange(2, dtype=np.int32), (3, 1)), np.zeros((3, 2), np.complex64), 1, 1e-30)
        s.iterate(1)
        U1 = s.get()[0].astype(np.complex128)
    finally:
        s.close()
    Q, _ = O.qr_positive(U.astype(np.complex128))
    assert np.linalg.norm(U1 - Q) <= 3 * 2.0 ** -24 * np.sqrt(r), np.linalg.norm(U1 - Q) / np.sqrt(r)


# Errors of B and U after two steps against the FP64 oracle, root mean square over
# three instances, of FP64 r x r solves and the FP64 Cholesky-QR2.  (B where the
# support has two pixels: a larger one's A s takes two rounded twiddles a term.)
FP64_FACTORS = {(64, 64, 24, 4, 1229, 20): (None, 6.28e-8), (32, 32, 60, 6, 400, 8): (None, 5.63e-8),
                (20, 20, 100, 4, 250, 2): (7.08e-8, 6.42e-8)}


@pytest.mark.parametrize("shape", FP64_FACTORS, ids=str)
def test_no_less_precise_than_fp64_factors(shape):
    """At most 1.02 of those errors: the sums of tens of thousands of roundings
    differ by less from one order of the float32 sums to another."""
    from tests.gpu_helpers import cast_state, rel, set_gpu_state
    nx, ny, q, r, m, rho = shape
    n, tot = nx * ny, np.zeros(2)
    for seed in range(3):
        inst = FourierInstance(nx=nx, ny=ny, q=q, r=r, m=m, rho=rho, seed=500 + seed, mask_law="uniform", b_law="gauss")
        P = Problem.fourier(inst)
        rng = np.random.default_rng(seed)
        g = lambda *sh: rng.standard_normal(sh) + 1j * rng.standard_normal(sh)
        U, _ = np.linalg.qr(inst.Ustar + 0.01 * g(n, r) / np.sqrt(n))
        U = U.astype(np.complex64).astype(np.complex128)
        val = (inst.S_val + 0.01 * inst.rms_L * g(q, rho)).astype(np.complex64).astype(np.complex128)
        eta = 0.3 / (m / n * np.linalg.norm(inst.Bstar, 2) ** 2)
        st = O.OracleState(U=U, B=U.conj().T @ inst.Ustar @ inst.Bstar, S=O.densify(inst.S_idx, val, n),
                           S_idx=inst.S_idx.copy(), eta=eta, t=5)
        s = new_fourier_solver(inst)
        try:
            set_gpu_state(s, st, True)
            s.iterate(2)
            U1, B1, Si, Sv = s.get()
        finally:
            s.close()
        ref = cast_state(st, np.complex128)
        for _ in range(2):
            O.iterate_alg1(P.op64, P.Y, ref, rho)
        assert np.array_equal(Si, ref.S_idx)
        tot += np.array([rel(B1, ref.B), rel(U1, ref.U)]) ** 2 / 3
    for err, bar in zip(np.sqrt(tot), FP64_FACTORS[shape]):
        assert bar is None or err <= 1.02 * bar, (err, bar)


def test_ill_conditioned_least_squares():
    """m = r + 1 samples per frame, as for the Gaussian operator: b_k of the frames of
    cond(G_k) > 1e3 within max(1e-5, 10 x the float32 probe's deviation, 2 cond(G_k)
    2^-24) of the FP64 step (the normal equations' float32 bound)."""
    from tests.gpu_helpers import cast_state, probe_step, set_gpu_state, state_of
    inst = FourierInstance(nx=8, ny=8, q=150, r=6, m=7, rho=1, seed=66, mask_law="uniform", b_law="gauss")
    T, P = 4, Problem.fourier(inst)
    _, log = O.run_alg1(O.FourierOperator(inst.masks, 8, 8), inst.Y, 6, 1, T, keep=tuple(range(T + 1)), Xstar=inst.Xstar)
    s = new_fourier_solver(inst)
    checked, worst = 0, 0.0
    try:
        for t in range(1, T):
            st = state_of(log, t, P.n)
            st64, _, dec, _ = probe_step(P, st)
            st32 = cast_state(st, np.complex64)
            O.iterate_alg1(P.op32, P.y32(P.Y), st32, P.rho)
            set_gpu_state(s, st, True)
            s.iterate(1)
            B1 = s.get()[1]
            W = P.op64.AU(st.U)
            cond = np.array([np.linalg.cond(w.conj().T @ w) for w in W])
            for k in np.where((cond > 1e3) & dec)[0]:
                b64 = st64.B[:, k]
                d32 = np.linalg.norm(st32.B[:, k] - b64) / np.linalg.norm(b64)
                dg = np.linalg.norm(B1[:, k] - b64) / np.linalg.norm(b64)
                assert dg <= max(1e-5, 10 * d32, 2 * cond[k] * 2.0 ** -24), (t, k, cond[k], dg, d32)
                checked += 1
                worst = max(worst, cond[k])
    finally:
        s.close()
    assert checked >= 20 and worst > 3e3, (checked, worst)
