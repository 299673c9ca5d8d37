"""The streaming engine (the library's choice for Gaussian operators) against
the FP64 oracle, step by step, at the edges of its shapes: rank widths and
their padding, rows that end inside a 16- or 32-row block, one to several
tiles and column chunks, no IHT, supports that fill the column, stored forms;
and bit for bit against itself under another grid, in a batch, as a replayed
graph and column-sharded.  Bars and exclusions as in tests/gpu_helpers.py."""
import numpy as np
import pytest

from lrsgen import GaussianInstance
from tests.gpu_helpers import gpu_available, new_solver
from tests.test_gpu_parity import run_one_step, run_trajectory
from tests.test_gpu_precision import form_one_step
from tests.test_gpu_sharded import run_shards

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not gpu_available():
        pytest.skip("no CUDA device")
    from paper_2311_03824_gb300 import build
    build.build()


def run(inst, T, **opts):
    from paper_2311_03824_gb300 import lrs as L
    s = new_solver(inst, **opts)
    try:
        assert L.lrs_describe(s.h)["engine"] == "stream"
        s.init()
        s.iterate(T)
        return s.get()
    finally:
        s.close()


@pytest.mark.parametrize("n,q,r,m,rho", [
    (40, 30, 1, 20, 1),        # one row block, two tiles, padded rank
    (64, 30, 3, 32, 0),        # no IHT
    (140, 24, 4, 300, 5),      # m > n, several row blocks and pieces
    (257, 30, 7, 97, 4),       # ragged tile, m = 96 + 1, rank 7 in width 8
    (330, 30, 9, 145, 5),      # rank 9 in width 10, 16-row blocks + 1
    (200, 30, 11, 130, 3),
    (300, 24, 16, 160, 3),
    (1100, 16, 5, 150, 40),    # more than 32 support entries, several chunks
], ids=str)
def test_one_step_shapes(n, q, r, m, rho):
    inst = GaussianInstance(n=n, q=q, r=r, m=m, rho=rho, seed=300 + n)
    run_one_step(inst, 10, min_whole=5, max_excluded=0.03)


def test_support_fills_the_column():
    inst = GaussianInstance(n=24, q=1, r=1, m=20, rho=24, seed=300)
    run_one_step(inst, 5, min_whole=5)


def test_trajectory():
    inst = GaussianInstance(n=200, q=200, r=3, m=80, rho=4, seed=1)
    run_trajectory(inst, 120, min_whole=115)


def test_kept_entries_exceed_the_true_support():
    """rho_max > rho: the extra entries are near zero, so their supports keep
    changing and every sweep needs its pass."""
    inst = GaussianInstance(n=200, q=60, r=3, m=90, rho=3, seed=14)
    run_one_step(inst, 16, min_whole=10, rho=8, rho_max=8, max_excluded=0.03)


@pytest.mark.parametrize("a_dtype", [1, 2, 3])
@pytest.mark.parametrize("n,q,r,m,rho", [(200, 48, 3, 80, 4), (230, 32, 8, 150, 6),
                                         (200, 24, 12, 130, 3)], ids=str)
def test_stored_forms(a_dtype, n, q, r, m, rho):
    inst = GaussianInstance(n=n, q=q, r=r, m=m, rho=rho, seed=90 + r)
    form_one_step(inst, a_dtype, 6, min_whole=4)


@pytest.mark.parametrize("a_dtype", [0, 1, 3])
def test_results_do_not_depend_on_the_launch(a_dtype):
    """Another grid, a replayed graph, a batch of uneven problems."""
    import torch
    from paper_2311_03824_gb300 import lrs as L
    insts = [GaussianInstance(n=200, q=60, r=3, m=80, rho=4, seed=61),
             GaussianInstance(n=430, q=32, r=3, m=150, rho=6, seed=62),
             GaussianInstance(n=150, q=50, r=3, m=61, rho=0, seed=63)]
    T = 9
    alone = [run(i, T, a_dtype=a_dtype) for i in insts]
    for i, a in zip(insts, alone):
        for opts in (dict(grid=16), dict(use_graph=1, stream=torch.cuda.Stream())):
            for x, y in zip(a, run(i, T, a_dtype=a_dtype, **opts)):
                assert np.array_equal(x, y)
    ss = [new_solver(i, a_dtype=a_dtype) for i in insts]
    try:
        for s in ss:
            s.init()
        L.lrs_iterate_batch([s.h for s in ss], T)
        for s, a in zip(ss, alone):
            for x, y in zip(a, s.get()):
                assert np.array_equal(x, y)
    finally:
        for s in ss:
            s.close()


def test_two_shards_equal_one_handle_bit_for_bit():
    inst = GaussianInstance(n=200, q=120, r=3, m=80, rho=4, seed=1)
    gb, T = 16, 6
    ranges, shards = run_shards(inst, 2, gb, T)
    s = new_solver(inst, grad_block=gb)
    try:
        s.init()
        s.iterate(T)
        U, B, Si, Sv = s.get()
    finally:
        s.close()
    for (k0, k1), states in zip(ranges, shards):
        Us, Bs, Sis, Svs = states[T]
        assert np.array_equal(Us, U) and np.array_equal(Bs, B[:, k0:k1])
        assert np.array_equal(Sis, Si[k0:k1]) and np.array_equal(Svs, Sv[k0:k1])


def test_autotune_call_keeps_the_iterate():
    from paper_2311_03824_gb300 import lrs as L
    inst = GaussianInstance(n=200, q=40, r=3, m=80, rho=4, seed=15)
    s = new_solver(inst)
    try:
        s.init()
        before = s.get()
        rep = L.lrs_autotune(s.h, 2)
        assert rep["chosen"]["ms"] > 0
        for a, b in zip(before, s.get()):
            assert np.array_equal(a, b)
    finally:
        s.close()


@pytest.mark.parametrize("withhold", [2, 3])
def test_expired_wait_returns_timeout_and_the_device_stays_usable(withhold):
    """Failure detection without a fault: a barrier of the W pass (2), or those of
    the column steps (3), wait for one arrival more than there is.  The waits
    run out after 100 ms, the warp (the CTA, which has other columns to come: two
    CTAs of the streaming grid) leaves, and the call reports LRS_ERR_TIMEOUT.  A solver created afterwards runs normally."""
    from paper_2311_03824_gb300 import lrs as L
    inst = GaussianInstance(n=64, q=40, r=2, m=32, rho=2, seed=7)
    good = run(inst, 4, grid=2)
    s = new_solver(inst, grid=2, wait_ms=100, test_withhold=withhold)
    try:
        assert L.lrs_describe(s.h)["engine"] == "stream"
        with pytest.raises(L.LrsError) as e:
            s.init()
        assert e.value.status == L.LRS_ERR_TIMEOUT, str(e.value)
    finally:
        s.close()
    for x, y in zip(good, run(inst, 4, grid=2)):
        assert np.array_equal(x, y)


def given_support_steps(P, s, log, ts, outside):
    """One step from the oracle's iterates with the support of every odd column
    cut to its first half, in the ways a caller may write that: an index again
    with value zero, a value in two parts, entries outside the column.  Each is
    the step from the dense s_k and the support that HardThreshold gives it."""
    import oracle.altgdmin_lrs as O
    from paper_2311_03824_gb300 import lrs as L
    from tests.gpu_helpers import compare_step, probe_step, state_of
    ct = np.complex64 if P.cplx else np.float32
    recs = []
    for t in ts:
        st = state_of(log, t, P.n)
        Si, rho = st.S_idx.astype(np.int32), st.S_idx.shape[1]
        keep = rho // 2
        for k in range(1, P.q, 2):
            st.S[k, st.S_idx[k, keep:]] = 0
        vals = np.take_along_axis(st.S, st.S_idx, 1).astype(ct)
        st.S = st.S.astype(ct).astype(P.dt)
        for k in range(1, P.q, 2):
            st.S_idx[k] = O.hard_threshold(st.S[k:k + 1], rho)[0][0]
        st64, _, dec, dev = probe_step(P, st)
        for form in ("zero", "split", "outside"):
            I, V = Si.copy(), vals.copy()
            I[1::2, keep:] = outside if form == "outside" else I[1::2, :1]
            V[1::2, keep:] = 7 if form == "outside" else 0
            if form == "split":
                V[1::2, 0] *= 0.5
                V[1::2, -1] = V[1::2, 0]
            L.lrs_set_state(s.h, np.ascontiguousarray(st.U.T, ct), np.ascontiguousarray(st.B.T, ct), I, V,
                            st.t, float(st.eta or 0.0))
            got = s.get()[2]
            assert np.array_equal(np.sort(got, 1), np.sort(st.S_idx, 1)), form
            s.iterate(1)
            recs.append(compare_step(st64, dec, s.get(), dev=dev))
    return recs


@pytest.mark.parametrize("engine", [0, 1, 2, 3])
def test_given_support_with_repeats_and_entries_outside(engine):
    from tests.gpu_helpers import Problem, check_records, oracle_run
    inst = GaussianInstance(n=200, q=40, r=3, m=80, rho=6, seed=71)
    P, (_, log) = Problem.gaussian(inst), oracle_run(inst, 4)
    s = new_solver(inst, engine=engine)
    try:
        recs = given_support_steps(P, s, log, range(1, 4), [-1, 200, 2 ** 31 - 1])
    finally:
        s.close()
    check_records(recs, min_whole=4, max_excluded=0.03)


def test_state_on_the_device_and_unsorted():
    """Device arrays take the same way; entries in another order are the same
    support, and the output is ascending."""
    import torch
    from paper_2311_03824_gb300 import lrs as L
    inst = GaussianInstance(n=1100, q=9, r=2, m=90, rho=40, seed=72)
    outs = []
    for how in ("host", "device", "unsorted"):
        s = new_solver(inst)
        try:
            s.init()
            U, B, Si, Sv = s.get()
            a = [np.ascontiguousarray(U.T), np.ascontiguousarray(B.T), Si.copy(), Sv.copy()]
            if how == "unsorted":
                p = np.random.default_rng(1).permutation(40)
                a[2], a[3] = np.ascontiguousarray(a[2][:, p]), np.ascontiguousarray(a[3][:, p])
            if how == "device":
                a = [torch.from_numpy(x).cuda() for x in a]
            L.lrs_set_state(s.h, *a, 1, 1e-3)
            s.iterate(2)
            outs.append(s.get())
        finally:
            s.close()
    for x, y, z in zip(*outs):
        assert np.array_equal(x, y)
        assert np.allclose(x, z, rtol=1e-4, atol=1e-5 * np.abs(x).max())
    assert (np.diff(outs[2][2], axis=1) > 0).all()


# The failure conventions and the ill-conditioned least squares of the other
# engines' tests, on the library's choice.

@pytest.mark.parametrize("name", ["test_out_of_order_calls_return_state_error_and_change_nothing",
                                  "test_rank_deficient_column_reports_numerical_error_with_column"])
def test_errors(name):
    import tests.test_gpu_errors as E
    getattr(E, name)(0)


def test_ill_conditioned_least_squares_of_the_default_engine():
    from tests.test_gpu_parity import test_ill_conditioned_least_squares
    test_ill_conditioned_least_squares(0)


def test_batch_of_handles_of_two_engines():
    """Handles of different engines share no launch; each ends as it would alone."""
    from paper_2311_03824_gb300 import lrs as L
    inst = GaussianInstance(n=120, q=20, r=2, m=50, rho=3, seed=73)
    outs = []
    for batch in (False, True):
        ss = [new_solver(inst), new_solver(inst, engine=2)]
        try:
            for s in ss:
                s.init()
            if batch:
                L.lrs_iterate_batch([s.h for s in ss], 4)
            else:
                for s in ss:
                    s.iterate(4)
            outs.append([x for s in ss for x in s.get()])
        finally:
            for s in ss:
                s.close()
    for x, y in zip(*outs):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("a_exp", [-40, 40])
def test_measurements_of_any_scale(a_exp):
    """y scaled by a power of two scales B and S and leaves U: no sum of the path
    (the fourth powers of the initialisation's Grams least of all) leaves
    float32's range."""
    inst = GaussianInstance(n=120, q=40, r=3, m=60, rho=3, seed=74)
    X = []
    for e in (0, a_exp):
        s = new_solver(inst)
        try:
            s.set_measurements(np.ldexp(np.ascontiguousarray(inst.Y, np.float32), e),
                               np.ascontiguousarray(inst.A, np.float32))
            s.init()
            s.iterate(20)
            X.append(np.ldexp(s.X(), -e))
        finally:
            s.close()
    assert np.linalg.norm(X[1] - X[0]) <= 1e-5 * np.linalg.norm(X[0])


# (least squares, support sums and the step's QR by exact products and FP64 or
# double-float r x r factors, as the task engine has them)
@pytest.mark.parametrize("n,q,r,m,rho,err", [(2000, 16, 4, 600, 400, 1e-3), (1200, 40, 3, 300, 8, 1e-2),
                                             (400, 200, 6, 150, 6, 0.05), (96, 64, 4, 900, 5, 1e-2)], ids=str)
def test_no_less_precise_than_the_task_engine(n, q, r, m, rho, err):
    """Two steps from one state, B, S and U against the FP64 oracle: the error is
    at most 1.15 of the task engine's (the spread of a norm over a few hundred
    rounding errors, seen on reruns with other instances)."""
    import oracle.altgdmin_lrs as O
    from tests.gpu_helpers import Problem, cast_state, rel, set_gpu_state
    tot = {0: np.zeros(3), 2: np.zeros(3)}
    for seed in range(3):
        inst = GaussianInstance(n=n, q=q, r=r, m=m, rho=rho, seed=400 + seed)
        P = Problem.gaussian(inst)
        rng = np.random.default_rng(seed)
        U, _ = np.linalg.qr(inst.Ustar + err * rng.standard_normal((n, r)) / np.sqrt(n))
        U = U.astype(np.float32).astype(np.float64)
        val = inst.S_val + err * inst.rms_L * rng.standard_normal((q, rho))
        eta = 0.3 / (m * np.linalg.norm(inst.Bstar, 2) ** 2)
        st = O.OracleState(U=U, B=U.T @ inst.Ustar @ inst.Bstar,
                           S=O.densify(inst.S_idx, val.astype(np.float32).astype(np.float64), n),
                           S_idx=inst.S_idx.copy(), eta=eta, t=5)
        for eng in (0, 2):
            s = new_solver(inst, engine=eng)
            try:
                set_gpu_state(s, st, False)
                s.iterate(2)
                g = s.get()
            finally:
                s.close()
            if eng == 0:
                ref = cast_state(st, np.float64)
                for _ in range(2):
                    O.iterate_alg1(P.op64, P.Y, ref, rho)
                Rv = np.take_along_axis(ref.S, ref.S_idx, 1)
            assert np.array_equal(g[2], ref.S_idx)
            tot[eng] += np.array([rel(g[1], ref.B), rel(g[3], Rv), rel(g[0], ref.U)]) ** 2
    print("B S U", np.sqrt(tot[0] / 3), np.sqrt(tot[2] / 3))
    assert (np.sqrt(tot[0]) <= 1.15 * np.sqrt(tot[2])).all(), (np.sqrt(tot[0] / 3), np.sqrt(tot[2] / 3))


def test_task_engine_where_the_streaming_scratch_does_not_fit():
    """rho = n: the support's columns are as large as A_k (1.07 GB).  With 1.9 GB
    free the task engine takes the problem; with memory to spare, streaming."""
    import torch
    from paper_2311_03824_gb300 import Solver
    from paper_2311_03824_gb300 import lrs as L
    engines, keep = [], None
    for room in (None, 1900 << 20):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        if room:
            keep = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
        s = Solver(2048, 512, 256, 4, 2048)
        try:
            engines.append(L.lrs_describe(s.h)["engine"])
        finally:
            s.close()
    del keep
    torch.cuda.empty_cache()
    assert engines == ["stream", "task"]
