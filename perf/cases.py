"""The work that a user of the solver has it do, as cases to time: GDmin
iterations of both operators from states that a solve passes through, whole
solves, a batch of requests, and the QR step alone.

Sizes are those of this repository's benchmark, tests and serving mix:
n = q = 200 (parity), n = q = 1000 (headline), n = 4096 q = 2048 (large
operator), 128 x 128 and 64 x 64 DFT frames, 20 x 20 frames of the paper's
Table 1, and the serving mix's ranges (n 256..4096, q 64..1024, r 2..10,
m/n 0.15..0.4, rho/n 0.01..0.02, A_k in BF16).

An iteration case starts from a state at distance `err` from the solution:
err 0.1 is early in a solve (supports still change, some are wrong), 1e-2 to
1e-4 the middle, 1e-6 the float32 floor where the default T = 200 spends most
of its iterations.
"""
import math

import torch

from paper_2311_03824_gb300 import Solver
from paper_2311_03824_gb300 import lrs as L

GAUSS, DFT = L.LRS_OP_GAUSSIAN, L.LRS_OP_DFT2D_MASK
TAU, TAU0 = 3, 10          # IHT sweeps per iteration and in the initialisation
C_ETA = 0.14               # step size rule of the whole solves
REFINE = 8                 # iterations between defect corrections of stored forms


def listed():
    return [
        # the QR step alone (lrs_orthonormalize), the smallest call: launches and latency
        dict(name="qr_n1000", kind="qr", n=1000, r=5),
        # parity-size problem near convergence: launch-bound iterations
        dict(name="gauss_n200_late", kind="gauss", n=200, q=200, r=3, m=80, rho=4, a_dtype=0,
             err=1e-6, iters=16),
        # the headline problem early in a solve: supports still change
        dict(name="gauss_n1000_early", kind="gauss", n=1000, q=1000, r=5, m=150, rho=10,
             a_dtype=0, err=0.1, iters=4),
        # the same near convergence, where most of the iterations of a solve are
        dict(name="gauss_n1000_late", kind="gauss", n=1000, q=1000, r=5, m=150, rho=10,
             a_dtype=0, err=1e-5, iters=8),
        # ragged sizes (no multiple of 32, odd m) in the middle of a solve
        dict(name="gauss_ragged", kind="gauss", n=1537, q=301, r=7, m=333, rho=23, a_dtype=0,
             err=1e-2, iters=4),
        # a large request of the serving mix, A_k stored in BF16, with its defect correction
        dict(name="gauss_n2048_bf16", kind="gauss", n=2048, q=512, r=8, m=563, rho=31, a_dtype=1,
             err=1e-3, iters=8),
        # the large operator (17 GB of A_k)
        dict(name="gauss_n4096", kind="gauss", n=4096, q=2048, r=10, m=512, rho=40, a_dtype=0,
             err=1e-3, iters=2),
        # 128 x 128 DFT frames (dynamic MRI), the second headline
        dict(name="dft_128x128", kind="dft", nx=128, ny=128, q=256, r=6, m=2048, rho=82,
             err=2e-2, iters=4),
        # 64 x 64 frames of the serving mix, ragged q and m
        dict(name="dft_64x64", kind="dft", nx=64, ny=64, q=99, r=4, m=1229, rho=61, err=1e-2,
             iters=4),
        # a whole solve from measurements to X: set-up, initialisation, 40 iterations
        dict(name="solve_n1000", kind="solve", n=1000, q=1000, r=5, m=150, rho=10, iters=40),
        # a whole solve of 20 x 20 DFT frames (the paper's Fourier experiment's shape)
        dict(name="solve_dft_20x20", kind="solve_dft", nx=20, ny=20, q=400, r=4, m=250, rho=2,
             iters=60),
        # requests of the serving mix that the server runs together
        dict(name="batch_serving", kind="batch", count=6, n=448, q=112, r=4, m=120, rho=7,
             a_dtype=1, err=1e-3, iters=8),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["gauss"] * 6 + ["dft"] * 3 + ["qr", "batch"])
    err = float("%.2g" % _log(rng, 1e-6, 0.05))
    if kind == "qr":
        return dict(kind=kind, n=int(_log(rng, 200, 65536)), r=rng.randint(2, 16))
    if kind == "batch":
        n = int(_log(rng, 200, 1000))
        return dict(kind=kind, count=rng.randint(2, 8), n=n, q=int(_log(rng, 64, 200)),
                    r=rng.randint(2, 10), m=int(rng.uniform(0.25, 0.4) * n),
                    rho=max(1, int(rng.uniform(0.01, 0.02) * n)), a_dtype=rng.choice([0, 1]),
                    err=min(err, 1e-2), iters=rng.choice([4, 8]))
    if kind == "dft":
        nx = rng.choice([16, 32, 64, 64, 128, 128, 20, 36])
        ny = nx if nx in (20, 36) else rng.choice([nx, nx // 2])
        n = nx * ny
        return dict(kind=kind, nx=nx, ny=ny, q=int(_log(rng, 48, 300)), r=rng.randint(2, 8),
                    m=int(rng.uniform(0.2, 0.4) * n),
                    rho=max(1, int(rng.uniform(0.004, 0.015) * n)), err=min(err, 2e-2),
                    iters=rng.randint(2, 4))
    n = int(_log(rng, 200, 4096))
    q = int(_log(rng, 64, 1100))
    m = max(60, int(rng.uniform(0.15, 0.4) * n))
    # at most 4 GB of float32 A_k
    q = max(48, min(q, int(1e9 / (m * n))))
    return dict(kind=kind, n=n, q=q, r=rng.randint(2, 10), m=m,
                rho=max(1, int(rng.uniform(0.01, 0.02) * n)),
                a_dtype=rng.choice([0, 0, 0, 1, 1, 2, 3]), err=err, iters=rng.choice([2, 4, 8]))


# ------------------------------------------------------------------ inputs --

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _orth(Z):
    """Q factor with a positive real diagonal of R."""
    Q, R = torch.linalg.qr(Z)
    d = torch.diagonal(R)
    return Q * (d / d.abs()).conj()


def _randn(g, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=g, device="cuda", dtype=dtype)


def _sparse(g, q, n, rho, rms, blobs=None):
    """rho distinct ascending indices per column and magnitudes U[1, 10] rms."""
    if blobs is None:
        idx = torch.rand(q, n, generator=g, device="cuda").topk(rho, dim=1).indices
    else:                                   # 3 x 3 blobs of pixels, the most central first
        nx, ny = blobs
        near = torch.rand(q, 1, nx, ny, generator=g, device="cuda")
        near = near.masked_fill(near < 1 - 1.5 * max(1, rho / 9) / n, 0)
        near = torch.nn.functional.max_pool2d(near, 3, 1, 1).reshape(q, n)
        near = near + 1e-3 * torch.rand(q, n, generator=g, device="cuda")
        idx = near.topk(rho, dim=1).indices
    mag = (1 + 9 * torch.rand(q, rho, generator=g, device="cuda", dtype=torch.float64)) * rms
    return idx.sort(dim=1).values, mag


def _gauss_problem(case, g):
    n, q, r, m, rho = (case[k] for k in ("n", "q", "r", "m", "rho"))
    U = _orth(_randn(g, n, r, dtype=torch.float64))
    B = _randn(g, r, q, dtype=torch.float64)
    rms = float((U @ B).square().mean().sqrt())
    idx, mag = _sparse(g, q, n, rho, rms)
    val = mag * torch.where(torch.rand(q, rho, generator=g, device="cuda") < 0.5, -1.0, 1.0)
    X = (U @ B).T.contiguous()
    X.scatter_add_(1, idx, val)
    A = _randn(g, q, m, n)
    Y = torch.empty(q, m, device="cuda")
    for k0, Ak in _chunks(A):
        Y[k0:k0 + len(Ak)] = torch.bmm(Ak, X[k0:k0 + len(Ak)].unsqueeze(2)).squeeze(2).float()
    return A, Y, U, B, idx, val, rms


def _masks(g, q, nx, ny, m, uniform):
    """Kept DFT rows per frame, ascending: the centre of k-space and, with
    weight (1 + k_r / 8)^-2, the rest (or uniformly random rows)."""
    n = nx * ny
    u = torch.rand(q, n, generator=g, device="cuda", dtype=torch.float64).clamp_min(1e-300)
    if uniform:
        key = u
    else:
        kx = torch.arange(nx, device="cuda")
        ky = torch.arange(ny, device="cuda")
        dx = torch.where(kx < nx - nx // 2, kx, kx - nx)[:, None].double()
        dy = torch.where(ky < ny - ny // 2, ky, ky - ny)[None, :].double()
        c = 8 if n >= 16384 else 4
        kr = (dx * dx + dy * dy).sqrt()
        key = u.log() * ((1 + kr / 8) ** 2).reshape(1, n)
        key = key.masked_fill(((dx.abs() < c) & (dy.abs() < c)).reshape(1, n), 1.0)
    return key.topk(m, dim=1).indices.sort(dim=1).values.to(torch.int32)


def _dft_problem(case, g):
    nx, ny, q, r, m, rho = (case[k] for k in ("nx", "ny", "q", "r", "m", "rho"))
    n, table1 = nx * ny, case["kind"] == "solve_dft"
    U = _orth(_randn(g, n, r, dtype=torch.complex128))
    if table1:
        B = _randn(g, r, q, dtype=torch.float64).to(torch.complex128)
    else:                                   # a smooth temporal basis with decaying weights
        j = torch.arange(r, device="cuda", dtype=torch.float64)[:, None]
        k = torch.arange(q, device="cuda", dtype=torch.float64)[None, :]
        B = (2.0 ** (-j / 2) * torch.cos(math.pi * j * (k + 0.5) / q)).to(torch.complex128)
        B = B / (U @ B).abs().square().mean().sqrt()
    rms = float((U @ B).abs().square().mean().sqrt())
    idx, mag = _sparse(g, q, n, rho, rms, None if table1 else (nx, ny))
    ph = 2 * math.pi * torch.rand(q, rho, generator=g, device="cuda", dtype=torch.float64)
    val = torch.polar(mag, ph)
    X = (U @ B).T.contiguous()
    X.scatter_add_(1, idx, val)
    mask = _masks(g, q, nx, ny, m, table1)
    Y = _dft_fwd(X, mask, nx, ny).to(torch.complex64)
    return mask, Y, U, B, idx, val, rms


def _state(case, g, U, B, idx, val, rms, n):
    """A state at relative distance err from the solution: U turned, S's values
    off, and for err >= 1e-2 one entry of the support wrong in a tenth of the
    columns."""
    err, q, rho = case["err"], B.shape[1], idx.shape[1]
    dt = U.dtype
    U1 = _orth(U + err * _randn(g, *U.shape, dtype=dt) / math.sqrt(n))
    B1 = U1.conj().T @ (U @ B)
    val1 = val + err * rms * _randn(g, q, rho, dtype=dt)
    idx1 = idx.clone()
    if err >= 1e-2:
        k = torch.nonzero(torch.rand(q, generator=g, device="cuda") < 0.1).squeeze(1)
        new = (idx1[k, 0] + 1 + torch.randint(n - 1, (len(k),), generator=g, device="cuda")) % n
        clash = (idx1[k] == new[:, None]).any(1)
        idx1[k, 0] = torch.where(clash, idx1[k, 0], new)
        val1[k, 0] = torch.where(clash, val1[k, 0], 0.5 * rms)
        idx1, o = idx1.sort(dim=1)
        val1 = val1.gather(1, o)
    f = torch.complex64 if dt.is_complex else torch.float32
    return (U1.T.to(f).contiguous(), B1.T.to(f).contiguous(), idx1.to(torch.int32).contiguous(),
            val1.to(f).contiguous())


def _eta(case, B):
    s2 = float(torch.linalg.matrix_norm(B, 2)) ** 2
    m_eff = case["m"] if "n" in case else case["m"] / (case["nx"] * case["ny"])
    return 0.3 / (m_eff * s2)


def _problem(case, seed):
    """(operator, measurements, solution parts, start state, eta) of one case."""
    g = _gen(seed)
    dft = case["kind"] in ("dft", "solve_dft")
    n = case["nx"] * case["ny"] if dft else case["n"]
    A, Y, U, B, idx, val, rms = (_dft_problem if dft else _gauss_problem)(case, g)
    st = _state(case, g, U, B, idx, val, rms, n) if "err" in case else None
    return A, Y, st, _eta(case, B)


def _members(case):
    """The problems of a batch: sizes around the case's."""
    return [dict(case, n=case["n"] + case["n"] * i // 8, m=case["m"] + case["m"] * i // 8,
                 q=case["q"] + 16 * (i % 3)) for i in range(case["count"])]


# ------------------------------------------------------------- the program --

def _solver(case, stream):
    if "nx" in case:
        return Solver(case["nx"] * case["ny"], case["m"], case["q"], case["r"], case["rho"], DFT,
                      nx=case["nx"], ny=case["ny"], stream=stream, use_graph=1)
    return Solver(case["n"], case["m"], case["q"], case["r"], case["rho"], GAUSS, stream=stream,
                  use_graph=1, a_dtype=case.get("a_dtype", 0), refine_every=REFINE)


def _member_state(case, seed, stream):
    A, Y, st, eta = _problem(case, seed)
    torch.cuda.synchronize()               # the inputs are complete on every stream
    s = _solver(case, stream)
    s.set_measurements(Y, A)
    out = tuple(torch.empty_like(t) for t in st)
    return dict(s=s, st=st, eta=eta, out=out)


def prepare(case, seed):
    if case["kind"] == "qr":
        Z = _randn(_gen(seed), case["n"], case["r"])
        return dict(kind="qr", Z=Z, Q=torch.empty_like(Z))
    stream = torch.cuda.Stream()
    if case["kind"] in ("solve", "solve_dft"):
        A, Y, _, _ = _problem(case, seed)
        n = A.shape[2] if case["kind"] == "solve" else case["nx"] * case["ny"]
        q, rho = case["q"], case["rho"]
        X = torch.empty(q, n, dtype=Y.dtype, device="cuda")
        Si = torch.empty(q, rho, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        return dict(kind="solve", s=_solver(case, stream), A=A, Y=Y, X=X, Si=Si,
                    iters=case["iters"])
    if case["kind"] == "batch":
        ms = [_member_state(c, 1000 * seed + i, stream) for i, c in enumerate(_members(case))]
        return dict(kind="batch", members=ms, iters=case["iters"])
    return dict(_member_state(case, seed, stream), kind="iterate", iters=case["iters"])


def _begin(d):
    U, B, Si, Sv = d["st"]
    L.lrs_set_state(d["s"].h, U, B, Si, Sv, 5, d["eta"])


def _end(d):
    U, B, Si, Sv = d["out"]
    L.lrs_get(d["s"].h, U, B, Si, Sv)
    return dict(U=U, B=B, S_idx=Si, S_val=Sv)


def run(state):
    if state["kind"] == "qr":
        L.lrs_orthonormalize(state["Z"], state["Q"])
        return state["Q"]
    if state["kind"] == "solve":
        s = state["s"]
        s.set_measurements(state["Y"], state["A"])
        s.init()
        s.iterate(state["iters"])
        L.lrs_get_x(s.h, state["X"])
        L.lrs_get(s.h, S_idx=state["Si"])
        return dict(X=state["X"], S_idx=state["Si"])
    if state["kind"] == "batch":
        for d in state["members"]:
            _begin(d)
        L.lrs_iterate_batch([d["s"].h for d in state["members"]], state["iters"])
        return [_end(d) for d in state["members"]]
    _begin(state)
    state["s"].iterate(state["iters"])
    return _end(state)


def work(case):
    if case["kind"] == "qr":
        n, r = case["n"], case["r"]
        return {"bytes": 8 * n * r, "flops": 4 * n * r * r}
    if case["kind"] == "batch":
        ws = [work(dict(c, kind="gauss")) for c in _members(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    q, r, m, rho, T = (case[k] for k in ("q", "r", "m", "rho", "iters"))
    if "nx" in case:
        # per iteration and frame: y and the mask, s in and out, b; A^H u and the gradient by FFT,
        # A s and A g_G at the m samples, W = (F U) at the samples and its Gram
        n = case["nx"] * case["ny"]
        fft = 5 * n * math.log2(n)
        b = q * (12 * m + 24 * rho + 8 * r) + 24 * n * r
        f = q * (TAU * fft + (TAU + 1) * 8 * m * rho + 8 * m * r * (r + 3)) + 2 * r * fft
    else:
        # per iteration: every A_k once; W = A_k U and tau + 1 products A_k^T v
        n, eb = case["n"], {0: 4, 1: 2, 2: 1, 3: 2}[case.get("a_dtype", 0)]
        b = q * (eb * m * n + 4 * m + 12 * rho + 4 * r) + 12 * n * r
        f = q * 2 * m * n * (r + TAU + 1)
    w = {"bytes": T * b, "flops": T * f}
    if case.get("a_dtype", 0):             # the defect correction reads the float32 operator
        w["bytes"] += -(-T // REFINE) * 4 * q * m * n
    if case["kind"].startswith("solve"):
        w["bytes"] += 2 * 4 * q * m * n if "n" in case else 0   # in, and into the solver's layout
        w["flops"] += q * 2 * m * n * (TAU0 + 2) if "n" in case else 0
    return w


# ---------------------------------------------- the same in 64 bits (torch) --

def _chunks(A):
    """(first column, float64 A_k) in pieces of at most 2 GB."""
    c = max(1, int(2.5e8 / (A.shape[1] * A.shape[2])))
    for k0 in range(0, A.shape[0], c):
        yield k0, A[k0:k0 + c].double()


def _stored(A, form):
    """The operator as its stored form holds it (float32 values)."""
    if form == 0:
        return A
    if form == 1:
        return A.bfloat16().float()
    e4 = torch.float8_e4m3fn
    s1 = (A.abs().amax(2, keepdim=True) / 448).clamp_min(1e-38)
    hi = (A / s1).to(e4).float()
    if form == 2:
        return hi * s1
    rest = (A.double() - hi.double() * s1.double()).float()
    s2 = (rest.abs().amax(2, keepdim=True) / 448).clamp_min(1e-38)
    return (hi.double() * s1.double() + (rest / s2).to(e4).double() * s2.double()).float()


class _Gauss:
    """A_k x and A_k^T u of a run of columns, A float64 (c, m, n)."""

    def __init__(self, A):
        self.A = A

    def fwd(self, x):
        return torch.bmm(self.A, x.unsqueeze(2)).squeeze(2)

    def adj(self, u):
        return torch.bmm(u.unsqueeze(1), self.A).squeeze(1)

    def W(self, U):
        return self.A @ U


def _dft_fwd(X, mask, nx, ny):
    F = torch.fft.fft2(X.reshape(-1, nx, ny), norm="ortho").reshape(len(X), nx * ny)
    return F.gather(1, mask.long())


class _Dft:
    def __init__(self, mask, nx, ny):
        self.mask, self.nx, self.ny = mask.long(), nx, ny

    def fwd(self, x):
        return _dft_fwd(x, self.mask, self.nx, self.ny)

    def adj(self, u):
        n = self.nx * self.ny
        K = torch.zeros(len(u), n, dtype=u.dtype, device=u.device).scatter_(1, self.mask, u)
        return torch.fft.ifft2(K.reshape(-1, self.nx, self.ny), norm="ortho").reshape(-1, n)

    def W(self, U):
        F = torch.fft.fft2(U.T.reshape(-1, self.nx, self.ny), norm="ortho").reshape(U.shape[1], -1)
        return F.T[self.mask]


def _sq(v):
    return (v.abs() ** 2).sum(1)


def _top(v, rho):
    """Indicator of the rho entries of largest modulus of each row."""
    return torch.zeros_like(v.real).scatter_(1, v.abs().topk(rho, dim=1).indices, 1.0)


def _iht(op, y, s, G, rho, sweeps, W=None, Gi=None):
    """Normalised IHT (Algorithm 2) on P y, P A with P the projector off range(W)."""
    def P(v):
        if W is None:
            return v
        c = Gi @ (W.mH @ v.unsqueeze(2))
        return v - (W @ c).squeeze(2)
    for _ in range(sweeps):
        g = op.adj(P(op.fwd(s) - y))
        if G is None:
            G = _top(g, rho)
        gG = g * G
        den = _sq(P(op.fwd(gG)))
        mu = torch.where(den > 0, _sq(gG) / den.clamp_min(1e-300), torch.zeros_like(den))
        v = s - mu[:, None] * g
        G = _top(v, rho)
        s = v * G
    return s, G


def _sweep(op, y, U, s, G, rho):
    """One column sweep: s, its support, b and the gradient's column A^T e."""
    W = op.W(U)
    Gi = torch.linalg.inv(W.mH @ W)
    s, G = _iht(op, y, s, G, rho, TAU, W, Gi)
    res = y - op.fwd(s)
    b = (Gi @ (W.mH @ res.unsqueeze(2))).squeeze(2)
    return s, G, b, op.adj((W @ b.unsqueeze(2)).squeeze(2) - res)


def _iterate64(ops, y, U, s, G, b, rho, eta, iters, fix=None):
    """GDmin iterations; ops() yields (first column, operator).  fix(it, U, b, s):
    the measurements of a stored form, corrected with the exact operator."""
    yc = y
    for it in range(iters):
        if fix is not None and it % REFINE == 0:
            yc = fix(U, b, s)
        grad = torch.zeros_like(U)
        b = torch.zeros(len(y), U.shape[1], dtype=U.dtype, device=U.device)
        for k0, op, c in ops():
            z = slice(k0, k0 + c)
            s[z], G[z], b[z], h = _sweep(op, yc[z], U, s[z], G[z], rho)
            grad += h.T @ b[z].conj()
        if eta is None:
            eta = C_ETA / float(torch.linalg.matrix_norm(grad, 2))
        U = _orth(U - eta * grad)
    return U, b, s, G


def _support(G, s, rho):
    idx = G.topk(rho, dim=1).indices.sort(dim=1).values
    return idx.to(torch.int32), s.gather(1, idx)


def _exact_iterate(case, seed):
    A, Y, (U, B, Si, Sv), eta = _problem(case, seed)
    dft = "nx" in case
    dt = torch.complex128 if dft else torch.float64
    n, rho = U.shape[1], case["rho"]
    y, U, b, Sv = Y.to(dt), U.T.to(dt), B.to(dt), Sv.to(dt)
    s = torch.zeros(len(Y), n, dtype=dt, device="cuda").scatter_(1, Si.long(), Sv)
    G = torch.zeros(len(Y), n, dtype=torch.float64, device="cuda").scatter_(1, Si.long(), 1.0)
    form = case.get("a_dtype", 0)
    fix = None
    if dft:
        def ops():
            yield 0, _Dft(A, case["nx"], case["ny"]), len(Y)
    else:
        def ops():
            for k0, Ak in _chunks(A):
                yield k0, _Gauss(_stored(Ak.float(), form).double() if form else Ak), len(Ak)
    if form:
        def fix(U, b, s):
            yc = y.clone()
            for k0, Ak in _chunks(A):
                z = slice(k0, k0 + len(Ak))
                d = Ak - _stored(Ak.float(), form).double()
                yc[z] -= _Gauss(d).fwd(b[z] @ U.T + s[z])
            return yc
    U, b, s, G = _iterate64(ops, y, U, s, G, b, rho, eta, case["iters"], fix)
    Si, Sv = _support(G, s, rho)
    return dict(U=U.T.contiguous(), B=b, S_idx=Si, S_val=Sv)


def _exact_solve(case, seed):
    A, Y, _, _ = _problem(case, seed)
    dft, rho, r = "nx" in case, case["rho"], case["r"]
    op = _Dft(A, case["nx"], case["ny"]) if dft else _Gauss(A.double())
    dt = torch.complex128 if dft else torch.float64
    n = case["nx"] * case["ny"] if dft else case["n"]
    y = Y.to(dt)
    s, G = _iht(op, y, torch.zeros(len(y), n, dtype=dt, device="cuda"), None, rho, TAU0)
    L0 = op.adj(y - op.fwd(s)).T
    U = torch.linalg.eigh(L0 @ L0.mH).eigenvectors[:, -r:]
    U, b, s, G = _iterate64(lambda: [(0, op, len(y))], y, U, s, G, None, rho, None, case["iters"])
    return dict(X=b @ U.T + s, S_idx=_support(G, s, rho)[0])


def exact(case, seed):
    if case["kind"] == "qr":
        return _orth(_randn(_gen(seed), case["n"], case["r"]).double())
    if case["kind"].startswith("solve"):
        return _exact_solve(case, seed)
    if case["kind"] == "batch":
        return [_exact_iterate(dict(c, kind="gauss"), 1000 * seed + i)
                for i, c in enumerate(_members(case))]
    return _exact_iterate(case, seed)
