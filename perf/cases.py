"""Measured cases of the library: what a program asks of the smoothers.

Each case goes through a public call of ``paper_2207_00426_gb300.binding``:
the linear smoother (``sqsm_lgssm_smooth``), the iterated smoother on
coordinated-turn bearings tracks (``sqsm_ipls_smooth``; single tracks and
ragged batches, every linearisation, with and without refinement, FP32 and
FP64), the Ricker population model, and the negative pseudo log-likelihood
with its gradient (``sqsm_ipls_nll_grad``).  ``exact`` is the same arithmetic
in 64 bits in plain torch: covariance-form Kalman filter and
Rauch-Tung-Striebel smoother, run in blocks of consecutive steps.

The simulated tracks follow the workloads of the package (dt = 0.01,
q_c = 0.01, q_omega = 0.1, bearing noise 0.05 rad from two sensors, prior
0.1^2 I about the true initial state), drawn on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_2207_00426_gb300 import binding as B
from paper_2207_00426_gb300 import costmodel as CM

RULES = {"cubature": B.CUBATURE, "extended": B.EXTENDED, "unscented": B.UNSCENTED,
         "gauss_hermite": B.GAUSS_HERMITE}
DT = 0.01
SENSORS = ((-1.5, 0.5), (1.0, 1.0))
SIGMA, QC, QW = 0.05, 0.01, 0.1
PRIOR_STD = 0.1
RICKER = (44.7, 10.0, 0.09)          # a, b, Q
RICKER_X0 = math.log(7.0)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _linear(n, nx, ny, dtype, varying):
    return dict(call="linear", n=n, nx=nx, ny=ny, dtype=dtype, varying=varying)


def _tracks(batch, lo, hi, M, rule="cubature", dtype="f32", refine=0):
    return dict(call="tracks", batch=batch, lo=lo, hi=hi, M=M, rule=rule, dtype=dtype,
                refine=refine, warm=True)


def _grad(batch, lo, hi, M, adj, n_theta, rule="cubature", dtype="f32"):
    return dict(call="grad", batch=batch, lo=lo, hi=hi, M=M, adj=adj, n_theta=n_theta, rule=rule,
                dtype=dtype, warm=True)


def _ricker(batch, lo, hi, M, rule, dtype="f32"):
    return dict(call="ricker", batch=batch, lo=lo, hi=hi, M=M, rule=rule, dtype=dtype)


def listed():
    return [
        # one pass over a short linear constant-velocity record: the smallest
        # call, all launches and latency
        dict(_linear(1000, 4, 2, "f32", False), name="cv_1000_f32"),
        # the linear smoother on a long time-varying model (what an outer
        # loop of the caller's own linearisation hands over)
        dict(_linear(100_000, 5, 2, "f32", True), name="linear_100k_f32"),
        # the same call in double, for reference results
        dict(_linear(20_011, 6, 3, "f64", True), name="linear_20k_f64"),
        # (tracks start from an estimate at hand, see draw)
        # a 1 s track smoothed while it is flown: short and latency-bound
        dict(_tracks(1, 100, 100, 20, "unscented"), name="track_100_ut"),
        # one 10 s track, the plain use of the iterated smoother
        dict(_tracks(1, 1000, 1000, 10), name="track_1000"),
        # one 1000 s track re-smoothed from the estimate at hand, with a
        # refinement pass: the accurate FP32 mode of long runs
        dict(_tracks(1, 100_000, 100_000, 10, refine=1), name="track_100k_refined"),
        # one track in double
        dict(_tracks(1, 4000, 4000, 10, dtype="f64"), name="track_4000_f64"),
        # the 243-point rule on one 40 s track
        dict(_tracks(1, 4000, 4000, 5, "gauss_hermite"), name="track_4000_gh"),
        # many recorded tracks of 1 to 50 s at once: throughput
        dict(_tracks(4096, 100, 5000, 2), name="batch_4096"),
        # one likelihood evaluation with its gradient inside an optimiser,
        # one noise level per sensor
        dict(_grad(1, 1000, 1000, 20, 20, 4), name="grad_1000"),
        # the same over a data set of 256 tracks
        dict(_grad(256, 2000, 2000, 10, 10, 3), name="grad_256x2000"),
        # the population model, n_x = n_y = 1
        dict(_ricker(1, 10_000, 10_000, 50, "cubature"), name="ricker_10k"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    # every track and batch starts from an estimate at hand (a previous
    # smoothing, a coarse fix): from the prior alone the iteration does not
    # settle on some tracks, and such results are noise in any precision
    call = rng.choice(["linear", "linear", "tracks", "tracks", "batch", "batch", "grad", "ricker"])
    dtype = rng.choice(["f32", "f32", "f64"])
    if call == "linear":
        nx, ny = rng.choice([(4, 2), (5, 2), (6, 3)])
        if nx == 4:     # short: the positions of this model grow with n^1.5
            return _linear(_log_uniform(rng, 300, 4000), nx, ny, dtype, False)
        return _linear(_log_uniform(rng, 1000, 100_000 if dtype == "f32" else 20_011), nx, ny,
                       dtype, True)
    f32 = dtype == "f32"
    if call == "tracks":
        rule = rng.choice(["cubature", "cubature", "extended", "unscented", "gauss_hermite"])
        if rng.random() < 0.5:      # long
            n = _log_uniform(rng, 4000, 100_000 if f32 else 20_000)
            return _tracks(1, n, n, 2, "cubature" if rule == "gauss_hermite" else rule, dtype,
                           int(f32))
        n = _log_uniform(rng, 100, 2000)
        if not f32:
            return _tracks(1, n, n, rng.randint(2, 8), "extended", dtype)
        return _tracks(1, n, n, rng.randint(5, 20), rule, dtype)
    if call == "batch":
        b = _log_uniform(rng, 16, 4096 if f32 else 64)
        lo = _log_uniform(rng, 50, 400 if f32 else 200)
        return _tracks(b, lo, lo * rng.randint(1, 10), 2, rng.choice(["cubature", "extended"]),
                       dtype)
    if call == "grad":
        b = _log_uniform(rng, 1, 256)
        lo = _log_uniform(rng, 100, 1000)
        return _grad(b, lo, min(2000, 2 * lo), rng.randint(5, 10), rng.randint(5, 10),
                     rng.choice([3, 4]), rng.choice(["cubature", "extended"]))
    b = rng.choice([1, 1, 7, 30])
    n = _log_uniform(rng, 100, 10_000)
    return _ricker(b, n, n + n // 3, rng.randint(10, 50), rng.choice(["cubature", "extended"]),
                   dtype)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _lengths(case):
    # the record lengths belong to the data set, not to its noise
    rng = np.random.default_rng([case["batch"], case["lo"], case["hi"]])
    return rng.integers(case["lo"], case["hi"] + 1, size=case["batch"])


def _offsets(lengths):
    return np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + 17)


def _csum(a):
    # cumulative sum over time, the first axis (one thread per column)
    return torch.cumsum(a, 0)


def _simulate_tracks(lengths, seed):
    """True states [n_max + 1, S, 5] and bearings [n_max, S, 2] of S >= 2
    independent coordinated-turn tracks in double, time first: the turn angle,
    the velocity in the turning frame and the position are running sums."""
    g = _gen(seed)
    S, n = max(2, len(lengths)), int(max(lengths))

    def randn(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)

    speed = 0.5 + 1.5 * torch.rand(S, generator=g, device="cuda", dtype=torch.float64)
    head = 2 * math.pi * torch.rand(S, generator=g, device="cuda", dtype=torch.float64)
    w0 = 0.3 * randn(S)
    w = torch.cat([w0[None], w0 + _csum(math.sqrt(QW * DT) * randn(n, S))])
    a = w[:-1] * DT
    turn = _csum(a)                                     # angle after step k
    e = randn(n, 2, S)
    vn = math.sqrt(QC) * (math.sqrt(3 * DT) / 2 * e + math.sqrt(DT) / 2 * randn(n, 2, S))
    pn = math.sqrt(QC * DT ** 3 / 3) * e
    c, s = torch.cos(turn), torch.sin(turn)
    vx0, vy0 = speed * torch.cos(head), speed * torch.sin(head)
    fx = vx0 + _csum(c * vn[:, 0] + s * vn[:, 1])       # velocity in the turning frame
    fy = vy0 + _csum(c * vn[:, 1] - s * vn[:, 0])
    vx = torch.cat([vx0[None], c * fx - s * fy])
    vy = torch.cat([vy0[None], s * fx + c * fy])
    safe = torch.where(a.abs() < 1e-9, torch.ones_like(a), a)
    S_ = DT * torch.where(a.abs() < 1e-9, torch.ones_like(a), torch.sin(safe) / safe)
    C_ = DT * torch.where(a.abs() < 1e-9, a / 2, 2 * torch.sin(safe / 2) ** 2 / safe)
    zero = torch.zeros(1, S, dtype=torch.float64, device="cuda")
    px = torch.cat([zero, _csum(S_ * vx[:-1] - C_ * vy[:-1] + pn[:, 0])])
    py = torch.cat([zero, _csum(C_ * vx[:-1] + S_ * vy[:-1] + pn[:, 1])])
    x = torch.stack([px, py, vx, vy, w], -1)
    sx = torch.tensor(SENSORS, dtype=torch.float64, device="cuda")
    y = torch.atan2(x[1:, :, None, 1] - sx[:, 1], x[1:, :, None, 0] - sx[:, 0])
    y = y + SIGMA * randn(n, S, 2)
    y = y - 2 * math.pi * torch.floor(y / (2 * math.pi) + 0.5)
    return x, y


def _ragged(a, lengths):
    """Rows 0 .. lengths[b] - 1 of every column b of a [n, S, ...], concatenated."""
    a = a[:, : len(lengths)].transpose(0, 1)
    live = torch.arange(a.shape[1], device="cuda")[None] < torch.as_tensor(
        np.asarray(lengths), device="cuda")[:, None]
    return a[live]


def _tracks_inputs(case, seed):
    lengths = _lengths(case)
    x, y = _simulate_tracks(lengths, seed)
    nb = len(lengths)
    dt = _dtype(case)
    eye = torch.eye(5, dtype=dt, device="cuda")
    d = dict(lengths=lengths, off=_offsets(lengths), y=_ragged(y, lengths).to(dt).contiguous(),
             m0=x[0, :nb].to(dt).contiguous(), N0=(PRIOR_STD * eye).repeat(nb, 1, 1))
    if case.get("warm"):
        # the estimate at hand: off by a slowly varying error of the prior's size
        g = _gen(seed + 1)
        ph = 2 * math.pi * torch.rand(x.shape[1], 5, generator=g, device="cuda",
                                      dtype=torch.float64)
        t = DT * torch.arange(x.shape[0], device="cuda", dtype=torch.float64)
        x0 = x + 0.5 * PRIOR_STD * torch.sin(t[:, None, None] + ph)
        d["init_ms"] = _ragged(x0, np.asarray(lengths) + 1).to(dt).contiguous()
        d["init_Ns"] = (PRIOR_STD * eye).repeat(d["init_ms"].shape[0], 1, 1)
    return d


def _ricker_inputs(case, seed):
    lengths = _lengths(case)
    a, b, q = RICKER
    rng = np.random.default_rng(seed + 7)
    S, n = len(lengths), int(max(lengths))
    e = math.sqrt(q) * rng.standard_normal((n, S))
    x = np.full(S, RICKER_X0)
    xs = np.empty((n, S))
    for t in range(n):
        x = math.log(a) + x - np.exp(x) + e[t]
        xs[t] = x
    counts = rng.poisson(b * np.exp(xs)).astype(np.float64)
    y = np.concatenate([counts[: lengths[i], i] for i in range(S)])[:, None]
    dt = _dtype(case)
    return dict(lengths=lengths, off=_offsets(lengths), y=torch.tensor(y, device="cuda").to(dt),
                m0=torch.full((S, 1), RICKER_X0, dtype=dt, device="cuda"),
                N0=torch.zeros((S, 1, 1), dtype=dt, device="cuda"))


def _linear_inputs(case, seed):
    """Constant-velocity model (dt = 0.1, q = 0.1, positions observed with
    noise 0.5), or a random contractive time-varying one; y simulated from it
    (the recursion composed by doubling)."""
    n, nx, ny = case["n"], case["nx"], case["ny"]
    g = _gen(seed)

    def randn(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)

    if case["varying"]:
        def lower(k, scale):
            L = torch.tril(scale * randn(n, k, k))
            i = torch.arange(k, device="cuda")
            L[:, i, i] = L[:, i, i].abs() + scale
            return L
        F = torch.eye(nx, dtype=torch.float64, device="cuda") + 0.3 * randn(n, nx, nx) / nx ** 0.5
        # at least the spectral norm: the square root of the 1- and inf-norms' product
        top = (F.abs().sum(-1).amax(-1) * F.abs().sum(-2).amax(-1)).sqrt()
        F = F * torch.clamp(0.98 / top, max=1.0)[:, None, None]
        c, SQ = 0.1 * randn(n, nx), lower(nx, 0.3)
        H, d, SR = randn(n, ny, nx), 0.1 * randn(n, ny), lower(ny, 0.3)
        m0, N0 = randn(nx), torch.tril(randn(nx, nx))
        N0.diagonal().abs_().add_(1.0)
    else:
        dt, q, sigma = 0.1, 0.1, 0.5
        I2 = torch.eye(2, dtype=torch.float64, device="cuda")
        Z2 = torch.zeros_like(I2)
        F = torch.cat([torch.cat([I2, dt * I2], 1), torch.cat([Z2, I2], 1)])
        SQ = math.sqrt(q) * torch.cat(
            [torch.cat([math.sqrt(dt ** 3 / 3) * I2, Z2], 1),
             torch.cat([math.sqrt(3 * dt) / 2 * I2, math.sqrt(dt) / 2 * I2], 1)])
        H, SR = torch.cat([I2, Z2], 1), sigma * I2
        c, d = F.new_zeros(4), F.new_zeros(2)
        m0, N0 = F.new_zeros(4), torch.eye(4, dtype=torch.float64, device="cuda")
    m = dict(F=F, c=c, SQ=SQ, H=H, d=d, SR=SR, m0=m0, N0=N0)
    m = {k: v.to(_dtype(case)) for k, v in m.items()}
    # x_{t+1} = F_t x_t + u_t: inclusive products of the affine maps
    f = {k: v.double() for k, v in m.items()}
    step = {k: (f[k] if case["varying"] else f[k].expand(n, *f[k].shape))
            for k in ("F", "c", "SQ", "H", "d", "SR")}
    A = step["F"].clone()
    u = step["c"] + (step["SQ"] @ randn(n, nx, 1))[..., 0]
    x0 = f["m0"] + f["N0"] @ randn(nx)
    k = 1
    while k < n:
        u = torch.cat([u[:k], (A[k:] @ u[:-k, :, None])[..., 0] + u[k:]])
        A = torch.cat([A[:k], A[k:] @ A[:-k]])
        k *= 2
    x = (A @ x0) + u
    y = (step["H"] @ x[..., None])[..., 0] + step["d"] + (step["SR"] @ randn(n, ny, 1))[..., 0]
    m["y"] = y.to(_dtype(case)).contiguous()
    return m


def _inputs(case, seed):
    return {"linear": _linear_inputs, "tracks": _tracks_inputs, "grad": _tracks_inputs,
            "ricker": _ricker_inputs}[case["call"]](case, seed)


def _theta(case):
    if case["call"] == "ricker":
        return np.log(np.array(RICKER))
    th = [SIGMA, QC, QW]
    th = np.log(np.array(th + [SIGMA] if case.get("n_theta") == 4 else th))
    if case["call"] == "grad":          # where an optimiser starts, not the optimum
        th[:3] += [0.3, -0.3, 0.3]
    return th


def prepare(case, seed):
    d = _inputs(case, seed)
    return dict(case=case, d=d, theta=_theta(case),
                ctx=B.Context(0, refine=case.get("refine", 0)))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _scalar(ll, case):
    # log-likelihoods and gradients of FP32 data are FP32 numbers that the
    # library sums in double; a program keeps them at the data's precision
    return ll.to(_dtype(case))


def run(state):
    case, d, ctx = state["case"], state["d"], state["ctx"]
    if case["call"] == "linear":
        mf, Nf, ms, Ns, ll = B.sqsm_lgssm_smooth(ctx, d["F"], d["c"], d["SQ"], d["H"], d["d"],
                                                 d["SR"], d["m0"], d["N0"], d["y"])
        return dict(mf=mf, Nf=Nf, ms=ms, Ns=Ns, ll=_scalar(ll, case))
    lin = RULES[case["rule"]]
    if case["call"] == "tracks":
        ms, Ns, ll = B.sqsm_ipls_smooth(ctx, state["theta"], d["y"], d["off"], d["m0"], d["N0"],
                                        case["M"], lin, init_ms=d.get("init_ms"),
                                        init_Ns=d.get("init_Ns"))
        return dict(ms=ms, Ns=Ns, ll=_scalar(ll, case))
    if case["call"] == "ricker":
        ms, Ns, ll = B.sqsm_ipls_smooth_population(ctx, state["theta"], d["y"], d["off"], d["m0"],
                                                   d["N0"], case["M"], lin)
        return dict(ms=ms, Ns=Ns, ll=_scalar(ll, case))
    nll, grad, _, ms, Ns = B.sqsm_ipls_nll_grad(ctx, state["theta"], d["y"], d["off"], d["m0"],
                                                d["N0"], case["M"], case["adj"],
                                                init_ms=d["init_ms"], init_Ns=d["init_Ns"],
                                                linearization=lin)
    return dict(nll=_scalar(nll, case), grad=_scalar(grad, case), ms=ms, Ns=Ns)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: caller's inputs and outputs once.  Flops: the sequential
    recursion (one linearisation, Kalman step and RTS step per time step and
    iteration; the gradient's adjoint counted as twice a smoothing pass per
    adjoint iteration)."""
    es = 4 if case["dtype"] == "f32" else 8
    if case["call"] == "linear":
        n, nx, ny = case["n"], case["nx"], case["ny"]
        model = nx * nx * 2 + nx + ny * nx + ny + ny * ny
        io = n * ny + 2 * (n + 1) * (nx + nx * nx) + (n if case["varying"] else 1) * model
        return dict(bytes=es * io, flops=n * (CM.kf_step(nx, ny) + CM.smoother_element(nx)
                                              + CM.smoother_apply(nx)))
    n = case["batch"] * (case["lo"] + case["hi"]) / 2
    rows = n + case["batch"]
    nx, ny = (1, 1) if case["call"] == "ricker" else (5, 2)
    smooth = CM.kf_step(nx, ny) + CM.smoother_element(nx) + CM.smoother_apply(nx)
    points = {"extended": 0, "cubature": 2 * nx, "unscented": 2 * nx + 1,
              "gauss_hermite": 3 ** nx}[case["rule"]]
    slr = 30 * points + CM.tria(nx, 2 * nx) + CM.tria(ny, nx + ny) + nx * nx * (nx + ny)
    if not points:
        slr = 4 * nx * nx + 60
    per = slr + smooth * (1 + case.get("refine", 0))
    its = case["M"]
    if case["call"] == "grad":
        its += 1 + 2 * case["adj"]
    states = rows * (nx + nx * nx)
    return dict(bytes=es * (n * ny + states * (2 if case.get("warm") else 1)),
                flops=n * per * its)


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _mm(*Ms):
    """Product of batched small matrices; of millions, entry by entry (batched
    library products of 5 x 5 doubles take seconds there)."""
    A = Ms[0]
    for M in Ms[1:]:
        if max(A.numel(), M.numel()) < 1_000_000:
            A = A @ M
            continue
        P = A[..., :, :1] * M[..., :1, :]
        for k in range(1, A.shape[-1]):
            P.addcmul_(A[..., :, k : k + 1], M[..., k : k + 1, :])
        A = P
    return A


def _mv(A, x):
    return _mm(A, x[..., None])[..., 0]


def _sym(P):
    return 0.5 * (P + P.mT)


def _inv(A):
    """Inverse and determinant of small symmetric matrices, 1 x 1 and 2 x 2
    in closed form (a batched factorisation of millions takes seconds)."""
    if A.shape[-1] == 1:
        return 1 / A, A[..., 0, 0]
    if A.shape[-1] == 2:
        det = A[..., 0, 0] * A[..., 1, 1] - A[..., 0, 1] * A[..., 1, 0]
        adj = torch.stack([A[..., 1, 1], -A[..., 0, 1], -A[..., 1, 0], A[..., 0, 0]], -1)
        return (adj / det[..., None]).reshape(A.shape), det
    return torch.linalg.inv(A), torch.linalg.det(A)


def _smooth64(F, c, Q, H, r, R, lengths, m0, P0):
    """Kalman filter and RTS smoother of S sequences, time first: F, c, Q
    [T, S, ...] transitions, H, r = y - d, R observations, rows past a
    sequence's length being ignored.  Steps run in K blocks of consecutive
    steps at once: each block's composed map, the blocks' starting states one
    after another, then the plain recursion inside all blocks.  Returns
    filtered and smoothed means / covariances [T + 1, S, ...] and the
    log-likelihood [S]."""
    T, S, nx = c.shape
    ny = r.shape[-1]
    L = max(1, int(math.sqrt(T)))          # steps per block
    nb = -(-T // L)
    dev, dt = c.device, torch.float64
    eye = torch.eye(nx, dtype=dt, device=dev)
    live = torch.arange(nb * L, device=dev)[:, None] < lengths[None]

    def blocks(a, fill):
        pad = nb * L - T
        if pad:
            a = torch.cat([a, a[:1].expand(pad, *a.shape[1:])])
        k = live.reshape(nb * L, S, *([1] * (a.dim() - 2)))
        a = torch.where(k, a, fill)
        return a.reshape(nb, L, *a.shape[1:]).transpose(0, 1)     # [L, nb, S, ...]

    zero = torch.zeros((), dtype=dt, device=dev)
    F, c, Q = blocks(F, eye), blocks(c, zero), blocks(Q, zero)
    H, r, R = blocks(H, zero), blocks(r, zero), blocks(R, torch.eye(ny, dtype=dt, device=dev))
    liveb = live.reshape(nb, L, S).transpose(0, 1)
    # every block's composed element (A, b, C, eta, J)
    A = eye.expand(nb, S, nx, nx)
    b = c.new_zeros(nb, S, nx)
    C = c.new_zeros(nb, S, nx, nx)
    eta, J = b.clone(), C.clone()
    for j in range(L):
        S0 = _mm(H[j], Q[j], H[j].mT) + R[j]
        Sj, _ = _inv(S0)
        Kg = _mm(Q[j], H[j].mT, Sj)
        IKH = eye - _mm(Kg, H[j])
        v = r[j] - _mv(H[j], c[j])
        HF = _mm(H[j], F[j])
        A2, b2, C2 = _mm(IKH, F[j]), c[j] + _mv(Kg, v), _sym(_mm(IKH, Q[j]))
        W = _mm(HF.mT, Sj)
        e2, J2 = _mv(W, v), _sym(_mm(W, HF))
        # (I + C J2)^{-1} with J2 = HF^T S0^{-1} HF
        CW = _mm(C, HF.mT)
        D = eye - _mm(CW, _inv(S0 + _mm(HF, CW))[0], HF)
        A2D = _mm(A2, D)
        AD = _mm(A.mT, D.mT)
        b, eta = _mv(A2D, b + _mv(C, e2)) + b2, _mv(AD, e2 - _mv(J2, b)) + eta
        J = _sym(_mm(AD, J2, A)) + J
        C = _sym(_mm(A2D, C, A2.mT)) + C2
        A = _mm(A2D, A)
    m, P = m0, P0
    ms, Ps = [], []
    for k in range(nb):
        ms.append(m)
        Ps.append(P)
        D = torch.linalg.inv(eye + P @ J[k])
        AD = A[k] @ D
        m, P = _mv(AD, m + _mv(P, eta[k])) + b[k], _sym(AD @ P @ A[k].mT) + C[k]
    m, P = torch.stack(ms), torch.stack(Ps)
    mf, Pf = [m], [P]
    ll = c.new_zeros(nb, S)
    for j in range(L):
        mp, Pp = _mv(F[j], m) + c[j], _sym(_mm(F[j], P, F[j].mT)) + Q[j]
        Sm = _sym(_mm(H[j], Pp, H[j].mT)) + R[j]
        Sj, det = _inv(Sm)
        v = r[j] - _mv(H[j], mp)
        Kg = _mm(Pp, H[j].mT, Sj)
        IKH = eye - _mm(Kg, H[j])
        m = mp + _mv(Kg, v)
        P = _sym(_mm(IKH, Pp, IKH.mT) + _mm(Kg, R[j], Kg.mT))
        l1 = -0.5 * (ny * math.log(2 * math.pi) + torch.log(det) + (v * _mv(Sj, v)).sum(-1))
        ll = ll + torch.where(liveb[j], l1, zero)
        mf.append(m)
        Pf.append(P)
    mT, PT = m[-1], P[-1]
    mf, Pf = torch.stack(mf[:-1]), torch.stack(Pf[:-1])           # [L, nb, S, ...], rows 0 .. nb L - 1
    # smoother: maps of row k onto row k + 1; a sequence's last row starts it
    Pp = _sym(_mm(F, Pf, F.mT)) + Q
    E = torch.linalg.solve(Pp, _mm(F, Pf)).mT
    g = mf - _mv(E, _mv(F, mf) + c)
    IEF = eye - _mm(E, F)
    V = _sym(_mm(IEF, Pf, IEF.mT) + _mm(E, Q, E.mT))
    del Pp, IEF
    last = (torch.arange(nb * L, device=dev)[:, None] == lengths[None]).reshape(nb, L, S)
    last = last.transpose(0, 1)
    E = torch.where(last[..., None, None], zero, E)
    g = torch.where(last[..., None], mf, g)
    V = torch.where(last[..., None, None], Pf, V)
    Eb, gb, Vb = eye.expand(nb, S, nx, nx), c.new_zeros(nb, S, nx), c.new_zeros(nb, S, nx, nx)
    for j in range(L - 1, -1, -1):
        gb = _mv(E[j], gb) + g[j]
        Vb = _sym(_mm(E[j], Vb, E[j].mT)) + V[j]
        Eb = _mm(E[j], Eb)
    m, P = mT, PT
    ms, Ps = [None] * nb, [None] * nb
    for k in range(nb - 1, -1, -1):
        ms[k], Ps[k] = m, P
        m, P = _mv(Eb[k], m) + gb[k], _sym(Eb[k] @ P @ Eb[k].mT) + Vb[k]
    m, P = torch.stack(ms), torch.stack(Ps)
    sm, sP = [None] * L, [None] * L
    for j in range(L - 1, -1, -1):
        m, P = _mv(E[j], m) + g[j], _sym(_mm(E[j], P, E[j].mT)) + V[j]
        sm[j], sP[j] = m, P

    def rows(a, end):
        a = a.transpose(0, 1).reshape(nb * L, *a.shape[2:])
        return torch.cat([a, end[None]])[: T + 1]

    return (rows(mf, mT), rows(Pf, PT), rows(torch.stack(sm), mT), rows(torch.stack(sP), PT),
            ll.sum(0))


def _points(rule, nx):
    eye = torch.eye(nx, dtype=torch.float64, device="cuda")
    if rule == "cubature":
        s = math.sqrt(nx)
        return torch.cat([s * eye, -s * eye]), torch.full((2 * nx,), 0.5 / nx, device="cuda",
                                                          dtype=torch.float64)
    if rule == "unscented":
        s = math.sqrt(nx + 1)
        w = torch.full((2 * nx + 1,), 0.5 / (nx + 1), device="cuda", dtype=torch.float64)
        w[0] = 1 / (nx + 1)
        return torch.cat([eye[:1] * 0, s * eye, -s * eye]), w
    node = torch.tensor([0.0, 3 ** 0.5, -3 ** 0.5], dtype=torch.float64, device="cuda")
    w1 = torch.tensor([2 / 3, 1 / 6, 1 / 6], dtype=torch.float64, device="cuda")
    idx = torch.cartesian_prod(*[torch.arange(3, device="cuda")] * nx)
    return node[idx], w1[idx].prod(-1)


def _regress(rule, m, N, f, S_cond, diff):
    """Statistical linear regression of f about N(m, N N^T): matrix, offset
    (relative to f(m)) and residual covariance.  diff(z, z0): z - z0;
    S_cond(X): the conditional covariance of each point."""
    xi, w = _points(rule, m.shape[-1])
    z0 = f(m)
    X = m[..., None, :] + (N @ xi.mT).mT
    Z = diff(f(X), z0[..., None, :])
    w_ = w[:, None]
    zb = (w_ * Z).sum(-2)
    D = (w_ * (Z - zb[..., None, :])).mT @ xi
    G = torch.linalg.solve_triangular(N, D, upper=False, left=False)
    res = (Z - zb[..., None, :]) - (D @ xi.mT).mT
    cov = (w_ * res).mT @ res + (w_[..., None] * S_cond(X)).sum(-3)
    return G, z0, zb, cov


def _turn64(w):
    a = w * DT
    small = a.abs() < 1e-3
    s = torch.where(small, torch.ones_like(a), a)
    a2 = a * a
    S = DT * torch.where(small, 1 - a2 / 6 + a2 * a2 / 120, torch.sin(s) / s)
    C = DT * torch.where(small, a * (0.5 - a2 / 24 + a2 * a2 / 720), 2 * torch.sin(s / 2) ** 2 / s)
    return a, S, C


def _ct_f(x):
    px, py, vx, vy, w = x.unbind(-1)
    a, S, C = _turn64(w)
    ca, sa = torch.cos(a), torch.sin(a)
    return torch.stack([px + S * vx - C * vy, py + C * vx + S * vy, ca * vx - sa * vy,
                        sa * vx + ca * vy, w], -1)


def _ct_h(x):
    s = torch.tensor(SENSORS, dtype=torch.float64, device="cuda")
    return torch.atan2(x[..., 1:2] - s[:, 1], x[..., 0:1] - s[:, 0])


def _ct_jacobians(x):
    """Jacobians of the transition and of the bearings."""
    vx, vy, w = x[..., 2], x[..., 3], x[..., 4]
    a, S, C = _turn64(w)
    ca, sa = torch.cos(a), torch.sin(a)
    small = a.abs() < 0.1
    s = torch.where(small, torch.ones_like(a), a)
    a2 = a * a
    dS = DT * DT * torch.where(
        small, a * (-1 / 3 + a2 * (1 / 30 + a2 * (-1 / 840 + a2 / 45360))),
        (s * torch.cos(s) - torch.sin(s)) / (s * s))
    dC = DT * DT * torch.where(
        small, 0.5 + a2 * (-1 / 8 + a2 * (1 / 144 + a2 * (-1 / 5760 + a2 / 403200))),
        (s * torch.sin(s) - 2 * torch.sin(s / 2) ** 2) / (s * s))
    F = torch.zeros(*x.shape, 5, dtype=torch.float64, device="cuda")
    F[..., range(5), range(5)] = 1.0
    F[..., 0, 2], F[..., 0, 3], F[..., 0, 4] = S, -C, vx * dS - vy * dC
    F[..., 1, 2], F[..., 1, 3], F[..., 1, 4] = C, S, vx * dC + vy * dS
    F[..., 2, 2], F[..., 2, 3], F[..., 2, 4] = ca, -sa, -DT * (sa * vx + ca * vy)
    F[..., 3, 2], F[..., 3, 3], F[..., 3, 4] = sa, ca, DT * (ca * vx - sa * vy)
    p = torch.tensor(SENSORS, dtype=torch.float64, device="cuda")
    dx, dy = x[..., 0:1] - p[:, 0], x[..., 1:2] - p[:, 1]
    r2 = dx * dx + dy * dy
    H = torch.zeros(*x.shape[:-1], 2, 5, dtype=torch.float64, device="cuda")
    H[..., 0], H[..., 1] = -dy / r2, dx / r2
    return F, H


def _wrap(z):
    return z - 2 * math.pi * torch.floor(z / (2 * math.pi) + 0.5)


def _linearise_ct(rule, m, N, y, theta):
    """Rows 0 .. T of the nominal -> transitions, observations of the T steps."""
    s1, QC, QW = np.exp(theta[:3])
    s2 = np.exp(theta[3]) if len(theta) == 4 else s1
    th = [s1 ** 2, s2 ** 2]
    Q = torch.zeros(5, 5, dtype=torch.float64, device="cuda")
    for i in (0, 1):
        Q[i, i], Q[i + 2, i + 2] = QC * DT ** 3 / 3, QC * DT
        Q[i, i + 2] = Q[i + 2, i] = QC * DT ** 2 / 2
    Q[4, 4] = QW * DT
    R = torch.diag(torch.tensor(th, dtype=torch.float64, device="cuda"))
    mp, mk = m[:-1], m[1:]
    if rule == "extended":
        F, _ = _ct_jacobians(mp)
        _, H = _ct_jacobians(mk)
        fb, hz, hb = _ct_f(mp), _ct_h(mk), 0.0
        Qk, Rk = Q.expand(*F.shape), R.expand(*H.shape[:-1], 2)
    else:
        F, f0, zb, cov = _regress(rule, mp, N[:-1], _ct_f, lambda X: 0 * X[..., None], torch.sub)
        fb, Qk = f0 + zb, Q + cov
        H, hz, hb, cov = _regress(rule, mk, N[1:], _ct_h, lambda X: 0 * X[..., :1, None],
                                  lambda a, b: _wrap(a - b))
        Rk = R + cov
    # r = y - d with y on the branch nearest h(m)
    return F, fb - _mv(F, mp), Qk, H, _wrap(y - hz) - hb + _mv(H, mk), Rk


def _linearise_ricker(rule, m, N, y, theta):
    a, b, q = np.exp(theta)
    ones = torch.ones_like(m)[..., None]

    def f(x):
        return math.log(a) + x - torch.exp(x)

    def h(x):
        return b * torch.exp(x)

    mp, mk = m[:-1], m[1:]
    F, fb, Qk = (1 - torch.exp(mp))[..., None], f(mp), q * ones[:-1]
    H, hb, Rk = h(mk)[..., None], h(mk), h(mk)[..., None]
    if rule != "extended":
        known = N[:-1] == 0                      # a point mass keeps the Taylor form
        Np = torch.where(known, torch.ones_like(N[:-1]), N[:-1])
        G, z0, zb, cov = _regress(rule, mp, Np, f, lambda X: 0 * X[..., None], torch.sub)
        F = torch.where(known, F, G)
        fb = torch.where(known[..., 0], fb, z0 + zb)
        Qk = torch.where(known, Qk, q + cov)
        known = N[1:] == 0
        Nk = torch.where(known, torch.ones_like(N[1:]), N[1:])
        G, z0, zb, cov = _regress(rule, mk, Nk, h, lambda X: h(X)[..., None], torch.sub)
        H = torch.where(known, H, G)
        hb = torch.where(known[..., 0], hb, z0 + zb)
        Rk = torch.where(known, Rk, cov)
    return F, fb - _mv(F, mp), Qk, H, y - hb + _mv(H, mk), Rk


def _padded(a, lengths, n):
    """Concatenated ragged rows -> [n, S, ...], missing rows repeating row 0."""
    off = _offsets(lengths)[:-1]
    k = np.arange(n)[:, None]
    idx = np.where(k < np.asarray(lengths)[None], off[None] + k, off[None])
    return a.double()[torch.as_tensor(idx, device="cuda")]


def _exact_ipls(case, d):
    """Sequences of similar length together (they are padded to the longest)."""
    lengths, off = np.asarray(d["lengths"]), d["off"]
    order = np.argsort(lengths, kind="stable")
    rows, m, N = int(off[-1]) + len(lengths), None, None
    ll = torch.empty(len(lengths), dtype=torch.float64, device="cuda")
    for idx in np.array_split(order, -(-len(order) // 512)):
        steps = np.concatenate([off[b] + np.arange(lengths[b]) for b in idx])
        states = np.concatenate([off[b] + b + np.arange(lengths[b] + 1) for b in idx])
        it, st = torch.as_tensor(steps, device="cuda"), torch.as_tensor(states, device="cuda")
        ib = torch.as_tensor(idx, device="cuda")
        sub = dict(lengths=lengths[idx], y=d["y"][it], m0=d["m0"][ib], N0=d["N0"][ib])
        if "init_ms" in d:
            sub.update(init_ms=d["init_ms"][st], init_Ns=d["init_Ns"][st])
        mg, Ng, lg = _exact_group(case, sub)
        if m is None:
            m, N = (a.new_empty(rows, *a.shape[1:]) for a in (mg, Ng))
        m[st], N[st], ll[ib] = mg, Ng, lg
    return m, N, ll


def _exact_group(case, d):
    lengths = np.asarray(d["lengths"])
    T = int(lengths.max())
    ln = torch.as_tensor(lengths, device="cuda")
    y = _padded(d["y"], lengths, T)
    m0, N0 = d["m0"].double(), d["N0"].double()
    if "init_ms" in d:
        m = _padded(d["init_ms"], lengths + 1, T + 1)
        N = _padded(d["init_Ns"], lengths + 1, T + 1)
    else:
        m, N = m0.expand(T + 1, *m0.shape), N0.expand(T + 1, *N0.shape)
    lin = _linearise_ricker if case["call"] == "ricker" else _linearise_ct
    P0, theta = N0 @ N0.mT, _theta(case)
    for _ in range(case["M"]):
        _, _, m, P, ll = _smooth64(*lin(case["rule"], m, N, y, theta), ln, m0, P0)
        N = P.clamp(min=0).sqrt() if P.shape[-1] == 1 else torch.linalg.cholesky(P)
    if case["call"] == "grad":
        ll = _smooth64(*lin(case["rule"], m, N, y, theta), ln, m0, P0)[4]
    return _ragged(m, lengths + 1), _ragged(N, lengths + 1), ll


def exact(case, seed):
    d = _inputs(case, seed)
    if case["call"] == "linear":
        n = case["n"]
        f = {k: v.double() for k, v in d.items()}
        s = {k: (f[k] if case["varying"] else f[k].expand(n, *f[k].shape))[:, None]
             for k in ("F", "c", "SQ", "H", "d", "SR")}
        mf, Pf, ms, Ps, ll = _smooth64(s["F"], s["c"], s["SQ"] @ s["SQ"].mT, s["H"],
                                       f["y"][:, None] - s["d"], s["SR"] @ s["SR"].mT,
                                       torch.tensor([n], device="cuda"), f["m0"][None],
                                       (f["N0"] @ f["N0"].mT)[None])
        return dict(mf=mf[:, 0], Nf=torch.linalg.cholesky(Pf[:, 0]), ms=ms[:, 0],
                    Ns=torch.linalg.cholesky(Ps[:, 0]), ll=ll)
    m, N, ll = _exact_ipls(case, d)
    if case["call"] == "grad":
        return dict(nll=-ll.sum().reshape(1), grad=None, ms=m, Ns=N)
    return dict(ms=m, Ns=N, ll=ll)
