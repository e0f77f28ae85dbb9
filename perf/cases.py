"""Performance cases of the framework: what its users have it do, through its public entry points.

Sizes are those of the repository's own workloads (inputs.workload, inputs.mixed_batch), benchmark
lines and tests: base-2 nets and lattices, n = 2^10 .. 2^22 points, d = 1 .. 128, kernels of
every order, FP64, FP32 (with a refinement step) and the float-float first column (f32w).

Every input is made here from the seed alone (generator columns, shifts, right-hand sides),
so that `exact` forms the same results in plain torch, in 64 bits, without the framework.
"""
from __future__ import annotations

import math

import torch

from paper_2502_14256_gb300 import qk
from paper_2502_14256_gb300.autograd import mll_and_mean

F64, F32 = torch.float64, torch.float32
M32 = 0xFFFFFFFF
INTEGRANDS = ["simple1", "simple2", "oakley", "gfun", "genz_osc", "genz_cp"]


def listed():
    return [
        # one evaluation and gradient of a small fit (the "plain" workload): latency, launches
        dict(name="fit_plain_1k", kind="fit", points="net", alpha=1, m=10, d=4, R=1, q=1, weights="j^-2"),
        # a higher-order (interlaced) net of moderate size, FP64: column, eigenvalues, solve, MLL and gradient
        dict(name="honet_16k_f64", kind="honet", net_alpha=2, alpha=2, m=14, d=6, R=4, q=1, precision="f64"),
        # the paper's RQMC example: corner-peak Genz function, d = 50, n = 2^15, R = 10, 99% interval
        dict(name="rqmc_genz50_f64", kind="rqmc", points="net", f="genz_cp", baker=False, d=50, R=10, i0=0, n=1 << 15,
             precision="f64"),
        # standalone column, eigenvalues, refined solve and matrix-vector product of FP32 nets
        dict(name="column_solve_f32", kind="ops", points="net", alpha=2, m=18, d=16, R=16, q=2, refine=1, precision="f32"),
        # an FP64 lattice fit step as one schedule (the "diff" workload, 16 shifts)
        dict(name="lattice18_f64", kind="schedule", precision="f64", weights="1", log_eta=-12.0,
             tasks="lattice m18 d32 a2 R16 q1"),
        # nets of uneven n with 8 right-hand sides each, FP64 (the "batch" workload, fewer instances)
        dict(name="batch8_f64", kind="schedule", precision="f64", weights="0.9^j", log_eta=math.log(1e-8),
             tasks="net m14 d16 a2 R16 q8; net m16 d16 a2 R16 q8; net m17 d16 a2 R8 q8"),
        # lattices and nets of uneven n and d, float-float column (the "mixed" workload, fewer instances)
        dict(name="mixed_f32w", kind="schedule", precision="f32w", weights="j^-2", log_eta=math.log(1e-8),
             tasks="lattice m12 d32 a1 R1 q1; net m13 d8 a2 R1 q1; lattice m16 d128 a1 R1 q1; net m18 d32 a2 R1 q1; "
                   "lattice m19 d8 a1 R1 q1; net m20 d128 a2 R1 q1; lattice m21 d32 a1 R1 q1; net m22 d8 a2 R1 q1"),
        # the benchmark's step: 64 randomizations of n = 2^20, FP32 with one refinement step
        dict(name="solve20_f32", kind="schedule", precision="f32", weights="0.9^j", log_eta=math.log(1e-8),
             tasks="net m20 d16 a2 R64 q1"),
        # doubling a set of 2^19 points: the new half's column and the doubled set's eigenvalues
        dict(name="extend19_f32", kind="extend", points="net", alpha=2, m=19, d=16, R=32, precision="f32"),
        # point generation over a ragged range of positions
        dict(name="points_ragged", kind="points", points="net", order="gray", d=13, R=32, i0=12345, n=1000003),
        # the transforms alone, in place, larger than L2
        dict(name="fwht20_f32", kind="transform", op="fwht", m=20, nvec=64, precision="f32"),
        dict(name="fftbr20_f32", kind="transform", op="fftbr", m=20, nvec=32, precision="f32"),
    ]


def _log2(rng, lo, hi):
    """An integer of [lo, hi], uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["fit", "honet", "rqmc", "ops", "schedule", "schedule", "extend", "points", "transform"])
    if kind == "fit":
        points = rng.choice(["net", "lattice"])
        return dict(kind=kind, points=points, alpha=rng.randint(1, 3 if points == "net" else 2), m=rng.randint(9, 16),
                    d=_log2(rng, 2, 40), R=_log2(rng, 1, 6), q=_log2(rng, 1, 5), weights=rng.choice(["j^-2", "0.9^j"]))
    if kind == "honet":
        return dict(kind=kind, net_alpha=rng.randint(2, 4), alpha=rng.randint(1, 3), m=rng.randint(10, 17),
                    d=_log2(rng, 2, 20), R=_log2(rng, 1, 6), q=_log2(rng, 1, 3), precision=rng.choice(["f64", "f32"]))
    if kind == "rqmc":
        f = rng.choice(INTEGRANDS)
        d = {"simple1": 1, "simple2": 2, "oakley": 2}.get(f) or _log2(rng, 2, 100)
        return dict(kind=kind, points=rng.choice(["net", "lattice"]), f=f, baker=rng.random() < 0.5, d=d, R=_log2(rng, 2, 40),
                    i0=rng.choice([0, 0, rng.randint(1, 1 << 20)]), n=_log2(rng, 1000, 1 << 19),
                    precision=rng.choice(["f64", "f32"]))
    if kind == "ops":
        points, m = rng.choice(["net", "lattice"]), rng.randint(9, 20)
        return dict(kind=kind, points=points, alpha=rng.randint(1, 4 if points == "net" else 2), m=m,
                    d=_log2(rng, 2, 40), R=min(_log2(rng, 1, 20), max(1, (1 << 22) >> m)), q=_log2(rng, 1, 4), refine=rng.randint(0, 1),
                    precision=rng.choice(["f64", "f32"]))
    if kind == "schedule":
        precision = rng.choice(["f64", "f32", "f32w"])
        tasks = []
        for _ in range(rng.randint(1, 3)):
            points = rng.choice(["net", "lattice"])
            m, d = rng.randint(12, 18 if precision == "f64" else 20), _log2(rng, 4, 64)
            room = (1 << 23) if precision == "f64" else (1 << 28)  # points x dimensions of one task
            R = max(1, min(_log2(rng, 1, 40), room // (d << m)))
            tasks.append("%s m%d d%d a%d R%d q%d" % (points, m, d, rng.randint(1, 3 if points == "net" else 2), R,
                                                     _log2(rng, 1, 8) if precision == "f64" else _log2(rng, 1, 3)))
        return dict(kind=kind, precision=precision, weights="0.9^j" if precision == "f64" else "j^-2",
                    log_eta=math.log(1e-3 if precision == "f32" else 1e-8), tasks="; ".join(tasks))
    if kind == "extend":
        points = rng.choice(["net", "lattice"])
        m = rng.randint(11, 20)
        return dict(kind=kind, points=points, alpha=rng.randint(1, 2), m=m, d=_log2(rng, 2, 40),
                    R=min(_log2(rng, 1, 40), max(1, (1 << 24) >> m)), precision=rng.choice(["f64", "f32"]))
    if kind == "points":
        d, R = _log2(rng, 1, 120), _log2(rng, 1, 60)
        n = min(_log2(rng, 1000, 1 << 21), max(1000, (1 << 29) // (d * R)))
        return dict(kind=kind, points=rng.choice(["net", "lattice"]), order=rng.choice(["gray", "natural"]), d=d, R=R,
                    i0=rng.choice([0, rng.randint(1, 1 << 22)]), n=n)
    op, precision, m = rng.choice(["fwht", "fftbr", "ifftbr"]), rng.choice(["f32", "f64"]), rng.randint(8, 21)
    return dict(kind="transform", op=op, m=m, nvec=_log2(rng, 1, max(1, (1 << 25) >> m)), precision=precision)


# ------------------------------------------------------------------- inputs, from the seed alone
def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed((seed * 1000003 + salt) % (1 << 62))


def _words(g, *shape):
    return torch.randint(0, 1 << 32, shape, dtype=torch.int64, device="cuda", generator=g)


def _i32(x):
    return torch.where(x >= 1 << 31, x - (1 << 32), x).to(torch.int32).contiguous()


def _net_columns(seed, R, d):
    """(R, d, 32) scrambled generator columns S C over GF(2), S unit lower triangular, C unit upper
    triangular (dimension 1 the identity), bit 31 - t = digit t; and (R, d) shifts."""
    g = _gen(seed, 1)
    bits = lambda *s: torch.randint(0, 2, s, device="cuda", generator=g).to(F32)  # noqa: E731
    eye = torch.eye(32, device="cuda")
    C = torch.triu(bits(d, 32, 32), 1) + eye
    C[0] = eye
    S = torch.tril(bits(R, d, 32, 32), -1) + eye
    digits = (S @ C).remainder(2).to(torch.int64)  # [t, k]
    shift = (31 - torch.arange(32, device="cuda")).view(32, 1)
    return (digits << shift).sum(dim=2), _words(g, R, d)


def _lattice_vector(seed, R, d, m):
    g = _gen(seed, 2)
    return 2 * torch.randint(0, 1 << (m - 1), (d,), dtype=torch.int64, device="cuda", generator=g) + 1, _words(g, R, d)


def _positions(i0, n):
    return torch.arange(i0, i0 + n, dtype=torch.int64, device="cuda")


def _brev(i, bits):
    r = torch.zeros_like(i)
    for b in range(bits):
        r |= ((i >> b) & 1) << (bits - 1 - b)
    return r


def _net_words(cols, order, i):
    """XOR of the columns (digits last) selected by the digits of i (natural) or of its Gray code."""
    v = i ^ (i >> 1) if order == "gray" else i
    X = torch.zeros(i.shape, dtype=torch.int64, device="cuda")
    for k in range(int(i[-1]).bit_length()):
        X ^= cols[k] * ((v >> k) & 1)
    return X


def _diff(ps, r, j, i):
    """The 32-digit difference word of points i and 0 in dimension j (the shift cancels)."""
    if ps["points"] == "net":
        return _net_words(ps["C"][r, j], ps["order"], i)
    return (_brev(i, 32) * ps["g"][j]) & M32


def _point(ps, r, j, i):
    w = _diff(ps, r, j, i)
    return w ^ ps["D"][r, j] if ps["points"] == "net" else (w + ps["D"][r, j]) & M32


def _points_of(seed, points, d, R, m, order="gray"):
    if points == "net":
        C, D = _net_columns(seed, R, d)
        return dict(points=points, order=order, C=C, D=D, d=d, R=R)
    g, D = _lattice_vector(seed, R, d, m)
    return dict(points=points, order="natural", g=g, D=D, d=d, R=R)


def _handle(ps):
    """The framework's point set, and the device arrays that it points to."""
    D = _i32(ps["D"])
    if ps["points"] == "net":
        Ct = _i32(ps["C"])
        return qk.pointset(qk.QK_NET_B2, ps["d"], ps["R"], Ct=Ct, D=D, order=qk.QK_GRAY if ps["order"] == "gray" else qk.QK_NATURAL), [Ct, D]
    g = _i32(ps["g"])
    return qk.pointset(qk.QK_LATTICE, ps["d"], ps["R"], g=g, D=D), [g, D]


def _weights(text, d):
    j = torch.arange(1, d + 1, dtype=F64, device="cuda")
    return {"j^-2": 1.0 / j ** 2, "0.9^j": 0.9 ** j, "1": torch.ones_like(j)}[text].contiguous()


def _rhs(seed, ps, m, q, dtype):
    """(R, q, n) right-hand sides: f(x) = prod_j (1 + (x_j - 1/2)/j^2) and noise of 1e-3."""
    n, g = 1 << m, _gen(seed, 3)
    y = torch.empty((ps["R"], q, n), dtype=dtype, device="cuda")
    i = _positions(0, n)
    for r in range(ps["R"]):
        f = torch.ones(n, dtype=F64, device="cuda")
        for j in range(min(ps["d"], 4)):  # later factors are within 1/32 of one
            f *= 1.0 + (_point(ps, r, j, i).to(F64) * 2.0 ** -32 - 0.5) / (j + 1) ** 2
        for k in range(q):
            noise = torch.randn(n, dtype=F32, device="cuda", generator=g).to(F64)
            y[r, k] = (f * (1.0 + 0.1 * k) + 1e-3 * noise).to(dtype)
    return y


def _dtype(precision):
    return F64 if precision == "f64" else F32


# ------------------------------------------------------------------- what a program has in hand
def prepare(case, seed):
    return {"fit": _prepare_fit, "honet": _prepare_honet, "rqmc": _prepare_rqmc, "ops": _prepare_ops,
            "schedule": _prepare_schedule, "extend": _prepare_extend, "points": _prepare_points,
            "transform": _prepare_transform}[case["kind"]](case, seed)


def run(state):
    return state["run"](state)


def exact(case, seed):
    return {"fit": _exact_fit, "honet": _exact_honet, "rqmc": _exact_rqmc, "ops": _exact_ops,
            "schedule": _exact_schedule, "extend": _exact_extend, "points": lambda c, s: None,
            "transform": _exact_transform}[case["kind"]](case, seed)


def _family(points):
    return qk.QK_DSI if points == "net" else qk.QK_SI


# one evaluation of the marginal log-likelihood and posterior mean with the gradient of both
def _fit_params(c):
    return _weights(c["weights"], c["d"]), torch.linspace(-0.3, 0.2, c["d"], dtype=F64, device="cuda"), math.log(1e-6)


def _prepare_fit(c, seed):
    ps = _points_of(seed, c["points"], c["d"], c["R"], c["m"])
    h, keep = _handle(ps)
    gamma, ls, le = _fit_params(c)
    params = [gamma.clone().requires_grad_(), ls.clone().requires_grad_(),
              torch.tensor(le, dtype=F64, device="cuda", requires_grad=True)]
    return dict(run=_run_fit, params=params, y=_rhs(seed, ps, c["m"], c["q"], F64), ps=h, keep=keep,
                spec=(_family(c["points"]), c["alpha"], c["m"]))


def _run_fit(s):
    fam, alpha, m = s["spec"]
    mll, mean = mll_and_mean(*s["params"], s["y"], s["ps"], fam, alpha, m)
    grads = torch.autograd.grad(mll.sum() + mean.sum(), s["params"])
    return [mll.detach(), mean.detach(), *grads]


# column, eigenvalues, solve and matrix-vector product, call by call
def _prepare_ops(c, seed):
    ps = _points_of(seed, c["points"], c["d"], c["R"], c["m"])
    h, keep = _handle(ps)
    dt, n, fam = _dtype(c["precision"]), 1 << c["m"], _family(c["points"])
    w = _weights("j^-2", c["d"])
    y = _rhs(seed, ps, c["m"], c["q"], dt)
    need = [qk.workspace_bytes(op, fam, c["m"], c["R"], c["q"], dt) for op in (qk.OP_EIGS, qk.OP_SOLVE, qk.OP_MATVEC)]
    return dict(run=_run_ops, ps=h, keep=keep + [w], kern=qk.kernel(fam, c["alpha"], w, 1.0), y=y, c=torch.empty_like(y),
                u=torch.empty_like(y), col=torch.empty((c["R"], n), dtype=dt, device="cuda"),
                lam=torch.empty((c["R"], n), dtype=F64, device="cuda"), ws=qk.workspace(max(need)),
                status=torch.zeros(1, dtype=torch.int32, device="cuda"), fam=fam, m=c["m"], R=c["R"], refine=c["refine"])


def _run_ops(s):
    qk.kernel_col(s["ps"], s["kern"], 0, s["R"], s["m"], s["col"], form=qk.QK_COL_P)
    qk.eigs(s["fam"], s["m"], s["col"], s["lam"], eta=1e-3, form=qk.QK_COL_P, ws=s["ws"], status=s["status"])
    qk.solve(s["fam"], s["m"], s["lam"], s["y"], s["c"], refine_steps=s["refine"], ws=s["ws"])
    qk.matvec(s["fam"], s["m"], s["lam"], s["y"], s["u"], ws=s["ws"])
    return [s["lam"], s["c"], s["u"]]


# a planned schedule: solve, MLL and gradient of every task
def _tasks(c):
    out = []
    for text in c["tasks"].split("; "):
        points, *rest = text.split()
        out.append((points, *[int(v[1:]) for v in rest]))  # points, m, d, alpha, R, q
    return out


def _prepare_schedule(c, seed):
    dt = {"f64": F64, "f32": F32, "f32w": qk.F32W}[c["precision"]]
    data = qk.data_dtype(dt)
    tasks, keep, outs = [], [], []
    for t, (points, m, d, alpha, R, q) in enumerate(_tasks(c)):
        ps = _points_of(seed + 7919 * t, points, d, R, m)
        h, k = _handle(ps)
        w = _weights(c["weights"], d)
        y = _rhs(seed + 7919 * t, ps, m, q, data)
        sol = torch.empty_like(y)
        out = torch.empty((R, q, qk.QK_MLL_NOUT), dtype=F64, device="cuda")
        grad = torch.empty((R, q, 2 * d + 2), dtype=F64, device="cuda")
        tasks.append(qk.Task(h, qk.kernel(_family(points), alpha, w, 1.0), m, q, math.exp(c["log_eta"]), y.data_ptr(),
                             sol.data_ptr(), None, out.data_ptr(), grad.data_ptr()))
        keep += [*k, w, y]
        outs += [sol, out, grad]
    ws = qk.workspace(qk.batch_workspace_bytes(tasks, dt))
    qk.batch_plan(tasks, dt, 0 if c["precision"] == "f64" else 1, ws)
    return dict(run=_run_schedule, ws=ws, outs=outs, keep=keep, status=torch.zeros(1, dtype=torch.int32, device="cuda"))


def _run_schedule(s):
    qk.batch_run(s["ws"], s["status"])
    return s["outs"]


# the eigenvalues of a doubled point set from those of its first half
def _prepare_extend(c, seed):
    ps = _points_of(seed, c["points"], c["d"], c["R"], c["m"] + 1)
    h, keep = _handle(ps)
    dt, n, fam = _dtype(c["precision"]), 1 << c["m"], _family(c["points"])
    w = _weights("0.9^j", c["d"])
    kern = qk.kernel(fam, c["alpha"], w, 1.0)
    col = torch.empty((c["R"], n), dtype=dt, device="cuda")
    old = torch.empty((c["R"], n), dtype=F64, device="cuda")
    ws = qk.workspace(qk.workspace_bytes(qk.OP_EIGS, fam, c["m"], c["R"], 1, dt))
    qk.kernel_col(h, kern, 0, c["R"], c["m"], col, form=qk.QK_COL_P)
    qk.eigs(fam, c["m"], col, old, eta=1e-3, form=qk.QK_COL_P, ws=ws)
    return dict(run=_run_extend, ps=h, keep=keep + [w], kern=kern, col=col, old=old, ws=ws, fam=fam, m=c["m"], R=c["R"],
                lam=torch.empty((c["R"], 2 * n), dtype=F64, device="cuda"))


def _run_extend(s):
    qk.kernel_col_at(s["ps"], s["kern"], 0, s["R"], 1 << s["m"], s["m"], s["col"], form=qk.QK_COL_P)
    qk.eigs_extend(s["fam"], s["m"], s["col"], s["old"], s["lam"], eta=1e-3, form=qk.QK_COL_P, ws=s["ws"])
    return s["lam"]


# a higher-order net: column, eigenvalues, solve, MLL and gradient
def _ho_columns(seed, R, d, net_alpha):
    """(R, d, 32) interlaced 64-digit columns as (high, low) words: digit t of matrix j is digit
    t // alpha of matrix alpha j + t mod alpha of an alpha d-dimensional net; and the shifts."""
    C, _ = _net_columns(seed, R, net_alpha * d)
    C = C.view(R, d, net_alpha, 32)
    words = [torch.zeros((R, d, 32), dtype=torch.int64, device="cuda") for _ in range(2)]
    for t in range(64):
        words[t // 32] |= ((C[:, :, t % net_alpha] >> (31 - t // net_alpha)) & 1) << (31 - t % 32)
    return words


def _prepare_honet(c, seed):
    hi, lo = _ho_columns(seed, c["R"], c["d"], c["net_alpha"])
    Chat = ((hi << 32) | lo).contiguous()
    dt, n, R = _dtype(c["precision"]), 1 << c["m"], c["R"]
    w = _weights("0.9^j", c["d"])
    y = _honet_rhs(c, seed, dt)
    need = max(qk.workspace_bytes(qk.OP_EIGS, qk.QK_DSI, c["m"], R, 1, dt),
               qk.workspace_bytes(qk.OP_SOLVE, qk.QK_DSI, c["m"], R, c["q"], dt),
               qk.workspace_bytes(qk.OP_MLL, qk.QK_DSI, c["m"], R, c["q"], dt, c["d"]))
    return dict(run=_run_honet, ps=qk.ho_pointset(c["d"], R, Chat), keep=[Chat, w], kern=qk.kernel(qk.QK_DSI, c["alpha"], w, 1.0),
                y=y, c=torch.empty_like(y), col=torch.empty((R, n), dtype=dt, device="cuda"),
                lam=torch.empty((R, n), dtype=F64, device="cuda"), ws=qk.workspace(need), m=c["m"], R=R, q=c["q"],
                out=torch.empty((R, c["q"], qk.QK_MLL_NOUT), dtype=F64, device="cuda"),
                grad=torch.empty((R, c["q"], 2 * c["d"] + 2), dtype=F64, device="cuda"),
                status=torch.zeros(1, dtype=torch.int32, device="cuda"))


def _honet_rhs(c, seed, dtype):
    g, x = _gen(seed, 4), torch.linspace(0, 1, 1 << c["m"], dtype=F64, device="cuda")
    y = torch.randn((c["R"], c["q"], 1 << c["m"]), dtype=F32, device="cuda", generator=g).to(F64)
    return (0.1 * y + torch.cos(3.0 * x)).to(dtype).contiguous()


def _run_honet(s):
    qk.kernel_col_ho(s["ps"], s["kern"], 0, s["R"], s["m"], s["col"], form=qk.QK_COL_P)
    qk.eigs(qk.QK_DSI, s["m"], s["col"], s["lam"], eta=1e-2, form=qk.QK_COL_P, ws=s["ws"], status=s["status"])
    qk.solve(qk.QK_DSI, s["m"], s["lam"], s["y"], s["c"], ws=s["ws"])
    qk.mll_ho(s["ps"], s["kern"], 0, s["R"], s["m"], s["q"], s["lam"], s["y"], s["out"], s["grad"], ws=s["ws"])
    return [s["lam"], s["c"], s["out"], s["grad"]]


# a randomized quasi-Monte Carlo estimate with its interval
def _prepare_rqmc(c, seed):
    ps = _points_of(seed, c["points"], c["d"], c["R"], 20)
    h, keep = _handle(ps)
    y = torch.empty((c["R"], c["n"]), dtype=_dtype(c["precision"]), device="cuda")
    return dict(run=_run_rqmc, ps=h, keep=keep, y=y, out=torch.empty(4 + c["R"], dtype=F64, device="cuda"), c=c)


def _run_rqmc(s):
    c = s["c"]
    qk.integrand(s["ps"], 0, c["R"], c["i0"], c["n"], c["f"], s["y"], baker=c["baker"])
    return [s["y"], qk.rqmc(s["y"], 0.01, out=s["out"])]


# points as 32-bit words
def _prepare_points(c, seed):
    ps = _points_of(seed, c["points"], c["d"], c["R"], 20, c["order"] if c["points"] == "net" else "natural")
    h, keep = _handle(ps)
    return dict(run=_run_points, ps=h, keep=keep, R=c["R"], i0=c["i0"], n=c["n"],
                X=torch.empty((c["R"], c["n"], c["d"]), dtype=torch.int32, device="cuda"))


def _run_points(s):
    return qk.gen_points(s["ps"], 0, s["R"], s["i0"], s["n"], s["X"])


# batched transforms in place (orthonormal: repeated passes keep the data's size)
def _transform_data(c, seed):
    per = (1 if c["op"] == "fwht" else 2) << c["m"]
    return torch.randn((c["nvec"], per), dtype=_dtype(c["precision"]), device="cuda", generator=_gen(seed, 5))


def _prepare_transform(c, seed):
    return dict(run=_run_transform, x=_transform_data(c, seed), ws=qk.fwht_workspace(c["nvec"]), m=c["m"], op=c["op"])


def _run_transform(s):
    if s["op"] == "fwht":
        return qk.fwht_ws(s["m"], s["x"], ws=s["ws"])
    return qk.fftbr_ws(s["m"], s["x"], inverse=s["op"] == "ifftbr", ws=s["ws"])


# ------------------------------------------------------------------- what a pass cannot do without
def _schedule_work(points, m, d, alpha, R, q, s):
    n, v = R << m, (R * q) << m
    # y in, c out; column and gradient sweeps, transforms of the column, y, c and g
    return 2 * s * v, n * d * 8 + v * (d * 4 + 12) + n * d * 6 + (n + 3 * v) * m * (1 if points == "net" else 2.5)


def work(c):
    s = 8 if c.get("precision", "f64") == "f64" else 4
    k = c["kind"]
    if k == "fit":
        b, f = _schedule_work(c["points"], c["m"], c["d"], c["alpha"], c["R"], c["q"], 8)
        return {"bytes": b // 2, "flops": f}
    if k == "schedule":
        parts = [_schedule_work(*t, s) for t in _tasks(c)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    n = c["R"] << c["m"] if "m" in c and "R" in c else 0
    if k == "honet":
        b, f = _schedule_work("net", c["m"], c["d"], c["alpha"], c["R"], c["q"], s)
        return {"bytes": b + 8 * n, "flops": f}
    if k == "ops":
        v = n * c["q"]
        stages = c["m"] * (1 if c["points"] == "net" else 2.5)
        return {"bytes": 8 * n + 3 * s * v, "flops": n * c["d"] * 8 + (n + (3 + 4 * c["refine"]) * v) * stages}
    if k == "extend":
        return {"bytes": 24 * n, "flops": n * c["d"] * 8 + n * c["m"] * (1 if c["points"] == "net" else 2.5)}
    if k == "rqmc":
        v = c["R"] * c["n"]
        return {"bytes": s * v, "flops": v * (3 * c["d"] + 20)}
    if k == "points":
        v = c["R"] * c["n"] * c["d"]
        return {"bytes": 4 * v, "flops": v}
    v = c["nvec"] << c["m"]
    return {"bytes": 2 * s * v * (1 if c["op"] == "fwht" else 2), "flops": v * c["m"] * (1 if c["op"] == "fwht" else 5)}


# ------------------------------------------------------------------- the same in plain torch, 64 bits
def _dsi(alpha, x, beta, digits):
    """The digitally-shift-invariant kernels at x = z 2^-t (beta = -floor(log2 x), 0 at x = 0)."""
    t1 = torch.where(beta > 0, torch.exp2(-beta), torch.zeros_like(x))
    if alpha == 1:
        return torch.where(beta > 0, 1.0 - 3.0 * t1, torch.ones_like(x))
    if alpha == 2:
        return 1.5 - beta * x - 2.5 * t1
    if alpha == 3:
        return -1.0 + beta * x * x - 5.0 * (1.0 - t1) * x + 43.0 / 18.0 * (1.0 - t1 * t1)
    return (-1.0 - 2.0 / 3.0 * beta * x ** 3 + 5.0 * (1.0 - t1) * x * x - 43.0 / 9.0 * (1.0 - t1 * t1) * x
            + 701.0 / 294.0 * (1.0 - t1 ** 3) - beta * digits / 24.0)


def _factor(ps, alpha, z):
    x = z.to(F64) * 2.0 ** -32
    if ps["points"] == "lattice":
        b = x * (1.0 - x)
        return math.pi ** 2 / 3 - 2 * math.pi ** 2 * b if alpha == 1 else math.pi ** 4 / 45 - 2 * math.pi ** 4 / 3 * b * b
    beta = torch.where(z > 0, 33.0 - torch.frexp(z.to(F64))[1].to(F64), torch.zeros_like(x))
    digits = None
    if alpha == 4:
        digits = torch.zeros_like(x)
        for a in range(24):
            digits += ((z >> (31 - a)) & 1).to(F64) * 8.0 ** -a
    return _dsi(alpha, x, beta, digits)


def _factor64(alpha, hi, lo):
    top = torch.where(hi > 0, hi, lo)
    e = torch.frexp(top.to(F64))[1].to(F64)
    beta = torch.where(hi > 0, 33.0 - e, torch.where(lo > 0, 65.0 - e, torch.zeros_like(e)))
    return _dsi(alpha, hi.to(F64) * 2.0 ** -32 + lo.to(F64) * 2.0 ** -64, beta, None)


def _column(factors, w):
    """prod_j (1 + c_j K_j) - 1 over the dimensions' factors."""
    p = None
    for j, K in enumerate(factors()):
        a = w[j] * K
        p = a if p is None else p + a + p * a
    return p


def _fwht(x):
    n, shape, h = x.shape[-1], x.shape, 1
    while h < n:
        x = x.reshape(-1, n // (2 * h), 2, h)
        x = torch.stack((x[:, :, 0] + x[:, :, 1], x[:, :, 0] - x[:, :, 1]), dim=2)
        h *= 2
    return x.reshape(shape)


def _forward(points, x):
    """The unnormalised transform over the last axis: Hadamard, or the DFT of the data in linear order."""
    if points == "net":
        return _fwht(x)
    n = x.shape[-1]
    return torch.fft.fft(x[..., _brev(_positions(0, n), n.bit_length() - 1)])


def _inverse(points, X):
    """Its transpose back to the points' order, real part, unnormalised."""
    if points == "net":
        return _fwht(X)
    n = X.shape[-1]
    return (torch.fft.ifft(X) * n).real[..., _brev(_positions(0, n), n.bit_length() - 1)]


def _spectral(points, factors, w, eta, Y, with_grad=True):
    """For one randomization (zeta = 1) and right-hand sides Y (q, n): eigenvalues, solutions, MLL pieces
    (q, 5) and gradient blocks (q, 2 d + 2)."""
    n, d = Y.shape[-1], len(w)
    p = _column(factors, w)
    lam = _forward(points, p)
    lam = (lam.real if lam.is_complex() else lam).clone()
    lam[0] += n
    lam += eta
    T = _forward(points, Y)
    a = (T.abs() ** 2) / n / lam
    sol = _inverse(points, T / lam) / n
    quad, logdet, lam0, sy = a.sum(-1), lam.log().sum(), n + p.sum() + eta, Y.sum(-1)
    out = torch.stack((quad, logdet.expand_as(quad), -0.5 * (quad + logdet + n * math.log(2 * math.pi)), sy / lam0,
                       ((p.sum() + eta) / lam0).expand_as(quad)), dim=-1)
    if not with_grad:
        return lam, sol, out, None
    g = 0.5 * (a - 1.0) / lam
    u = _inverse(points, g)
    mfac = -sy / lam0 ** 2
    grad = torch.empty((Y.shape[0], 2 * d + 2), dtype=F64, device="cuda")
    for j, K in enumerate(factors()):
        dk = (1.0 + p) * K / (1.0 + w[j] * K)
        grad[:, j] = (u * dk).sum(-1)
        grad[:, d + 1 + j] = mfac * dk.sum()
    grad[:, d] = g.sum(-1)
    grad[:, 2 * d + 1] = mfac
    return lam, sol, out, grad


def _factors_of(ps, alpha, r, i):
    return lambda: (_factor(ps, alpha, _diff(ps, r, j, i)) for j in range(ps["d"]))


def _exact_all(ps, alpha, m, w, eta, y):
    i = _positions(0, 1 << m)
    parts = [_spectral(ps["points"], _factors_of(ps, alpha, r, i), w, eta, y[r].to(F64)) for r in range(ps["R"])]
    return [torch.stack([p[k] for p in parts]) for k in range(4)]


def _exact_fit(c, seed):
    ps = _points_of(seed, c["points"], c["d"], c["R"], c["m"])
    gamma, ls, le = _fit_params(c)
    w, eta, d = gamma * torch.exp(ls), math.exp(le), c["d"]
    _, _, out, grad = _exact_all(ps, c["alpha"], c["m"], w, eta, _rhs(seed, ps, c["m"], c["q"], F64))
    dw = (grad[..., :d] + grad[..., d + 1:2 * d + 1]).sum((0, 1))
    return [out[..., 2], out[..., 3], dw * torch.exp(ls), dw * w, (grad[..., d] + grad[..., 2 * d + 1]).sum() * eta]


def _exact_ops(c, seed):
    ps = _points_of(seed, c["points"], c["d"], c["R"], c["m"])
    w, i, n = _weights("j^-2", c["d"]), _positions(0, 1 << c["m"]), 1 << c["m"]
    y = _rhs(seed, ps, c["m"], c["q"], _dtype(c["precision"])).to(F64)
    lams, sols, mats = [], [], []
    for r in range(c["R"]):
        lam, sol, _, _ = _spectral(c["points"], _factors_of(ps, c["alpha"], r, i), w, 1e-3, y[r], with_grad=False)
        lams.append(lam)
        sols.append(sol)
        mats.append(_inverse(c["points"], _forward(c["points"], y[r]) * lam) / n)
    return [torch.stack(lams), torch.stack(sols), torch.stack(mats)]


def _exact_schedule(c, seed):
    outs = []
    for t, (points, m, d, alpha, R, q) in enumerate(_tasks(c)):
        ps = _points_of(seed + 7919 * t, points, d, R, m)
        y = _rhs(seed + 7919 * t, ps, m, q, _dtype(c["precision"]))
        outs += _exact_all(ps, alpha, m, _weights(c["weights"], d), math.exp(c["log_eta"]), y)[1:]
    return outs


def _exact_extend(c, seed):
    ps = _points_of(seed, c["points"], c["d"], c["R"], c["m"] + 1)
    w, n = _weights("0.9^j", c["d"]), 2 << c["m"]
    i, lams = _positions(0, n), []
    for r in range(c["R"]):
        lam = _forward(c["points"], _column(_factors_of(ps, c["alpha"], r, i), w))
        lam = (lam.real if lam.is_complex() else lam).clone()
        lam[0] += n
        lams.append(lam + 1e-3)
    return torch.stack(lams)


def _exact_honet(c, seed):
    hi, lo = _ho_columns(seed, c["R"], c["d"], c["net_alpha"])
    i, w, y = _positions(0, 1 << c["m"]), _weights("0.9^j", c["d"]), _honet_rhs(c, seed, _dtype(c["precision"])).to(F64)
    parts = []
    for r in range(c["R"]):
        def factors(r=r):
            return (_factor64(c["alpha"], _net_words(hi[r, j], "gray", i), _net_words(lo[r, j], "gray", i)) for j in range(c["d"]))
        parts.append(_spectral("net", factors, w, 1e-2, y[r]))
    return [torch.stack([p[k] for p in parts]) for k in range(4)]


def _exact_rqmc(c, seed):
    ps, d = _points_of(seed, c["points"], c["d"], c["R"], 20), c["d"]
    i, rows, j1 = _positions(c["i0"], c["n"]), [], torch.arange(1, d + 1, dtype=F64, device="cuda")
    ct = torch.exp(j1 * math.log(1e-8) / d) if c["f"] == "genz_osc" else 1.0 / j1 ** 2
    ct = ct * ((4.5 if c["f"] == "genz_osc" else 0.25) / ct.sum())
    for r in range(c["R"]):
        xs, lin, prod = [], torch.zeros(c["n"], dtype=F64, device="cuda"), torch.ones(c["n"], dtype=F64, device="cuda")
        for j in range(d):
            x = _point(ps, r, j, i).to(F64) * 2.0 ** -32
            x = 1.0 - 2.0 * (x - 0.5).abs() if c["baker"] else x
            if j < 2:
                xs.append(x)
            a = (j - 1) / 2.0
            prod = prod * ((4.0 * x - 2.0).abs() - a) / (1.0 + a) if c["f"] == "gfun" else prod
            lin = lin + ct[j] * x
        if c["f"] == "simple1":
            y = xs[0] * torch.exp(xs[0]) - 1.0
        elif c["f"] == "simple2":
            y = xs[1] * torch.exp(xs[0] * xs[1]) / (math.e - 2.0) - 1.0
        elif c["f"] == "oakley":
            t = [(x - 0.5) / 50.0 for x in xs]
            y = 5.0 + t[0] + t[1] + 2.0 * torch.cos(t[0]) + 2.0 * torch.cos(t[1])
        else:
            y = {"gfun": lambda: prod, "genz_osc": lambda: torch.cos(lin), "genz_cp": lambda: (1.0 + lin) ** -(d + 1.0)}[c["f"]]()
        rows.append(y)
    return [torch.stack(rows), None]  # the interval's parts follow from these values and a quantile


def _exact_transform(c, seed):
    x, n = _transform_data(c, seed).to(F64), 1 << c["m"]
    rows = []
    for v in x.split(max(1, (1 << 23) // n)):
        if c["op"] == "fwht":
            rows.append(_fwht(v) / math.sqrt(n))
            continue
        z = torch.view_as_complex(v.view(-1, n, 2))
        perm = _brev(_positions(0, n), c["m"])
        z = torch.fft.fft(z[:, perm]) / math.sqrt(n) if c["op"] == "fftbr" else (torch.fft.ifft(z) * math.sqrt(n))[:, perm]
        rows.append(torch.view_as_real(z).reshape(-1, 2 * n))
    return torch.cat(rows)
