"""The work a user of the library has it do, as cases that can be timed.

Each case is one kind of call through the public binding (``Context``): a QR
factorization (FP64 or FP32, FULL or PANEL T), forming Q or applying it, a
least-squares solve (FP64 or mixed precision), a batch of uneven tall-skinny
QRs, or a burst of requests to the least-squares server.  Shapes and
distributions are those of the repository's benchmark, tests and workload
generators, and odd ones between them.

Matrices are column-major; columns are Gaussian, graded over ``decades``
decades (column j scaled by 10**(-decades j / n)).  The library factors in
place, so a pass copies the inputs into the working buffers first, as a
program does that factors one matrix after another.
"""

import math

import torch

import paper_1805_05278_gb300 as gb

DEV = "cuda:0"


# ------------------------------------------------------------------ cases

def listed():
    return [
        # One small tall-skinny matrix with Algorithm 2's full T, and its
        # Q^T b: a call where launches and the panel's chain are everything.
        dict(name="qr_full_1024x128", kind="factor", dtype="f64", layout="full", m=1024, n=128, decades=0.0, pad=0, rhs=1),
        # A ragged mid-size matrix with the full T and an odd leading dimension.
        dict(name="qr_full_4099x1031", kind="factor", dtype="f64", layout="full", m=4099, n=1031, decades=2.0, pad=3, rhs=0),
        # The tall benchmark matrix, PANEL layout.
        dict(name="qr_panel_32768x2048", kind="factor", dtype="f64", layout="panel", m=32768, n=2048, decades=6.0, pad=0, rhs=0),
        # The square benchmark matrix, PANEL layout: the headline.
        dict(name="qr_panel_8192x8192", kind="factor", dtype="f64", layout="panel", m=8192, n=8192, decades=6.0, pad=0, rhs=0),
        # The FP32 factorization of a single matrix.
        dict(name="qr_f32_16384x1000", kind="factor", dtype="f32", layout="panel", m=16384, n=1000, decades=1.0, pad=0, rhs=0),
        # The thin Q of a factored matrix, ragged rows (apply in reverse order).
        dict(name="form_q_16001x1000", kind="apply", op="form_q", m=16001, n=1000, nrhs=1000, decades=0.0),
        # A mid-size FP64 least-squares solve out of the serving range, ragged.
        dict(name="ls_fp64_20011x523", kind="ls", prec="fp64", m=20011, n=523, decades=3.0),
        # The tall mixed-precision least-squares benchmark.
        dict(name="ls_mixed_32768x2048", kind="ls", prec="mixed", m=32768, n=2048, decades=6.0),
        # The square mixed-precision solve (a linear system).
        dict(name="ls_mixed_8192x8192", kind="ls", prec="mixed", m=8192, n=8192, decades=0.0),
        # The batched benchmark: 2000 uneven tall-skinny FP64 matrices.
        dict(name="batched_f64_2000", kind="batched", dtype="f64", count=2000, m_hi=16384, n_hi=256, shapes=20),
        # The same kind of batch in FP32, smaller and shorter matrices.
        dict(name="batched_f32_500", kind="batched", dtype="f32", count=500, m_hi=8192, n_hi=200, shapes=21),
        # A burst of least-squares requests to the server, precision chosen by it.
        dict(name="serve_48", kind="serve", count=48, m_hi=65536, n_hi=1024, shapes=30),
    ]


def _log_int(rng, lo, hi):
    return int(math.floor(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def _tall(rng, m_lo, m_hi, n_lo, n_hi, elems=1 << 26, ratio=1.0):
    while True:
        m, n = _log_int(rng, m_lo, m_hi), _log_int(rng, n_lo, n_hi)
        if m >= ratio * n and m * n <= elems:
            return m, n


def draw(rng):
    kind = rng.choice(["factor", "factor", "factor32", "apply", "ls64", "mixed", "batched", "serve"])
    if kind in ("factor", "factor32"):
        m, n = _tall(rng, 256, 65536, 16, 6000, elems=1 << 25, ratio=2.0 if kind == "factor32" else 1.0)
        layout = rng.choice(["full", "panel", "panel"]) if n <= 2048 else "panel"
        return dict(kind="factor", dtype="f32" if kind == "factor32" else "f64", layout=layout, m=m, n=n,
                    decades=rng.uniform(0.0, 1.0 if kind == "factor32" else 6.0), pad=rng.choice([0, 0, 1, 8]),
                    rhs=rng.choice([0, 1]) if kind == "factor" else 0)
    if kind == "apply":
        op = rng.choice(["form_q", "apply_q", "apply_qt"])
        m, n = _tall(rng, 512, 65536, 16, 3000, elems=1 << 25)
        nrhs = n if op == "form_q" else _log_int(rng, 1, 512)
        return dict(kind="apply", op=op, m=m, n=n, nrhs=nrhs, decades=rng.uniform(0.0, 3.0))
    if kind == "ls64":
        m, n = _tall(rng, 512, 65536, 32, 1024, ratio=1.5)
        return dict(kind="ls", prec="fp64", m=m, n=n, decades=rng.uniform(1.0, 5.0))
    if kind == "mixed":
        m, n = _tall(rng, 2048, 65536, 256, 5000, ratio=1.5)
        return dict(kind="ls", prec="mixed", m=m, n=n, decades=rng.uniform(1.0, 5.0))
    if kind == "batched":
        return dict(kind="batched", dtype=rng.choice(["f64", "f32"]), count=_log_int(rng, 40, 1000),
                    m_hi=_log_int(rng, 1024, 16384), n_hi=_log_int(rng, 32, 256), shapes=rng.randrange(1 << 20))
    return dict(kind="serve", count=rng.randrange(16, 65), m_hi=_log_int(rng, 4096, 65536),
                n_hi=_log_int(rng, 128, 1024), shapes=rng.randrange(1 << 20))


def _shapes(case):
    """(m, n) of every matrix of a batch or burst: m log-uniform, n uniform
    (batch) or log-uniform (requests), n <= m.  FP32 batches and requests are
    overdetermined, as such problems are in use (a nearly square Gaussian
    matrix is ill-conditioned)."""
    import random
    rng = random.Random(case["shapes"])
    ratio = 1.5 if case["kind"] == "serve" else 2.0 if case["dtype"] == "f32" else 1.0
    out = []
    while len(out) < case["count"]:
        if case["kind"] == "batched":
            m, n = _log_int(rng, 256, case["m_hi"]), rng.randint(16, case["n_hi"])
        else:
            m, n = _log_int(rng, 512, case["m_hi"]), _log_int(rng, 32, case["n_hi"])
        if m >= ratio * n:
            out.append((m, n))
    return out


# ----------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _matrix(m, n, decades, g, pad=0, dtype=torch.float64):
    """Column-major m x n view (leading dimension m + pad) of graded Gaussian
    columns."""
    buf = torch.empty((n, m + pad), dtype=torch.float64, device=DEV)
    buf.normal_(generator=g)
    if decades:
        j = torch.arange(n, dtype=torch.float64, device=DEV)
        buf *= (10.0 ** (-decades * j / n))[:, None]
    return buf.to(dtype).T[:m]


def _blank(m, n, pad=0, dtype=torch.float64):
    return torch.zeros((n, m + pad), dtype=dtype, device=DEV).T[:m]


def _ls_problem(m, n, decades, g):
    a = _matrix(m, n, decades, g)
    x = torch.empty(n, dtype=torch.float64, device=DEV).normal_(generator=g)
    e = torch.empty(m, dtype=torch.float64, device=DEV).normal_(generator=g)
    return a, a @ x + 1e-8 * e


def _request_decades(case, k):
    return 1.0 + 4.0 * ((k * 7919 + case["shapes"]) % 97) / 97.0


def _layout(case):
    return gb.GBQR_T_FULL if case.get("layout") == "full" else gb.GBQR_T_PANEL


def _nb(m, n):
    return min(128, n)


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = dict(case=case, ctx=gb.Context(0))
    if kind == "factor":
        dt = torch.float32 if case["dtype"] == "f32" else torch.float64
        m, n = case["m"], case["n"]
        s["A0"] = _matrix(m, n, case["decades"], g, case["pad"], dt)
        s["A"] = _blank(m, n, case["pad"], dt)
        s["T"] = _blank(n if case["layout"] == "full" else _nb(m, n), n, 0, dt)
        if case["rhs"]:
            s["b0"] = _matrix(m, case["rhs"], 0.0, g)
            s["b"] = _blank(m, case["rhs"])
    elif kind == "apply":
        m, n = case["m"], case["n"]
        s["VR"] = _matrix(m, n, case["decades"], g)
        s["T"] = _blank(_nb(m, n), n)
        s["ctx"].factor(s["VR"], s["T"], gb.GBQR_T_PANEL)
        s["B"] = _blank(m, case["nrhs"])
        if case["op"] != "form_q":
            s["B0"] = _matrix(m, case["nrhs"], 0.0, g)
    elif kind == "ls":
        s["A"], s["b"] = _ls_problem(case["m"], case["n"], case["decades"], g)
        s["x"] = torch.zeros(case["n"], dtype=torch.float64, device=DEV)
    elif kind == "batched":
        dt = torch.float32 if case["dtype"] == "f32" else torch.float64
        shapes = _shapes(case)
        s["A0"] = torch.empty(sum(m * n for m, n in shapes), dtype=dt, device=DEV).normal_(generator=g)
        s["A"] = torch.zeros_like(s["A0"])
        s["T"] = torch.zeros(sum(_nb(m, n) * n for m, n in shapes), dtype=dt, device=DEV)
        s["As"], s["Ts"], a, t = [], [], 0, 0
        for m, n in shapes:
            nb = _nb(m, n)
            s["As"].append(s["A"][a:a + m * n].view(n, m).T)
            s["Ts"].append(s["T"][t:t + nb * n].view(n, nb).T)
            a, t = a + m * n, t + nb * n
    else:
        shapes = _shapes(case)
        s["problems"] = [_ls_problem(m, n, _request_decades(case, k), g) for k, (m, n) in enumerate(shapes)]
        s["x"] = torch.zeros(sum(n for _, n in shapes), dtype=torch.float64, device=DEV)
        s["xs"] = list(torch.split(s["x"], [n for _, n in shapes]))
        torch.cuda.synchronize()
        s["ctx"].serve(16)
    return s


# ------------------------------------------------------------------ a pass

def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "factor":
        s["A"].copy_(s["A0"])
        ctx.factor(s["A"], s["T"], _layout(case))
        if not case["rhs"]:
            return s["A"], s["T"]
        s["b"].copy_(s["b0"])
        ctx.apply_qt(s["A"], s["T"], s["b"], _layout(case), 0 if case["layout"] == "full" else _nb(case["m"], case["n"]))
        return s["A"], s["T"], s["b"]
    if kind == "apply":
        nb = _nb(case["m"], case["n"])
        if case["op"] == "form_q":
            ctx.form_q(s["VR"], s["T"], s["B"], gb.GBQR_T_PANEL, nb)
        else:
            s["B"].copy_(s["B0"])
            (ctx.apply_q if case["op"] == "apply_q" else ctx.apply_qt)(s["VR"], s["T"], s["B"], gb.GBQR_T_PANEL, nb)
        return s["B"]
    if kind == "ls":
        ctx.ls_solve(s["A"], s["b"], s["x"], gb.GBQR_FP64 if case["prec"] == "fp64" else gb.GBQR_MIXED_SPLITBF16)
        return s["x"]
    if kind == "batched":
        s["A"].copy_(s["A0"])
        ctx.factor_batched(s["As"], s["Ts"])
        return s["A"], s["T"]
    ids = [ctx.submit(a, b, x, gb.GBQR_PREC_AUTO) for (a, b), x in zip(s["problems"], s["xs"])]
    for r in ids:
        ctx.poll(r, wait=True)
    return s["x"]


# ------------------------------------------------------------------- work

def _qr_flops(m, n):
    return 2.0 * m * n * n - 2.0 * n ** 3 / 3.0


def work(case):
    """Bytes: inputs read once, outputs written once.  Flops: the Householder
    QR count 2 m n^2 - 2 n^3 / 3, and 4 m n - 2 n^2 per vector Q is applied to."""
    kind = case["kind"]
    if kind in ("factor", "apply", "ls"):
        m, n = case["m"], case["n"]
        q1 = 4.0 * m * n - 2.0 * n * n
    if kind == "factor":
        e = 4 if case["dtype"] == "f32" else 8
        t = n if case["layout"] == "full" else _nb(m, n)
        return {"bytes": e * (2.0 * m * n + t * n) + 16.0 * m * case["rhs"], "flops": _qr_flops(m, n) + q1 * case["rhs"]}
    if kind == "apply":
        nrhs = case["nrhs"]
        if case["op"] == "form_q":
            return {"bytes": 16.0 * m * n, "flops": _qr_flops(m, n)}
        return {"bytes": 8.0 * m * n + 16.0 * m * nrhs, "flops": q1 * nrhs}
    if kind == "ls":
        return {"bytes": 8.0 * (m * n + m + n), "flops": _qr_flops(m, n) + q1 + float(n) * n}
    shapes = _shapes(case)
    if kind == "batched":
        e = 4 if case["dtype"] == "f32" else 8
        return {"bytes": e * sum(2.0 * m * n + 16 * n for m, n in shapes), "flops": sum(_qr_flops(m, n) for m, n in shapes)}
    return {"bytes": 8.0 * sum(m * n + m + n for m, n in shapes),
            "flops": sum(_qr_flops(m, n) + 4.0 * m * n for m, n in shapes)}


# ------------------------------------------------ the same in 64 bits, plainly

def _plain_qr(a):
    """LAPACK-style V\\R and tau in the library's sign convention: an empty
    last subcolumn is reflected too (tau = 2, R negated)."""
    vr, tau = torch.geqrf(a.double().contiguous())
    m, n = a.shape
    if m == n:
        vr[-1, -1] = -vr[-1, -1]
        tau = tau.clone()
        tau[-1] = 2.0
    return vr, tau


def _plain_t(vr, nb):
    """Panel kernels (nb x n): T^-1 = striu(V^T V) + diag(V^T V) / 2."""
    m, n = vr.shape
    t = torch.zeros((nb, n), dtype=torch.float64, device=vr.device)
    for j in range(0, n, nb):
        w = min(nb, n - j)
        v = torch.tril(vr[j:, j:j + w], -1)
        v[:w].diagonal().fill_(1.0)
        g = v.T @ v
        k = torch.triu(g, 1) + torch.diag(g.diagonal() / 2)
        t[:w, j:j + w] = torch.linalg.solve_triangular(k, torch.eye(w, dtype=torch.float64, device=vr.device), upper=True)
    return t


def _reflect(vr, t, b, trans):
    """Q^T b or Q b from the panel kernels."""
    n, nb = vr.shape[1], t.shape[0]
    b = b.clone()
    js = list(range(0, n, nb))
    for j in js if trans else js[::-1]:
        w = min(nb, n - j)
        v = torch.tril(vr[j:, j:j + w], -1)
        v[:w].diagonal().fill_(1.0)
        tk = t[:w, j:j + w]
        b[j:] -= v @ ((tk.T if trans else tk) @ (v.T @ b[j:]))
    return b


def exact(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "factor":
        dt = torch.float32 if case["dtype"] == "f32" else torch.float64
        m, n = case["m"], case["n"]
        a = _matrix(m, n, case["decades"], g, case["pad"], dt)
        b = _matrix(m, case["rhs"], 0.0, g) if case["rhs"] else None
        vr, _ = _plain_qr(a)
        t = _plain_t(vr, n if case["layout"] == "full" else _nb(m, n))
        if b is None:
            return vr, t
        return vr, t, _reflect(vr, _plain_t(vr, _nb(m, n)), b, True)
    if kind == "apply":
        m, n = case["m"], case["n"]
        vr, _ = _plain_qr(_matrix(m, n, case["decades"], g))
        t = _plain_t(vr, _nb(m, n))
        if case["op"] == "form_q":
            return _reflect(vr, t, torch.eye(m, n, dtype=torch.float64, device=DEV), False)
        return _reflect(vr, t, _matrix(m, case["nrhs"], 0.0, g), case["op"] == "apply_qt")
    if kind == "ls":
        return _plain_ls(*_ls_problem(case["m"], case["n"], case["decades"], g))
    shapes = _shapes(case)
    if kind == "serve":
        return torch.cat([_plain_ls(*_ls_problem(m, n, _request_decades(case, k), g)) for k, (m, n) in enumerate(shapes)])
    if len(shapes) > 600:
        return None
    dt = torch.float32 if case["dtype"] == "f32" else torch.float64
    flat = torch.empty(sum(m * n for m, n in shapes), dtype=dt, device=DEV).normal_(generator=g)
    As, Ts, a = [], [], 0
    for m, n in shapes:
        nb = _nb(m, n)
        vr, _ = _plain_qr(flat[a:a + m * n].view(n, m).T)
        t = torch.zeros((nb, n), dtype=torch.float64, device=DEV)
        w = min(16, n)   # the batch's panel width
        t[:w] = _plain_t(vr, w)
        As.append(vr.T.reshape(-1))
        Ts.append(t.T.reshape(-1))
        a += m * n
    return torch.cat(As), torch.cat(Ts)


def _plain_ls(a, b):
    vr, _ = _plain_qr(a)
    n = a.shape[1]
    t = _plain_t(vr, min(128, n))
    r = torch.triu(vr[:n])

    def solve(v):
        return torch.linalg.solve_triangular(r, _reflect(vr, t, v[:, None], True)[:n], upper=True)[:, 0]

    x = solve(b)
    return x + solve(b - a @ x)
