"""The work that a user of this package has it do, as cases that can be timed: single
least-squares solves and QR decompositions in complex double, double-double and quad-double
(one Newton correction of a tracked path), ragged batches (many paths at once), the
differentiated solve, and a run of gated Newton steps.

Values: leading limbs uniform in [-1, 1), each lower limb uniform within half an ulp of the
limb above (normalised expansions); the "extreme" cases scale row i by 10^e_i and column j by
10^f_j, e_i in -12..12, f_j in -4..4, as Jacobians of badly scaled systems come.  Right-hand
sides are generic (a Newton residual is not in the range of the Jacobian).
"""

import math

import numpy as np
import torch

import paper_1210_0800_gb300 as mg

#: unit roundoff exponents are 53 bits per limb
NAMES = {1: "d", 2: "dd", 4: "qd"}


def listed():
    return [
        # the smallest calls: one correction of a small system, latency decides
        {"name": "dd solve 32x32", "op": "solve", "limbs": 2, "m": 32, "n": 32, "extreme": False},
        {"name": "qd solve 65x64", "op": "solve", "limbs": 4, "m": 65, "n": 64, "extreme": False},
        # plain complex double, the precision a tracker starts with
        {"name": "d solve 128x128", "op": "solve", "limbs": 1, "m": 128, "n": 128, "extreme": False},
        # a decomposition without a right-hand side, odd sizes
        {"name": "dd qr 131x97", "op": "qr", "limbs": 2, "m": 131, "n": 97, "extreme": False},
        # an ordinary corrector solve on a badly scaled Jacobian
        {"name": "dd solve 256x256 extreme", "op": "solve", "limbs": 2, "m": 256, "n": 256, "extreme": True},
        # the overdetermined quad-double system of the benchmark
        {"name": "qd solve 320x256", "op": "solve", "limbs": 4, "m": 320, "n": 256, "extreme": False},
        # the largest single systems of the size sweep
        {"name": "dd solve 512x512", "op": "solve", "limbs": 2, "m": 512, "n": 512, "extreme": False},
        {"name": "qd solve 512x512", "op": "solve", "limbs": 4, "m": 512, "n": 512, "extreme": False},
        # many paths at once: ragged batches in one launch
        {"name": "dd batch of 512", "op": "batch", "limbs": 2, "count": 512, "n_lo": 16, "n_hi": 192, "extra": 16},
        {"name": "qd batch of 64", "op": "batch", "limbs": 4, "count": 64, "n_lo": 16, "n_hi": 80, "extra": 8},
        # the differentiated solve: forward and backward of a uniform batch
        {"name": "dd lstsq 64 x 160x128", "op": "lstsq", "limbs": 2, "count": 64, "m": 160, "n": 128},
        # a corrector run: four gated Newton steps
        {"name": "qd newton 4 x 40x32", "op": "newton", "limbs": 4, "m": 40, "n": 32, "steps": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["solve", "solve", "solve", "qr", "batch", "batch", "lstsq", "newton"])
    limbs = rng.choice([2, 2, 4] if op in ("batch", "lstsq", "newton") else [1, 2, 2, 4, 4])
    if op in ("solve", "qr"):
        extreme = op == "solve" and limbs == 2 and rng.random() < 0.25
        n = _log_int(rng, 8, 256 if extreme else 448)
        return {"op": op, "limbs": limbs, "m": n + rng.randint(0, max(1, n // 8)), "n": n, "extreme": extreme}
    if op == "batch":
        return {"op": op, "limbs": limbs, "count": _log_int(rng, 4, 448 if limbs == 2 else 64),
                "n_lo": rng.randint(4, 32), "n_hi": rng.randint(40, 176 if limbs == 2 else 80), "extra": rng.randint(0, 16)}
    if op == "lstsq":
        n = _log_int(rng, 8, 128 if limbs == 2 else 40)
        return {"op": op, "limbs": limbs, "count": _log_int(rng, 2, 64), "m": n + rng.randint(0, n // 4), "n": n}
    n = _log_int(rng, 8, 128 if limbs == 2 else 64)
    return {"op": op, "limbs": limbs, "m": n + rng.randint(0, n // 4), "n": n, "steps": rng.randint(2, 6)}


# ------------------------------------------------------------------------------- inputs


def _limbs(lead, L, rng):
    """`lead` as leading limbs, lower limbs uniform within half an ulp of the limb above."""
    out = np.empty(lead.shape + (L,))
    out[..., 0] = lead
    for k in range(1, L):
        out[..., k] = (rng.random(lead.shape) - 0.5) * np.spacing(np.abs(out[..., k - 1]))
    return out


def _uniform(shape, L, rng, scale=None):
    lead = rng.uniform(-1.0, 1.0, tuple(shape) + (2,))
    return _limbs(lead if scale is None else lead * scale[..., None], L, rng)


def _system(m, n, L, rng, extreme=False):
    """A (n, m, 2, L), column-major by element, and b (m, 2, L)."""
    if not extreme:
        return _uniform((n, m), L, rng), _uniform((m,), L, rng)
    rows = 10.0 ** rng.integers(-12, 13, m).astype(np.float64)
    cols = 10.0 ** rng.integers(-4, 5, n).astype(np.float64)
    return _uniform((n, m), L, rng, cols[:, None] * rows[None, :]), _uniform((m,), L, rng, rows)


def _host_inputs(case, seed):
    """The case's systems [(A, b)] (and x0 of a Newton run) from the seed alone."""
    rng = np.random.default_rng([seed, 20130113])
    L, op = case["limbs"], case["op"]
    if op in ("solve", "qr"):
        return [_system(case["m"], case["n"], L, rng, case["extreme"])]
    if op == "batch":
        sizes = np.random.default_rng([case["count"], case["n_lo"], case["n_hi"], case["extra"]])
        ns = sizes.integers(case["n_lo"], case["n_hi"] + 1, case["count"])
        ms = ns + sizes.integers(0, case["extra"] + 1, case["count"])
        return [_system(int(m), int(n), L, rng) for m, n in zip(ms, ns)]
    if op == "lstsq":
        return [_system(case["m"], case["n"], L, rng) for _ in range(case["count"])]
    return [_system(case["m"], case["n"], L, rng) for _ in range(case["steps"])] + [_uniform((case["n"],), L, rng)]


def _tall(systems):
    return any(s[0].shape[1] > s[0].shape[0] for s in systems if isinstance(s, tuple))


def prepare(case, seed):
    """Inputs on the GPU and the buffers that a tracker keeps from call to call."""
    dev = torch.device("cuda:0")
    L, op = case["limbs"], case["op"]
    systems = _host_inputs(case, seed)

    def new(*shape):
        return torch.zeros(shape, dtype=torch.float64, device=dev)

    def up(a):
        return torch.from_numpy(a).to(dev)

    st = {"op": op, "limbs": L, "tall": _tall(systems), "status": torch.zeros(1, dtype=torch.int32, device=dev)}
    if op in ("solve", "qr"):
        m, n = case["m"], case["n"]
        A, b = systems[0]
        st.update(A=up(A), b=up(b), Aw=new(n, m, 2, L), bw=new(m, 2, L), x=new(n, 2, L), R=new(n, n, 2, L), z=new(L),
                  ws=torch.empty(mg.mgs_workspace_bytes(L, m, n, op == "solve"), dtype=torch.uint8, device=dev))
    elif op == "batch":
        bt = mg.make_batch(systems, dev)
        st.update(bt=bt, A=bt.A_pool.clone(), b=bt.b_pool.clone())
    elif op == "lstsq":
        st.update(A=up(np.stack([A for A, _ in systems])).requires_grad_(True),
                  b=up(np.stack([b for _, b in systems])).requires_grad_(True))
    else:
        m, n = case["m"], case["n"]
        st.update(J=[up(A) for A, _ in systems[:-1]], F=[up(b) for _, b in systems[:-1]], x0=up(systems[-1]),
                  Jw=new(n, m, 2, L), Fw=new(m, 2, L), x=new(n, 2, L), state=mg.NewtonState(dev),
                  ws=torch.empty(mg.newton.workspace_bytes(L, m, n), dtype=torch.uint8, device=dev))
    return st


def _with_residual(st, out, **more):
    """The residual b - A x of a square system is zero but for rounding, so that no two
    implementations share a digit of it: it is an output where some system has m > n."""
    return {**out, **more} if st["tall"] else out


def run(st):
    """One pass: the evaluated Jacobian and residual are written into the working buffers
    (the solve overwrites them, so a tracker does this for every correction), then the call."""
    op, L = st["op"], st["limbs"]
    if op == "solve":
        st["Aw"].copy_(st["A"])
        st["bw"].copy_(st["b"])
        fn = {1: mg.ls_solve_d, 2: mg.ls_solve_dd, 4: mg.ls_solve_qd}[L]
        fn(st["Aw"], st["bw"], x=st["x"], R=st["R"], z=st["z"], workspace=st["ws"], status=st["status"])
        return _with_residual(st, {"x": st["x"], "Q": st["Aw"], "R": st["R"], "status": st["status"]}, residual=st["bw"], z=st["z"])
    if op == "qr":
        st["Aw"].copy_(st["A"])
        fn = {1: mg.mgs_qr_d, 2: mg.mgs_qr_dd, 4: mg.mgs_qr_qd}[L]
        fn(st["Aw"], R=st["R"], workspace=st["ws"], status=st["status"])
        return {"Q": st["Aw"], "R": st["R"], "status": st["status"]}
    if op == "batch":
        bt = st["bt"]
        bt.A_pool.copy_(st["A"])
        bt.b_pool.copy_(st["b"])
        status = mg.ls_solve_batched(bt)
        return _with_residual(st, {"x": bt.x_pool, "Q": bt.A_pool, "status": status}, residual=bt.b_pool)
    if op == "lstsq":
        st["A"].grad = st["b"].grad = None
        x = mg.lstsq(st["A"], st["b"])
        x.backward(gradient=2.0 * x.detach())  # the loss sum |x|^2
        return {"x": x.detach(), "grad_A": st["A"].grad, "grad_b": st["b"].grad}
    st["x"].copy_(st["x0"])
    st["state"].reset()
    for J, F in zip(st["J"], st["F"]):
        st["Jw"].copy_(J)
        st["Fw"].copy_(F)
        mg.newton_step(st["Jw"], st["Fw"], st["x"], 0.0, st["state"], workspace=st["ws"], status=st["status"])
    return _with_residual(st, {"x": st["x"], "Q": st["Jw"], "status": st["status"]}, residual=st["Fw"])


# ------------------------------------------------------------------------- work and bounds


def _shapes(case):
    op = case["op"]
    if op == "batch":  # the mean shape, `count` times
        n = 0.5 * (case["n_lo"] + case["n_hi"])
        n3 = (case["n_hi"] ** 4 - case["n_lo"] ** 4) / (4.0 * max(1, case["n_hi"] - case["n_lo"]))
        return case["count"], n + 0.5 * case["extra"], n, n3 * (1.0 + 0.5 * case["extra"] / n)
    m, n = case["m"], case["n"]
    return case.get("count", case.get("steps", 1)), m, n, float(m) * n * (n + 1)


def work(case):
    """Bytes: each input read once and each output written once.  Flops: multiplications and
    additions on numbers of the working precision (8 per complex multiply-add, one for the
    projection and one for the update of every element of every trailing column), not the
    instructions that a multi-limb operation takes."""
    count, m, n, mnn = _shapes(case)
    e = 16.0 * case["limbs"]
    one = {"solve": 2 * m * (n + 1) + n + n * (n + 1) / 2, "qr": 2 * m * n + n * (n + 1) / 2,
           "batch": 2 * m * (n + 1) + n, "lstsq": 2 * m * (n + 1) + n, "newton": 2 * m * (n + 1) + 2 * n}[case["op"]]
    extra = 8.0 * (2 * m * n + m * n + n * n) if case["op"] == "lstsq" else 0.0
    return {"bytes": count * e * one, "flops": count * (8.0 * mnn + extra)}


def tolerance(case):
    """Relative errors in the 2-norm over each output, all limbs.  Well-conditioned inputs:
    1e-14, 1e-30 and 1e-62 are seen on single systems; the condition of random square systems
    varies by a factor of some hundred (the worst of a batch sets its error).  Extreme
    scaling: x agrees to about 1e-14 and R to 1e-32, but Q has lost orthogonality to the
    conditioning (1e-8 between double-double and quad-double sums of the same system)."""
    if case.get("extreme"):
        return {"rel": 2e-7, "max": 2e-5}
    rel = {1: 1e-11, 2: 1e-27, 4: 1e-59}[case["limbs"]]
    return {"rel": rel, "max": 100 * rel}


# --------------------------------------------------------------------------------- exact


class _Fixed:
    """Complex arrays of fixed-point integers (Python integers scaled by 2^bits)."""

    def __init__(self, bits):
        self.bits = bits

    def of(self, limbs):
        """(re, im) object arrays of limbs (..., 2, L), exactly (bits below 2^-bits rounded off)."""
        mant, ex = np.frexp(limbs)
        mant = (mant * 2.0 ** 53).astype(np.int64).astype(object)
        sh = ex.astype(np.int64) - 53 + self.bits
        up, down = np.maximum(sh, 0).astype(object), np.maximum(-sh, 0).astype(object)
        v = ((mant << up) >> down).sum(axis=-1)
        return v[..., 0], v[..., 1]

    def limbs(self, z, L):
        """The nearest doubles, one after another, of (re, im) object arrays."""
        out = np.empty(z[0].shape + (2, L))
        one = 1 << self.bits
        for p in range(2):
            rest = z[p]
            for k in range(L):
                d = np.array([r / one for r in rest.ravel()], dtype=np.float64).reshape(rest.shape)
                out[..., p, k] = d
                back = np.zeros(d.shape + (2, 1))
                back[..., 0, 0] = d
                rest = rest - self.of(back)[0]
        return out

    def lead(self, z):
        """The leading doubles as a complex array."""
        out = self.limbs(z, 1)[..., 0]
        return out[..., 0] + 1j * out[..., 1]

    def of_complex(self, c):
        return self.of(np.stack([c.real, c.imag], -1)[..., None])


def _matvec(F, A, v):
    """A v for A (n, m), column j at A[j]."""
    re, im = (A[0].T.dot(v[0]) - A[1].T.dot(v[1])), (A[0].T.dot(v[1]) + A[1].T.dot(v[0]))
    return re >> F.bits, im >> F.bits


def _matvec_h(F, A, v):
    """A^H v."""
    re, im = (A[0].dot(v[0]) + A[1].dot(v[1])), (A[0].dot(v[1]) - A[1].dot(v[0]))
    return re >> F.bits, im >> F.bits


def _exact_mgs(F, A, b):
    """Modified Gram-Schmidt of [A b] in fixed point: Q, R (upper, [column, row]), x, residual, z."""
    n = A[0].shape[0]
    re = np.concatenate([A[0], b[0][None]]) if b is not None else A[0].copy()
    im = np.concatenate([A[1], b[1][None]]) if b is not None else A[1].copy()
    nc, P = re.shape[0], F.bits
    Rre, Rim = np.zeros((nc, n), dtype=object), np.zeros((nc, n), dtype=object)
    for k in range(n):
        ar, ai = re[k], im[k]
        G = int(ar.dot(ar) + ai.dot(ai))  # scaled by 2^2P
        r = math.isqrt(G)
        re[k], im[k] = (ar << P) // r, (ai << P) // r
        Rre[k, k] = r
        if k + 1 < nc:
            qr, qi, tr, ti = re[k], im[k], re[k + 1:], im[k + 1:]
            cr, ci = (tr.dot(qr) + ti.dot(qi)) >> P, (ti.dot(qr) - tr.dot(qi)) >> P
            Rre[k + 1:, k], Rim[k + 1:, k] = cr, ci
            c, d = cr[:, None], ci[:, None]
            re[k + 1:] = tr - ((c * qr - d * qi) >> P)
            im[k + 1:] = ti - ((c * qi + d * qr) >> P)
    out = {"Q": (re[:n], im[:n]), "R": (Rre[:n], Rim[:n])}
    if b is not None:
        xr, xi = Rre[n].copy(), Rim[n].copy()
        for k in range(n - 1, -1, -1):
            xr[k], xi[k] = (int(xr[k]) << P) // int(Rre[k, k]), (int(xi[k]) << P) // int(Rre[k, k])
            xr[:k] -= (Rre[k, :k] * xr[k] - Rim[k, :k] * xi[k]) >> P
            xi[:k] -= (Rre[k, :k] * xi[k] + Rim[k, :k] * xr[k]) >> P
        z = math.isqrt(int(re[n].dot(re[n]) + im[n].dot(im[n])))
        out.update(x=(xr, xi), residual=(re[n], im[n]), z=z)
    return out


def _refine(F, A, b, G=None):
    """x = argmin |b - A x| (or (A^H A)^-1 G) of a well-conditioned system by refinement of a
    double-precision solve with fixed-point residuals; also b - A x."""
    Ac = F.lead(A).T
    R = np.linalg.qr(Ac, mode="r")
    n = Ac.shape[1]
    zero = np.array([0] * n, dtype=object)
    x, last = (zero, zero), None
    for _ in range(60):
        Ax = _matvec(F, A, x)
        if G is None:
            r = (b[0] - Ax[0], b[1] - Ax[1])
            g = _matvec_h(F, A, r)
        else:
            r, h = Ax, _matvec_h(F, A, Ax)
            g = (G[0] - h[0], G[1] - h[1])
        top = max(max(abs(int(v)) for v in g[0]), max(abs(int(v)) for v in g[1]))
        if last is not None and (top >= last or top < 1 << 24):
            break
        last = top
        sh = max(0, top.bit_length() - 900)  # keep the doubles in range
        up = max(0, F.bits - top.bit_length())
        gc = F.lead(((g[0] >> sh) << up, (g[1] >> sh) << up))
        d = F.of_complex(np.linalg.solve(R, np.linalg.solve(R.conj().T, gc)))
        x = (x[0] + ((d[0] << sh) >> up), x[1] + ((d[1] << sh) >> up))
    return x, r


def _z_limbs(F, r, L):
    z = math.isqrt(int(r[0].dot(r[0]) + r[1].dot(r[1])))
    return F.limbs((np.array([z], dtype=object), np.array([0], dtype=object)), L)[0, 0]


def exact(case, seed):
    """The outputs of run() from fixed-point integers of several hundred bits: modified
    Gram-Schmidt where its m n^2 steps take seconds, else x and the residual by refinement
    (Q and R are then left out); None where that takes too long as well."""
    L, op = case["limbs"], case["op"]
    systems = _host_inputs(case, seed)
    F = _Fixed(53 * L + (320 if case.get("extreme") else 128))
    if op in ("solve", "qr", "batch"):
        sizes = [A.shape[0] ** 2 * A.shape[1] for A, _ in systems]
        full = sum(sizes) <= 6e6
        if not full and (op == "qr" or case.get("extreme") or sum(A.shape[0] * A.shape[1] for A, _ in systems) > 300000):
            return None
        parts = []
        for A, b in systems:
            Af, bf = F.of(A), F.of(b)
            if full:
                parts.append(_exact_mgs(F, Af, bf if op != "qr" else None))
            else:
                x, r = _refine(F, Af, bf)
                parts.append({"x": x, "residual": r})
        if op == "batch":
            def pool(k):
                return np.concatenate([F.limbs(p[k], L).reshape(-1, 2, L) for p in parts]) if full or k != "Q" else None

            return {"x": pool("x"), "Q": pool("Q"), "residual": pool("residual") if _tall(systems) else None, "status": None}
        p = parts[0]
        out = {"Q": F.limbs(p["Q"], L) if full else None, "R": F.limbs(p["R"], L) if full else None, "status": None}
        if op == "solve":
            out.update(x=F.limbs(p["x"], L))
            if _tall(systems):
                out.update(residual=F.limbs(p["residual"], L), z=_z_limbs(F, p["residual"], L))
        return out
    if op == "lstsq":
        if case["count"] * case["m"] * case["n"] > 200000:
            return None
        xs, gA, gb = [], [], []
        for A, b in systems:
            Af, bf = F.of(A), F.of(b)
            x, r = _refine(F, Af, bf)
            w, g = _refine(F, Af, bf, G=(2 * x[0], 2 * x[1]))  # g = A w = grad_b
            wr, wi, xr, xi = (v[:, None] for v in (w[0], w[1], x[0], x[1]))
            re = (r[0] * wr + r[1] * wi - g[0] * xr - g[1] * xi) >> F.bits
            im = (r[1] * wr - r[0] * wi - g[1] * xr + g[0] * xi) >> F.bits
            xs.append(F.limbs(x, L))
            gb.append(F.limbs(g, L))
            gA.append(F.limbs((re, im), L))
        return {"x": np.stack(xs), "grad_A": np.stack(gA), "grad_b": np.stack(gb)}
    x0 = F.of(systems[-1])
    re, im = x0
    for A, b in systems[:-1]:
        s, r = _refine(F, F.of(A), F.of(b))
        re, im = re - s[0], im - s[1]
    return {"x": F.limbs((re, im), L), "Q": None, "residual": F.limbs(r, L) if _tall(systems) else None, "status": None}
