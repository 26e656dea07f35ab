"""What a user of this library has it compute, as cases that can be timed and compared.

The cases stand for the calls that make up a PEPS program: the environments of a
whole lattice (plain calls and recorded plans, both truncation modes, FP64 and
the split tensor-core precisions), the norm sweep, the cluster environments of
every site, a Trotter step of the imaginary-time evolution with the full and
with the cluster update, and the closure network's inference and gradient.

Lattices come in two kinds.  "flat" has entries 0.5 + 0.1 N(0,1): a state close
to a product state, whose boundaries truncate with almost no loss.  "weighted"
has N(0,1) entries with the square root of a bond spectrum 1/(1+k)^2 on every
virtual leg, the form Gamma sqrt(lambda) in which a simple update hands its
tensors out: every bond is entangled and the fit has something to drop.  Every
site tensor has unit norm, and outward legs hold index 0 only.

A lattice in single precision stands for a program that works in single
precision: it keeps the observables that it reads in that type as well.
"""
import math

import numpy as np
import torch

from paper_1311_6696_gb300 import peps

WIDTH = peps.CLOSURE_WIDTH
SZ = np.array([[0.5, 0.0], [0.0, -0.5]])
SX = np.array([[0.0, 0.5], [0.5, 0.0]])
# S.S of a bond on (s1 s2), spin 1/2
SS = 0.25 * np.array([[1.0, 0, 0, 0], [0, -1.0, 2.0, 0], [0, 2.0, -1.0, 0], [0, 0, 0, 1.0]])
TAU = 0.01


# ---------------------------------------------------------------- the cases
def _full(name, Ly, Lx, D, chi, mode, precision, state, f32=False, plan=False):
    return dict(name=name, kind="full", Ly=Ly, Lx=Lx, D=D, chi=chi, mode=mode, precision=precision, state=state,
                f32=f32, plan=plan)


def _norm(name, Ly, Lx, D, chi, precision, state, f32=False):
    return dict(name=name, kind="norm", Ly=Ly, Lx=Lx, D=D, chi=chi, mode="var", precision=precision, state=state,
                f32=f32)


def _cluster(name, Ly, Lx, D, n, chi, precision, state, f32=False, plan=False):
    return dict(name=name, kind="cluster", Ly=Ly, Lx=Lx, D=D, n=n, chi=chi, mode="var", precision=precision,
                state=state, f32=f32, plan=plan)


def _evolve(name, Ly, Lx, D, chi, delta, precision, f32=False):
    return dict(name=name, kind="evolve", Ly=Ly, Lx=Lx, D=D, chi=chi, mode="var", delta=delta, precision=precision,
                state="weighted", f32=f32)


def listed():
    return [
        # The smallest lattice anybody contracts, in the default mode: a check, a unit test, the inner step of a
        # script over many small states.  Launches and latency are all of it.
        _full("full_4x4_D2_svd_fp64", 4, 4, 2, 16, "svd", "fp64", "flat"),
        # An odd lattice with odd bonds, truncated by SVD: nothing is a multiple of anything.
        _full("full_5x7_D3_svd_fp64", 5, 7, 3, 20, "svd", "fp64", "weighted"),
        # The ordinary calculation in FP64: every density matrix of a 10x10 lattice with variational boundaries.
        _full("full_10x10_D4_var_fp64", 10, 10, 4, 32, "var", "fp64", "flat"),
        # The same lattice in single precision at a larger bond, as a program that measures again and again keeps
        # it: one recorded plan, replayed after the tensors were overwritten.
        _full("plan_10x10_D4_var_tf32x3", 10, 10, 4, 64, "var", "tf32x3", "flat", f32=True, plan=True),
        # The norm in FP64 at the bonds where FP64 arithmetic dominates.
        _norm("norm_4x11_D6_fp64", 4, 11, 6, 64, "fp64", "weighted"),
        # The largest bonds in use, D = 8 and chi = 128 on the tensor cores: three absorbed rows of a 20-wide lattice.
        _norm("norm_4x20_D8_bf16x3", 4, 20, 8, 128, "bf16x3", "weighted", f32=True),
        # Cluster environments of every site: small windows, one plain call.
        _cluster("cluster_14x14_D6_n2_tf32x3", 14, 14, 6, 2, 36, "tf32x3", "flat", f32=True),
        # Cluster environments with windows that truncate, replayed as a recorded plan.
        _cluster("plan_cluster_16x16_D4_n4_tf32x3", 16, 16, 4, 4, 32, "tf32x3", "flat", f32=True, plan=True),
        # One Trotter step of the full update: the imaginary-time evolution's inner call.
        _evolve("evolve_full_8x8_D4_fp64", 8, 8, 4, 16, -1, "fp64"),
        # One Trotter step of the cluster update on an odd lattice with the split tensor-core environments.
        _evolve("evolve_cluster_7x5_D3_tf32x3", 7, 5, 3, 12, 1, "tf32x3", f32=True),
        # The closure network's gradient on one large batch, and its inference on every rim of many lattices.
        dict(name="mlp_grad_D4_n4999", kind="grad", D=4, n=4999),
        dict(name="mlp_predict_D4_n50000", kind="predict", D=4, n=50000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["svd", "full", "full", "norm", "norm", "cluster", "evolve", "evolve", "grad", "predict"])
    if kind == "svd":
        D = rng.choice([2, 2, 3])
        side = (3, 9) if D == 2 else (3, 5)
        return _strip(_full("", rng.randint(*side), rng.randint(*side), D, rng.randint(8, 20), "svd", "fp64",
                            rng.choice(["flat", "weighted"])))
    if kind == "full":
        D, fast = rng.choice([2, 3, 4, 5]), rng.random() < 0.6
        prec = rng.choice(["tf32x3", "bf16x3"]) if fast else "fp64"
        chi = _log(rng, 12, 64 if fast else 32) if D < 5 else _log(rng, 12, 32 if fast else 20)
        return _strip(_full("", rng.randint(4, 10), rng.randint(4, 10), D, chi, "var", prec,
                            rng.choice(["flat", "weighted"]), f32=fast and rng.random() < 0.8,
                            plan=rng.random() < 0.4))
    if kind == "norm":
        D, fast = rng.randint(3, 8), rng.random() < 0.5
        prec = rng.choice(["tf32x3", "bf16x3"]) if fast else "fp64"
        chi = _log(rng, 16, 128 if fast else (96 if D < 6 else 48))
        return _strip(_norm("", rng.randint(3, 4), rng.randint(5, 20 if fast else 10), D, chi, prec,
                            rng.choice(["flat", "weighted"]), f32=fast))
    if kind == "cluster":
        n = rng.choice([1, 2, 2, 3, 4])
        D = rng.randint(2, 6) if n < 4 else rng.randint(2, 4)
        fast = n > 2 or rng.random() < 0.7
        return _strip(_cluster("", rng.randint(5, 16), rng.randint(5, 16), D, n, rng.choice([16, 25, 32, 36]),
                               "tf32x3" if fast else "fp64", "flat", f32=fast, plan=rng.random() < 0.4))
    if kind == "evolve":
        D, fast = rng.choice([2, 3, 4]), rng.random() < 0.5
        return _strip(_evolve("", rng.randint(3, 8), rng.randint(3, 8), D, _log(rng, 6, 24), rng.choice([-1, 0, 1]),
                              "tf32x3" if fast else "fp64", f32=fast))
    D = rng.choice([2, 3, 4, 4])
    return dict(kind=kind, D=D, n=_log(rng, 100, 20000 if kind == "grad" else 100000))


def _strip(c):
    return {k: v for k, v in c.items() if k != "name"}


# ---------------------------------------------------------------- inputs
def _lattice(case, seed):
    """Dense FP64 lattice on the GPU, (Ly, Lx, d, D, D, D, D)."""
    Ly, Lx, D, d = case["Ly"], case["Lx"], case["D"], 2
    g = torch.Generator(device="cuda").manual_seed(1 + seed)
    A = torch.randn(Ly, Lx, d, D, D, D, D, generator=g, device="cuda", dtype=torch.float64)
    if case["state"] == "flat":
        A = 0.5 + 0.1 * A
    else:
        w = 1.0 / (1.0 + torch.arange(D, device="cuda", dtype=torch.float64))
        for leg in range(4):
            A = A * w.reshape([-1 if k == 3 + leg else 1 for k in range(7)])
    A[0, :, :, 1:] = 0.0
    A[:, 0, :, :, 1:] = 0.0
    A[-1, :, :, :, :, 1:] = 0.0
    A[:, -1, :, :, :, :, 1:] = 0.0
    A = A / A.square().sum(dim=(2, 3, 4, 5, 6), keepdim=True).sqrt()
    return (A.float() if case["f32"] else A).contiguous()


def _features(D):
    return 2 * D ** 4 + 2 * D * D


def _mlp(case, seed):
    """Weights and a training set as the closure has them: unit-norm site tensors, a positive CU_0 matrix and its
    Cholesky factor as features, positive matrices close to the CU_0 ones as labels."""
    D, n = case["D"], case["n"]
    g = torch.Generator(device="cuda").manual_seed(1 + seed)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)

    def unit(t):
        return t / t.square().sum(dim=tuple(range(1, t.dim())), keepdim=True).sqrt()

    site = unit(0.5 + 0.1 * normal(n, 2 * D ** 4))
    eye = torch.eye(D, device="cuda", dtype=torch.float64)
    low = torch.tril(0.3 * normal(n, D, D), -1) + eye * (1.0 + 0.3 * normal(n, D, 1).clamp(-2.0, 2.0))
    sig = low @ low.mT
    size = sig.square().sum(dim=(1, 2), keepdim=True).sqrt()
    sig, low = sig / size, low / size.sqrt()
    X = torch.cat([site, sig.reshape(n, -1), low.reshape(n, -1)], dim=1).float().contiguous()
    near = low + 0.05 * normal(n, D, D)
    Y = unit(near @ near.mT).reshape(n, -1).float().contiguous()
    w = peps.mlp_init(2, D, seed=seed)
    # a network that has been trained for a while: the output layer is no longer zero
    F = _features(D)
    k = WIDTH * F + WIDTH + WIDTH * WIDTH + WIDTH
    w[k:k + D * D * WIDTH] = (0.01 * normal(D * D * WIDTH)).float()
    return w, X, Y


def _gate():
    w, v = np.linalg.eigh(SS)
    return (v * np.exp(-TAU * w)) @ v.T


def prepare(case, seed):
    if case["kind"] in ("grad", "predict"):
        w, X, Y = _mlp(case, seed)
        return dict(case=case, w=w, X=X, Y=Y)
    s = dict(case=case, A=_lattice(case, seed), gate=_gate())
    if case.get("plan"):
        n = case["n"] if case["kind"] == "cluster" else None
        s["plan"] = peps.Plan(s["A"], case["chi"], mode=case["mode"], precision=case["precision"], cluster_n=n)
    return s


# ---------------------------------------------------------------- one pass
def _observables(env, case):
    """What a measurement of a spin-1/2 state reads: both spin components on every site, S.S on every bond."""
    out = {"sz": env.expect("site", SZ), "sx": env.expect("site", SX)}
    if case.get("n", 2) > 1:
        out["ss_h"], out["ss_v"] = env.expect("hbond", SS), env.expect("vbond", SS)
    if case["f32"]:
        return {k: v.astype(np.float32) for k, v in out.items()}
    out["rho_site"] = env.rho("site")
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "grad":
        loss, g = peps.mlp_loss_grad(state["w"], state["X"], state["Y"], 2, case["D"])
        return {"loss": loss, "grad": g}
    if kind == "predict":
        return {"sigma": peps.mlp_predict(state["w"], state["X"], 2, case["D"])}
    A = state["A"]
    opt = dict(mode=case["mode"], precision=case["precision"])
    if kind == "norm":
        ln, sign = peps.norm(A, case["chi"], **opt)
        return {"ln": ln, "sign": sign}
    if kind == "evolve":
        delta = case["delta"] if case["delta"] >= 0 else None
        return {"A": peps.evolve(A.clone(), state["gate"], 1, case["chi"], delta=delta, **opt)}
    if "plan" in state:
        env = state["plan"].run()
    elif kind == "cluster":
        env = peps.env_cluster(A, case["n"], case["chi"], **opt)
    else:
        env = peps.env_full(A, case["chi"], **opt)
    out = _observables(env, case)
    if kind == "full":
        out["ln"], out["sign"] = env.ln_norm()
    return out


# ---------------------------------------------------------------- what a pass cannot do without
def _dim(case, y, x):
    D, Ly, Lx = case["D"], case["Ly"], case["Lx"]
    return (1 if y == 0 else D, 1 if x == 0 else D, 1 if y == Ly - 1 else D, 1 if x == Lx - 1 else D)


def _sweep(rows, chi, d, mode):
    """Flops of the boundary sweep over rows of (u, l, n, r) dimensions, and the bond dimensions it leaves."""
    fl, bonds = 0.0, [1] * (len(rows[0]) - 1)
    out = [list(bonds)]
    for row in rows:
        L = len(row)
        prod = [bonds[k] * row[k][3] ** 2 for k in range(L - 1)]
        caps = []
        for k in range(L - 1):
            left = math.prod(min(s[2] ** 2, 1 << 20) for s in row[:k + 1])
            right = math.prod(min(s[2] ** 2, 1 << 20) for s in row[k + 1:])
            caps.append(min(chi, left, right, prod[k]))
        full = [1] + prod + [1]
        new = [1] + caps + [1]
        old = [1] + bonds + [1]
        fit = mode == "var" and any(p > c for p, c in zip(prod, caps))
        for x, (u, l, n, r) in enumerate(row):
            if not fit:
                a, b = old[x], old[x + 1]
                fl += 2.0 * a * b * d * u * u * l * n * r + 2.0 * a * b * d * u * l * l * n * n * r * r
                m, k = new[x] * n * n, full[x + 1]
                fl += 2.0 * m * k * min(m, k) if x + 1 < L else 0.0
            else:   # three absorb chains: right environments, then two half-sweeps, each with a QR
                c, a, b, e = new[x], old[x], old[x + 1], new[x + 1]
                chain = 2.0 * c * l * l * a * u * u * b + 2.0 * c * b * l * l * u * u * d * n * r \
                    + 2.0 * c * b * l * u * d * n * n * r * r
                close = 2.0 * c * n * n * r * r * b * e
                fl += 3 * chain + 5 * close + 2 * 4.0 * c * n * n * e * min(c, e)
        bonds = caps
        out.append(list(bonds))
    return fl, out


def _rows(case, transpose=False, h0=0, h1=None, flip=False):
    Ly, Lx = case["Ly"], case["Lx"]
    if transpose:
        rows = [[(t[1], t[0], t[3], t[2]) for t in (_dim(case, y, x) for y in range(Ly))] for x in range(Lx)]
    else:
        rows = [[_dim(case, y, x) for x in range(Lx)] for y in range(Ly)]
    rows = rows[h0:h1]
    return [[(t[2], t[1], t[0], t[3]) for t in r] for r in rows[::-1]] if flip else rows


def _row_pass(row, top, bot, d, opened):
    """Environments of one row from both sides, and the open-site chains of `opened` columns."""
    fl = 0.0
    T, B = [1] + top + [1], [1] + bot + [1]
    for x, (u, l, n, r) in enumerate(row):
        a, b, c, e = T[x], T[x + 1], B[x], B[x + 1]
        one = 2.0 * c * l * l * a * u * u * b
        two = 2.0 * c * b * l * l * u * u * d * n * r
        three = 2.0 * c * b * l * u * d * n * n * r * r
        fl += 2 * (one + two + three + 2.0 * c * n * n * r * r * b * e)
        fl += opened * (one + two + three * d + 2.0 * c * n * n * r * r * b * e * d * d)
    return fl


def work(case):
    d = 2
    if case["kind"] in ("grad", "predict"):
        n, o, F = case["n"], case["D"] ** 2, _features(case["D"])
        params = WIDTH * F + WIDTH + WIDTH * WIDTH + WIDTH + o * WIDTH + o
        mac = n * (F * WIDTH + WIDTH * WIDTH + WIDTH * o)
        if case["kind"] == "predict":
            return {"bytes": 4.0 * (n * F + params + n * o), "flops": 2.0 * mac}
        return {"bytes": 4.0 * (n * F + n * o + 2 * params), "flops": 2.0 * (3 * mac - n * F * WIDTH)}
    Ly, Lx, D, chi, mode = case["Ly"], case["Lx"], case["D"], case["chi"], case["mode"]
    size = (4.0 if case["f32"] else 8.0) * Ly * Lx * d * D ** 4
    found = 8.0 * (Ly * Lx * d * d + (2 * Ly * Lx - Ly - Lx) * d ** 4)
    if case["kind"] == "norm":
        fl, tops = _sweep(_rows(case)[:-1], chi, d, mode)
        return {"bytes": size + 16.0, "flops": fl + _row_pass(_rows(case)[-1], tops[-1], [1] * (Lx - 1), d, 0) / 2}
    if case["kind"] == "full" or (case["kind"] == "evolve" and case["delta"] < 0):
        fl = 0.0
        for t in (False, True):
            rows = _rows(case, t)
            f0, top = _sweep(rows[:-1], chi, d, mode)
            f1, bot = _sweep(_rows(case, t, flip=True)[:-1], chi, d, mode)
            fl += f0 + f1
            bot = bot[::-1]
            fl += sum(_row_pass(r, top[i], bot[i], d, 1 if t else 2) for i, r in enumerate(rows))
        return {"bytes": size + found, "flops": fl} if case["kind"] == "full" else {"bytes": 8 * size, "flops": 2 * fl}
    if case["kind"] == "evolve":   # four bond sets, each with its strips of 2 delta + 1 rows
        fl = 0.0
        for t in (False, True):
            rows = _rows(case, t)
            for i, r in enumerate(rows):
                lo, hi = max(0, i - case["delta"]), min(len(rows), i + case["delta"] + 1)
                f0, top = _sweep(rows[lo:i] or [r], chi, d, mode)
                fl += (f0 if i > lo else 0.0) * (2 if hi > i + 1 else 1) + _row_pass(r, top[-1], top[-1], d, 2)
        return {"bytes": 8 * size, "flops": 2 * fl}
    fl = 0.0
    for y in range(Ly):
        for x in range(Lx):
            n = case["n"]
            y0, x0 = y - (n + 1) // 2 + 1, x - (n + 1) // 2 + 1
            y1, x1 = min(Ly - 1, y0 + n - 1), min(Lx - 1, x0 + n - 1)
            y0, x0 = max(0, y0), max(0, x0)
            rows = [[_dim(case, i, j) for j in range(x0, x1 + 1)] for i in range(y0, y1 + 1)]
            f0, top = _sweep(rows, chi, d, mode)
            fl += 2 * f0 + 2 * _row_pass(rows[y - y0], top[y - y0], top[min(len(rows) - 1, y1 - y)], d, 2)
    return {"bytes": size + found, "flops": fl}


# ---------------------------------------------------------------- the values in 64 bits
def _site(A, y, x):
    """Site tensor with its effective legs, FP64."""
    Ly, Lx = A.shape[:2]
    t = A[y, x].double()
    return t[:, :1 if y == 0 else None, :1 if x == 0 else None, :1 if y == Ly - 1 else None,
             :1 if x == Lx - 1 else None]


def _strip_value(A, opened=(), ends=None):
    """<psi|psi> of a lattice contracted exactly, column by column, with the physical pairs of the sites in `opened`
    left open (one or two sites), as (tensor, ln of the scale taken out).  ends: closure matrices (top, bottom, left,
    right) on the outward legs, else those legs have dimension 1."""
    Ly, Lx = A.shape[:2]
    ln = 0.0

    def close(side, i):
        return ends[side][i] if ends else torch.ones(1, 1, device=A.device, dtype=torch.float64)

    # state: [open..., (l, m) of row 0, ..., (l, m) of row Ly - 1]; the open pairs are one leading index
    v = torch.ones(1, device=A.device, dtype=torch.float64)
    for y in range(Ly):
        v = torch.outer(v, close(2, y).reshape(-1)).reshape(-1)
    v = v.reshape(1, -1)
    dims = [close(2, y).shape[0] for y in range(Ly)]
    for x in range(Lx):
        top = close(0, x)
        # [o, done, (u v), rest]
        v = torch.einsum("or,uv->ouvr", v, top)
        done = 1
        for y in range(Ly):
            t = _site(A, y, x) if ends is None else A[y, x].double()
            d, du, dl, dn, dr = t.shape
            rest = math.prod(k * k for k in dims[y + 1:])
            v = v.reshape(-1, done, du, du, dl, dl, rest)
            v = torch.einsum("opuvlmz,sulnr->opvmznrs", v, t)
            if (y, x) in opened:
                v = torch.einsum("opvmznrs,tvmjq->ostprqnjz", v, t)
                v = v.reshape(v.shape[0] * d * d, -1)
            else:
                v = torch.einsum("opvmznrs,svmjq->oprqnjz", v, t)
                v = v.reshape(v.shape[0], -1)
            done *= dr * dr
            dims[y] = dr
            top = (dn, dn)
        v = torch.einsum("opuvz,uv->opz", v.reshape(v.shape[0], done, dn, dn, 1), close(1, x)).reshape(v.shape[0], -1)
        s = v.norm()
        v, ln = v / s, ln + float(s.log())
    for y in range(Ly - 1, -1, -1):
        c = close(3, y).reshape(-1)
        v = (v.reshape(v.shape[0], -1, c.numel()) * c).sum(-1)
    return v.reshape(-1), ln


def _bond_rho(A, one, two, ends=None):
    d = A.shape[2]
    r, _ = _strip_value(A, (one, two), ends)
    first_left = one[1] == two[1] or one[1] < two[1]
    assert first_left
    # leading index order: the site met first by the column sweep first, each as (s, t)
    return r.reshape(d, d, d, d).permute(0, 2, 1, 3).reshape(d * d, d * d)


def _mean(rho, op):
    op = torch.as_tensor(op, device=rho.device)
    return float((rho * op.T).sum() / rho.diagonal().sum())


def _measured(case, site, hbond, vbond):
    """The outputs of _observables from functions that give one density matrix each."""
    Ly, Lx = case["Ly"], case["Lx"]
    rs = [site(y, x) for y in range(Ly) for x in range(Lx)]
    out = {"sz": np.array([_mean(r, SZ) for r in rs]), "sx": np.array([_mean(r, SX) for r in rs])}
    if case.get("n", 2) > 1:
        out["ss_h"] = np.array([_mean(hbond(y, x), SS) for y in range(Ly) for x in range(Lx - 1)])
        out["ss_v"] = np.array([_mean(vbond(y, x), SS) for y in range(Ly - 1) for x in range(Lx)])
    if not case["f32"]:
        out["rho_site"] = None   # its scale is the library's own
    return out


def _cu0(rows, d):
    """Separable boundary matrices of rows of site tensors from the top: out[r][x] on the up legs of row r.  Each is
    the local contraction itself at unit norm, swept until nothing moves."""
    one = torch.ones(1, 1, device=rows[0][0].device, dtype=torch.float64)

    def unit(t):
        return t / t.norm()

    W = len(rows[0])
    out = [[one] * W]
    for row in rows[:-1]:
        # double-layer site with the matrix above it absorbed: [(l m), (n o), (r q)]
        E = []
        for t, S in zip(row, out[-1]):
            _, _, dl, dn, dr = t.shape
            z = torch.einsum("uv,sulnr,svmoq->lmnorq", S, t, t)
            E.append(z.reshape(dl * dl, dn * dn, dr * dr))
        new = [unit(torch.eye(t.shape[3], device=t.device, dtype=torch.float64)).reshape(-1) for t in row]
        L, R = [None] * W, [None] * W
        L[0], R[W - 1] = one.reshape(-1), one.reshape(-1)
        for x in range(W - 1, 0, -1):
            R[x - 1] = unit(torch.einsum("lnr,n,r->l", E[x], new[x], R[x]))
        for h in range(400):
            moved = torch.zeros((), device=one.device, dtype=torch.float64)
            for x in range(W) if h % 2 == 0 else range(W - 1, -1, -1):
                b = unit(torch.einsum("l,lnr,r->n", L[x], E[x], R[x]))
                moved = torch.maximum(moved, (b - new[x]).norm())
                new[x] = b
                if h % 2 == 0 and x < W - 1:
                    L[x + 1] = unit(torch.einsum("l,lnr,n->r", L[x], E[x], b))
                if h % 2 == 1 and x > 0:
                    R[x - 1] = unit(torch.einsum("lnr,n,r->l", E[x], b, R[x]))
            if float(moved) < 1e-13:
                break
        out.append([v.reshape(t.shape[3], t.shape[3]) for v, t in zip(new, row)])
    return out


def _exact_cluster(case, A):
    """Windows of at most 2x2 sites: the four CU_0 boundaries, then each window contracted exactly."""
    Ly, Lx, n, d = case["Ly"], case["Lx"], case["n"], 2
    S = [[_site(A, y, x) for x in range(Lx)] for y in range(Ly)]
    perm = {"t": (0, 1, 2, 3, 4), "b": (0, 3, 2, 1, 4), "l": (0, 2, 1, 4, 3), "r": (0, 4, 1, 2, 3)}
    top = _cu0([[t.permute(perm["t"]) for t in r] for r in S], d)
    bot = _cu0([[t.permute(perm["b"]) for t in r] for r in S[::-1]], d)[::-1]
    left = _cu0([[S[y][x].permute(perm["l"]) for y in range(Ly)] for x in range(Lx)], d)
    right = _cu0([[S[y][x].permute(perm["r"]) for y in range(Ly)] for x in range(Lx - 1, -1, -1)], d)[::-1]

    def value(y, x, opened):
        y0, x0 = max(0, y - (n + 1) // 2 + 1), max(0, x - (n + 1) // 2 + 1)
        y1 = min(Ly - 1, y - (n + 1) // 2 + n)
        x1 = min(Lx - 1, x - (n + 1) // 2 + n)
        w = _Window([[S[i][j] for j in range(x0, x1 + 1)] for i in range(y0, y1 + 1)])
        ends = ([top[y0][j] for j in range(x0, x1 + 1)], [bot[y1][j] for j in range(x0, x1 + 1)],
                [left[x0][i] for i in range(y0, y1 + 1)], [right[x1][i] for i in range(y0, y1 + 1)])
        r, _ = _strip_value(w, [(i - y0, j - x0) for i, j in opened], ends)
        if len(opened) == 1:
            return r.reshape(d, d)
        return r.reshape(d, d, d, d).permute(0, 2, 1, 3).reshape(d * d, d * d)

    return _measured(case, lambda y, x: value(y, x, [(y, x)]), lambda y, x: value(y, x, [(y, x), (y, x + 1)]),
                     lambda y, x: value(y, x, [(y, x), (y + 1, x)]))


class _Window:
    """Site tensors of unequal legs behind the two things _strip_value asks of a lattice."""

    def __init__(self, sites):
        self.sites = sites
        self.shape = (len(sites), len(sites[0]))
        self.device = sites[0][0].device

    def __getitem__(self, yx):
        return self.sites[yx[0]][yx[1]]


def _exact_mlp(case, seed):
    w, X, Y = _mlp(case, seed)
    D, F = case["D"], _features(case["D"])
    o, w = D * D, w.double().requires_grad_(case["kind"] == "grad")
    cuts = [WIDTH * F, WIDTH, WIDTH * WIDTH, WIDTH, o * WIDTH, o]
    W1, b1, W2, b2, W3, b3 = torch.split(w, cuts)
    x = X.double()
    h = torch.relu(x @ W1.reshape(WIDTH, F).T + b1)
    h = torch.relu(h @ W2.reshape(WIDTH, WIDTH).T + b2)
    m = x[:, F - o:].reshape(-1, D, D) + (h @ W3.reshape(o, WIDTH).T + b3).reshape(-1, D, D)
    s = m @ m.mT
    s = s / s.square().sum(dim=(1, 2), keepdim=True).sqrt()
    if case["kind"] == "predict":
        return {"sigma": s.reshape(-1, o)}
    loss = (s.reshape(-1, o) - Y.double()).square().sum() / case["n"]
    return {"loss": float(loss), "grad": torch.autograd.grad(loss, w)[0]}


def exact(case, seed):
    if case["kind"] in ("grad", "predict"):
        return _exact_mlp(case, seed)
    if case["kind"] == "evolve" or (case["kind"] == "cluster" and case["n"] > 2):
        return None
    if case["kind"] == "cluster":
        # the window's two-row boundaries keep all of D^2
        return _exact_cluster(case, _lattice(case, seed)) if case["chi"] >= case["D"] ** 2 else None
    A = _lattice(case, seed)
    h = min(case["Ly"], case["Lx"])
    if case["kind"] == "norm" and case["D"] ** (2 * case["Ly"]) <= 1 << 22:
        # the truncation of the boundaries is part of what run() returns: it is small for these states
        v, ln = _strip_value(A)
        return {"ln": ln + float(v.abs().log()), "sign": int(v.sign())}
    if case["kind"] == "full" and case["D"] ** (2 * h) <= 1 << 10 and case["Ly"] <= case["Lx"] \
            and case["chi"] >= case["D"] ** (2 * (h // 2)):
        out = _measured(case, lambda y, x: _strip_value(A, [(y, x)])[0].reshape(2, 2),
                        lambda y, x: _bond_rho(A, (y, x), (y, x + 1)), lambda y, x: _bond_rho(A, (y, x), (y + 1, x)))
        v, ln = _strip_value(A)
        return {**out, "ln": ln + float(v.abs().log()), "sign": int(v.sign())}
    return None
