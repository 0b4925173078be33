"""What this framework is used for, as measurable cases: solves of IgA stiffness
systems with the matching-AMG preconditioner (setup and solve together, and
solves on a kept hierarchy), the V-cycle as a preconditioner of a caller's own
Krylov method, several right-hand sides, batches, the paper's configuration,
the learned damping (inference and training) and the assembly.

Every case goes through the public entry points of
``paper_2511_21268_gb300.amg``.  Right-hand sides are F = K u for a smooth u
drawn from the seed (a load that a discretised PDE has), so the solution is
known; solves run to a relative residual of 1e-10, well below the
discretisation error, so that u is determined far more closely than one CG
iteration moves it.
"""
import math

import numpy as np
import torch

from paper_2511_21268_gb300 import amg as A
from paper_2511_21268_gb300 import inputs as I

RTOL = 1e-10
PRECISION = {"fp64": A.AMG_FP64, "fp32": A.AMG_FP32, "bf16": A.AMG_FP32_BF16FINE}
KAPPA = {"M": 256, "ell": 0.2, "sigma": 1.0}  # the coefficient field of the annulus workload


# ------------------------------------------------------------------ cases
def listed():
    return [
        # An implicit time step on a small 2-D patch, hierarchy kept: the
        # smallest solve, all launches and latency (N = 1,024).
        {"name": "solve_2d_small", "kind": "solve", "geom": "box", "d": 2, "p": 2, "n": 32, "precision": "fp64",
         "damping": 1.0},
        # One small 2-D system from scratch, setup and solve (a parameter
        # study, one patch of a nonlinear iteration); odd size.
        {"name": "tts_2d", "kind": "tts", "geom": "box", "d": 2, "p": 3, "n": 101, "precision": "fp64",
         "damping": 1.0},
        # The V-cycle as the preconditioner of a caller's own Krylov method.
        {"name": "vcycle_3d", "kind": "vcycle", "geom": "box", "d": 3, "p": 2, "n": 49, "precision": "fp64",
         "damping": 1.0},
        # The benchmark's workload, time to solution in FP64 (N = 274,625,
        # 86.9 M nonzeros): the largest solve.
        {"name": "tts_3d_fp64", "kind": "tts", "geom": "box", "d": 3, "p": 3, "n": 64, "precision": "fp64",
         "damping": 1.0},
        # The same system with its hierarchy kept (time stepping), mixed
        # precision with BF16 finest values.
        {"name": "solve_3d_mixed", "kind": "solve", "geom": "box", "d": 3, "p": 3, "n": 64, "precision": "bf16",
         "damping": 1.0},
        # A variable coefficient on the quarter annulus from scratch, mixed
        # precision with a constant damping; odd size.
        {"name": "tts_3d_mixed", "kind": "tts", "geom": "annulus", "d": 3, "p": 2, "n": 47, "precision": "fp32",
         "damping": 1.8},
        # The learned damping in earnest: setup given the network's weights,
        # then the solve, on the annulus workload at n = 40.
        {"name": "learned_3d", "kind": "learned", "geom": "annulus", "d": 3, "p": 3, "n": 40, "precision": "bf16",
         "damping": 1.0},
        # Two Adam steps of the network on three annulus hierarchies (the
        # backward direction).
        {"name": "train", "kind": "train", "geom": "annulus", "d": 3, "n": 16, "probes": 4, "steps": 2},
        # 16 load cases of one stiffness matrix.
        {"name": "multi_rhs", "kind": "multi", "geom": "box", "d": 3, "p": 3, "n": 32, "rhs": 16,
         "precision": "fp32", "damping": 1.0},
        # A mixed batch of 2-D patches, setup and solve as one hierarchy.
        {"name": "batch_2d", "kind": "batch", "d": 2, "count": 24, "n_lo": 32, "n_hi": 160, "shapes": 20251126,
         "precision": "fp32"},
        # The paper's own configuration (size-8 aggregates, smoothed
        # prolongators, Chebyshev, coarse CG, flexible CG) on its cube case.
        {"name": "paper_cube", "kind": "paper", "geom": "cube_mixed", "d": 3, "p": 3, "n": 32, "precision": "fp64"},
        # Assembly of the annulus workload at full size.
        {"name": "assemble_3d", "kind": "assemble", "geom": "annulus", "d": 3, "p": 3, "n": 64, "kappa": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# Largest n of a drawn 3-D case by degree: entries and CG iterations together
# stay below those of the listed cube.
_N3 = {2: 64, 3: 60, 4: 30}


def draw(rng):
    kind = rng.choice(["solve", "solve", "tts", "tts", "tts", "vcycle", "learned", "train", "multi", "batch", "paper",
                       "assemble"])
    if kind == "train":
        return {"kind": kind, "geom": "annulus", "d": 3, "n": rng.randint(8, 16), "probes": rng.randint(2, 4),
                "steps": rng.randint(1, 2)}
    if kind == "batch":
        lo = rng.randint(24, 64)
        return {"kind": kind, "d": 2, "count": rng.randint(4, 24), "n_lo": lo, "n_hi": lo + rng.randint(8, 96),
                "shapes": rng.randint(1, 1 << 30), "precision": rng.choice(["fp64", "fp32", "bf16"])}
    if kind == "paper":
        p = rng.choice([2, 3])
        return {"kind": kind, "geom": "cube_mixed", "d": 3, "p": p, "n": _log_int(rng, 10, 32),
                "precision": rng.choice(["fp64", "fp32"])}
    if kind == "assemble":
        p = rng.randint(2, 4)
        return {"kind": kind, "geom": rng.choice(["annulus", "box"]), "d": 3, "p": p,
                "n": _log_int(rng, 8, {2: 72, 3: 62, 4: 40}[p]), "kappa": rng.random() < 0.7}
    if kind == "multi":
        p = rng.choice([2, 3])
        return {"kind": kind, "geom": "box", "d": 3, "p": p, "n": _log_int(rng, 8, 30), "rhs": rng.randint(2, 16),
                "precision": rng.choice(["fp64", "fp32"]), "damping": 1.0}
    d = 3 if kind == "learned" else rng.choice([2, 3, 3])
    p = rng.choice([2, 3, 3, 4])
    if d == 2:
        return {"kind": kind, "geom": "box", "d": 2, "p": p, "n": _log_int(rng, 24, 220),
                "precision": "fp64" if kind == "vcycle" else rng.choice(["fp64", "fp64", "fp32"]),
                "damping": 1.0}
    hi = {2: 48, 3: 40, 4: 24}[p] if kind == "learned" else _N3[p]
    return {"kind": kind, "geom": "annulus" if kind == "learned" else rng.choice(["box", "annulus"]), "d": 3, "p": p,
            "n": _log_int(rng, 10, hi),
            "precision": "fp64" if kind == "vcycle" else
            rng.choice(["fp32", "bf16"] if kind == "learned" else ["fp64", "fp32", "bf16"]),
            "damping": 1.0 if kind in ("learned", "vcycle") else rng.choice([1.0, 1.8])}


# ----------------------------------------------------------------- inputs
def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _kappa(seed):
    g = _gen(seed)
    om = torch.randn(KAPPA["M"], 3, dtype=torch.float64, device="cuda", generator=g) / KAPPA["ell"]
    ph = torch.rand(KAPPA["M"], dtype=torch.float64, device="cuda", generator=g) * (2.0 * math.pi)
    return om, ph, KAPPA["sigma"]


def _system(geom, d, p, n, seed):
    """Device CSR of one system and its tensor shape (slowest direction first)."""
    if geom == "annulus":
        s = A.iga_assemble(n, p, geometry=A.AMG_GEOM_ANNULUS, kappa=_kappa(seed + 17), load=False)
        return (s["rowptr"], s["col"], s["val"]), (n + p - 2,) * 3
    if geom == "cube_mixed":
        nb = n + p
        rp, ci, va = I.assemble_kron_box(n, p, (1, 1, 0), (nb - 1, nb, nb))
        return (_dev(rp), _dev(ci), _dev(va)), (nb, nb - 1, nb - 2)
    rp, ci, va = I.assemble_kron(d, n, p)
    return (_dev(rp), _dev(ci), _dev(va)), (n + p - 2,) * d


def _smooth(shape, seed, count=1):
    """(count, prod(shape)) smooth fields: a few low sine modes each, with
    seeded frequencies, phases and amplitudes, zero at no particular place."""
    g = np.random.default_rng([int(seed), 11])
    out = torch.zeros(count, *shape, dtype=torch.float64, device="cuda")
    axes = [torch.linspace(0.0, 1.0, s, dtype=torch.float64, device="cuda") for s in shape]
    for k in range(count):
        for _ in range(5):
            term = torch.full((), float(g.normal()), dtype=torch.float64, device="cuda")
            for a, x in enumerate(axes):
                v = torch.sin(math.pi * float(g.uniform(0.5, 3.0)) * x + float(g.uniform(0.0, 2.0 * math.pi)))
                term = term[..., None] * v if a else term * v
            out[k] += term
    return out.reshape(count, -1)


def _apply(csr, u):
    """K u, each row's products summed by torch."""
    rp, ci, va = csr
    return torch.segment_reduce(va * u[ci.long()], "sum", lengths=rp[1:] - rp[:-1], unsafe=True)


def _opts(case):
    return {"precision": PRECISION[case["precision"]]}


def _batch_shapes(case):
    return I.batch_params(case["shapes"], case["count"], n_lo=case["n_lo"], n_hi=case["n_hi"])


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "case": case}
    if kind == "assemble":
        st["kappa"] = _kappa(seed + 17) if case["kappa"] else None
        st["geometry"] = A.AMG_GEOM_ANNULUS if case["geom"] == "annulus" else A.AMG_GEOM_CUBE
        # the load: f = 1 or the sine source
        st["source"] = seed % 2
        return st
    if kind == "train":
        st["H"] = []
        for k, p in enumerate((2, 3, 4)):
            csr, _ = _system("annulus", 3, p, case["n"], seed + 100 * k)
            st["H"].append(A.Hierarchy(*csr))
        st["w"] = _dev(I.mpnn_init_weights(seed + 1).astype(np.float32))
        st["seed"] = seed + 1000
        return st
    if kind == "batch":
        st["systems"], st["F"] = [], []
        for k, (p, n) in enumerate(_batch_shapes(case)):
            csr, shape = _system("box", 2, p, n, seed)
            st["systems"].append(csr)
            st["F"].append(_apply(csr, _smooth(shape, seed + k)[0]))
        st["opts"] = _opts(case)
        return st
    csr, shape = _system(case["geom"], case["d"], case["p"], case["n"], seed)
    if kind == "vcycle":
        # a residual, as the caller's Krylov method has it: rough
        st["r"] = torch.randn(len(csr[0]) - 1, dtype=torch.float64, device="cuda", generator=_gen(seed))
        st["H"] = A.Hierarchy(*csr, **_opts(case))
        return st
    U = _smooth(shape, seed, case["rhs"] if kind == "multi" else 1)
    F = torch.stack([_apply(csr, u) for u in U])
    st["F"] = F if kind == "multi" else F[0]
    st["opts"] = _opts(case)
    if kind in ("solve", "multi"):
        st["H"] = A.Hierarchy(*csr, **st["opts"])
        if case["damping"] != 1.0:
            st["H"].set_damping(case["damping"])
        return st
    st["csr"] = csr
    if kind == "learned":
        st["opts"]["mpnn_weights"] = _dev(I.mpnn_init_weights(seed + 1).astype(np.float32))
    if kind == "paper":
        st["opts"].update(match_passes=3, smooth_levels=-1, cheb_degree=8, coarse_solver=1, flexible=1)
    return st


# -------------------------------------------------------------------- run
def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "assemble":
        s = A.iga_assemble(case["n"], case["p"], geometry=st["geometry"], source=st["source"], kappa=st["kappa"])
        return {"rowptr": s["rowptr"], "col": s["col"], "val": s["val"], "F": s["F"]}
    if kind == "train":
        w = st["w"].clone()
        st["H"][0].mpnn_train(w, steps=case["steps"], nprobe=case["probes"], seed=st["seed"], lr=1e-2,
                              others=st["H"][1:])
        return {"w": w}
    if kind == "vcycle":
        return {"z": st["H"].vcycle(st["r"])}
    if kind == "solve":
        return {"u": st["H"].solve(st["F"], rtol=RTOL)["u"]}
    if kind == "multi":
        return {"u": st["H"].solve_multi(st["F"], rtol=RTOL)["u"]}
    if kind == "batch":
        with A.BatchHierarchy(st["systems"], **st["opts"]) as B:
            return {"u": B.solve_batch(st["F"], rtol=RTOL)["u"], "rows": _rows(B)}
    with A.Hierarchy(*st["csr"], **st["opts"]) as H:
        if case.get("damping", 1.0) != 1.0:
            H.set_damping(case["damping"])
        return {"u": H.solve(st["F"], rtol=RTOL)["u"], "rows": _rows(H)}


def _rows(H):
    """Rows of each level: the hierarchy the setup built."""
    return [H.level_n(l) for l in range(H.num_levels)]


# ------------------------------------------------------------------- work
def _size(geom, d, p, n):
    """(rows, stored entries) of one system."""
    def band(m):
        return m * (2 * p + 1) - p * (p + 1)

    ms = (n + p, n + p - 1, n + p - 2) if geom == "cube_mixed" else (n + p - 2,) * d
    return math.prod(ms), math.prod(band(m) for m in ms)


# CG iterations to 1e-10 of the plain method by degree, for a system past the
# smallest sizes (the method's own counts; the paper's configuration takes few).
_ITS = {(2, 2): 30, (2, 3): 50, (2, 4): 100, (3, 2): 60, (3, 3): 165, (3, 4): 450}


def work(case):
    """One pass's floor: the system read once and the solution written once,
    and the multiply-adds of the iterations' three finest-level matrix
    products (Chebyshev of degree 8: 17 of them) on a hierarchy of operator
    complexity 1.2."""
    kind = case["kind"]
    if kind == "assemble":
        N, Z = _size("box", 3, case["p"], case["n"])
        p, q = case["p"], case["p"] + 1
        Q, R = case["n"] * q, (2 * p + 1) * (case["n"] + p - 2)
        share = q * q / (2 * p + 1)  # mean Gauss points of a 1-D pair of the band
        flops = 2.0 * 4.0 * share * (R * Q * Q + R * R * Q + R * R * R)
        if case["kappa"]:
            flops += 2.0 * 2.0 * KAPPA["M"] * float(Q) ** 3
        return {"bytes": 12.0 * Z + 16.0 * N, "flops": flops}
    if kind == "train":
        flops = bytes_ = 0.0
        for p in (2, 3, 4):
            N, Z = _size("box", 3, p, case["n"])
            # network forward and backward (width 32, two layers) and four
            # V-cycle passes each way per probe
            flops += 2.0 * case["steps"] * (4.0 * 32 * Z + 12.0 * 1024 * N + 8.0 * case["probes"] * Z)
            bytes_ += 12.0 * Z
        return {"bytes": bytes_, "flops": flops}
    if kind == "batch":
        flops = bytes_ = 0.0
        for p, n in _batch_shapes(case):
            N, Z = _size("box", 2, p, n)
            flops += 2.0 * 3.6 * Z * _ITS[2, p]
            bytes_ += 12.0 * Z + 24.0 * N
        return {"bytes": bytes_, "flops": flops}
    N, Z = _size(case["geom"], case["d"], case["p"], case["n"])
    if kind == "vcycle":
        return {"bytes": 8.0 * Z + 16.0 * N, "flops": 2.0 * 2.4 * Z}
    if kind == "paper":
        return {"bytes": 12.0 * Z + 24.0 * N, "flops": 2.0 * 30 * 20.0 * Z}
    its = _ITS[case["d"], case["p"]]
    if kind == "multi":
        return {"bytes": 8.0 * Z + 16.0 * N * case["rhs"], "flops": 2.0 * 3.6 * Z * its * case["rhs"]}
    flops = 2.0 * 3.6 * Z * its
    if kind == "learned":
        flops += 4.0 * 32 * Z
    return {"bytes": 12.0 * Z + 24.0 * N, "flops": flops}


# ------------------------------------------------------------------ exact
def exact(case, seed):
    """Solves: the field u the right-hand side was made from.  Assembly: the
    same integrals by dense contractions in FP64.  The V-cycle (one step of
    the hierarchy's own making) and the training have no such value."""
    kind = case["kind"]
    if kind in ("vcycle", "train"):
        return None
    if kind == "assemble":
        return _exact_assembly(case, seed)
    if kind == "batch":
        return {"u": [_smooth((n + p - 2,) * 2, seed + k)[0] for k, (p, n) in enumerate(_batch_shapes(case))],
                "rows": None}
    p, n = case["p"], case["n"]
    shape = (n + p, n + p - 1, n + p - 2) if case["geom"] == "cube_mixed" else (n + p - 2,) * case["d"]
    if kind == "multi":
        return {"u": _smooth(shape, seed, case["rhs"])}
    u = _smooth(shape, seed)[0]
    return {"u": u} if kind == "solve" else {"u": u, "rows": None}


def _bsplines(n, p, x):
    """Values and derivatives at x of the n + p B-splines of degree p on the
    open uniform knot vector (Cox-de Boor recursion)."""
    t = np.concatenate([np.zeros(p), np.linspace(0.0, 1.0, n + 1), np.ones(p)])
    t = t.copy()
    e = np.minimum((x * n).astype(int), n - 1)
    B = np.zeros((len(x), n + 2 * p))
    B[np.arange(len(x)), e + p] = 1.0
    dB = np.zeros((len(x), n + p))
    for k in range(1, p + 1):
        cnt = n + 2 * p - k
        nB = np.zeros((len(x), cnt))
        dB = np.zeros((len(x), cnt))
        for i in range(cnt):
            a, b = t[i + k] - t[i], t[i + k + 1] - t[i + 1]
            if a > 0:
                nB[:, i] += (x - t[i]) / a * B[:, i]
                dB[:, i] += k / a * B[:, i]
            if b > 0:
                nB[:, i] += (t[i + k + 1] - x) / b * B[:, i + 1]
                dB[:, i] -= k / b * B[:, i + 1]
        B = nB
    return B, dB


def _exact_assembly(case, seed):
    n, p = case["n"], case["p"]
    q, m = p + 1, n + p - 2
    gx, gw = np.polynomial.legendre.leggauss(q)
    x = ((np.arange(n)[:, None] + 0.5 * (gx[None, :] + 1.0)) / n).reshape(-1)
    w = np.tile(0.5 * gw / n, n)
    B, dB = (b[:, 1:-1] for b in _bsplines(n, p, x))
    Bt, dBt, x, w = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (B.T, dB.T, x, w))
    D = 2 * p + 1

    def pairs(f, g):
        """W[i, delta, q] = f_i(q) g_{i + delta}(q), zero outside the range."""
        out = torch.zeros(m, D, len(x), dtype=torch.float64, device="cuda")
        for k in range(D):
            s = k - p
            lo, hi = max(0, -s), min(m, m - s)
            if hi > lo:
                out[lo:hi, k] = f[lo:hi] * g[lo + s:hi + s]
        return out.reshape(m * D, -1)

    vv, vd, dv, dd = pairs(Bt, Bt), pairs(Bt, dBt), pairs(dBt, Bt), pairs(dBt, dBt)
    one = torch.ones_like(x)
    if case["geom"] == "annulus":
        P = [(1.0, 0.0), (1.0, 1.0), (0.0, 1.0)]
        wt = [1.0, math.sqrt(0.5), 1.0]
        b = [(1 - x) ** 2, 2 * x * (1 - x), x ** 2]
        db = [-2 * (1 - x), 2 - 4 * x, 2 * x]
        W = sum(wt[k] * b[k] for k in range(3))
        dW = sum(wt[k] * db[k] for k in range(3))
        c, dc = [], []
        for a in range(2):
            num = sum(wt[k] * P[k][a] * b[k] for k in range(3))
            dnum = sum(wt[k] * P[k][a] * db[k] for k in range(3))
            c.append(num / W)
            dc.append((dnum - num / W * dW) / W)
        r = 1.0 + x  # direction 1, the radius
        X, Y = (c[a][:, None] * r[None, :] for a in range(2))  # [xi2][xi1]
        j1 = [c[a][:, None] * one[None, :] for a in range(2)]
        j2 = [dc[a][:, None] * r[None, :] for a in range(2)]
    else:
        X, Y = one[:, None] * x[None, :], x[:, None] * one[None, :]
        o, z = one[:, None] * one[None, :], torch.zeros(len(x), len(x), dtype=torch.float64, device="cuda")
        j1, j2 = [o, z], [z, o]
    g11, g12, g22 = (sum(a * b for a, b in zip(u, v)) for u, v in ((j1, j1), (j1, j2), (j2, j2)))
    det = (j1[0] * j2[1] - j1[1] * j2[0]).abs()
    gram = g11 * g22 - g12 * g12
    w3 = w[:, None, None] * w[None, :, None] * w[None, None, :] * det[None]
    kap = torch.ones(1, 1, 1, dtype=torch.float64, device="cuda")
    if case["kappa"]:
        om, ph, sigma = _kappa(seed + 17)
        ab = X[..., None] * om[:, 0] + Y[..., None] * om[:, 1] + ph  # [q2, q1, M]
        bz = x[:, None] * om[:, 2]
        s = torch.einsum("yxm,zm->zyx", torch.cos(ab), torch.cos(bz))
        s -= torch.einsum("yxm,zm->zyx", torch.sin(ab), torch.sin(bz))
        kap = torch.exp(sigma * math.sqrt(2.0 / om.shape[0]) * s)
        del ab, bz, s
    C = kap * w3

    def contract(W3, W2, W1, coef):
        Q = len(x)
        t = (W3 @ coef.reshape(Q, Q * Q)).reshape(-1, Q, Q)
        t = torch.matmul(W2, t)
        return torch.matmul(t.reshape(-1, Q), W1.T).reshape(W3.shape[0], W2.shape[0], W1.shape[0])

    K = contract(vv, vv, dd, C * (g22 / gram))
    K += contract(vv, dd, vv, C * (g11 / gram))
    K += contract(dd, vv, vv, C.expand(len(x), -1, -1))
    if case["geom"] == "annulus":
        K -= contract(vv, vd, dv, C * (g12 / gram))
        K -= contract(vv, dv, vd, C * (g12 / gram))
    i = torch.arange(m, device="cuda")[:, None] + torch.arange(-p, p + 1, device="cuda")[None, :]
    ok = (i >= 0) & (i < m)
    keep = ok[:, None, None, :, None, None] & ok[None, :, None, None, :, None] & ok[None, None, :, None, None, :]
    K = K.reshape(m, D, m, D, m, D).permute(0, 2, 4, 1, 3, 5)
    val = K[keep]
    del K, keep
    f = w3
    if seed % 2:  # the sine source
        s = (torch.sin(math.pi * v) for v in (X, Y))
        f = w3 * (3.0 * math.pi ** 2) * (next(s) * next(s))[None] * torch.sin(math.pi * x)[:, None, None]
    F = torch.einsum("zyx,cz,by,ax->cba", f.contiguous(), Bt, Bt, Bt) if len(x) <= 64 else \
        torch.matmul(torch.matmul(Bt, torch.einsum("zyx,cz->cyx", f, Bt)), Bt.T)
    return {"rowptr": None, "col": None, "val": val, "F": F.reshape(-1)}
