"""The work a user of this framework has it do, as cases that can be timed and checked.

Three kinds of call, all through the public entry points:

* ``run``: a whole job of the binding (``HOTRG``): the site tensors from host temperatures and
  field (``init_tensor``), a schedule of coarse-graining steps along x, y, z, t, and the
  observables read back (ln Z/V; with the impure tensors E/V, <sigma sigma> and <sigma> too).
  This is what the benchmark, the T_c bracket and the temperature scans do.
* ``step``: one step of a tensor given by the caller (``set_tensor``, ``step``, ``tensor``):
  ragged bond dimensions, a general (not Ising) tensor, the whole coarse tensor back.
* ``isometry``: ``hotrg_isometry_noalloc`` of the C ABI on caller-owned device buffers.

Results of the mixed modes (FP32-stored tensors) are handed on in FP32, the precision those
modes keep; results of the FP64-stored modes stay FP64.
"""

from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1911_12954_gb300 import HOTRG, library_path

T_LO, T_HI = 6.60, 6.72           # temperatures of the sweeps and of the fixed-temperature runs
STORED_F64 = ("fp64", "fp64oz")
# dense multiply-add rate (TFLOP/s) a precision mode can count on: bounds the cost of drawn cases
RATE = {"fp16x3": 650.0, "tf32x3": 220.0, "fp32": 20.0, "fp64oz": 75.0, "fp64": 1.1}


def listed():
    def run(name, precision, batch, dcut, steps, h=0.0, impure=0, graphs=False):
        return dict(name=name, kind="run", precision=precision, batch=batch, dcut=dcut, steps=steps, h=h,
                    impure=impure, graphs=graphs)

    return [
        # the smallest call: one isometry of a small tensor, inside a caller's own memory
        dict(name="isometry_d4", kind="isometry", d0=4, d1=4, d2=4, d3=4, mu=0, nu=2, dcut=6),
        # the largest tensor that entry takes, ragged: FP64 Gram build and 64 x 64 eigenproblems
        dict(name="isometry_d8", kind="isometry", d0=8, d1=8, d2=7, d3=8, mu=3, nu=1, dcut=8),
        # one step of a caller's ragged tensor, FP32 CUDA cores, whole tensor back
        dict(name="step_ragged_fp32", kind="step", precision="fp32", d0=5, d1=3, d2=6, d3=4, mu=1, dcut=7),
        # the same kind of call on the tensor cores (dense: no symmetry in the entries)
        dict(name="step_ragged_fp16x3", kind="step", precision="fp16x3", d0=6, d1=5, d2=5, d3=7, mu=2, dcut=6),
        # the 16^4 reference run: FP64 throughout, one temperature
        run("ising16_d4_fp64", "fp64", 1, 4, 16),
        # one round of a T_c bracket at a small cut: 8 temperatures to 1024^4, replayed graphs
        run("tc_sweep_d4", "fp16x3", 8, 4, 40, graphs=True),
        # an energy / magnetisation scan at a small cut: T, S and M of 4 temperatures in a field
        run("scan_d5_impure", "fp16x3", 4, 5, 8, h=1e-5, impure=3),
        # the other tensor-core mode, in a field, at the cut between the small and the large ones
        run("field_d6_tf32x3", "tf32x3", 1, 6, 8, h=1e-5),
        # the FP64-grade reference the mixed runs are checked against
        run("reference_d6_fp64oz", "fp64oz", 1, 6, 6),
        # the headline run: D_cut = 8, T near T_c, h = 0
        run("ising1024_d8", "fp16x3", 1, 8, 6),
        # the batched sweep in a field with the impure tensors (pure, sigma, sigma sigma)
        run("sweep_d8_impure", "fp16x3", 2, 8, 4, h=1e-5, impure=3),
        # the next cut up, odd: every extent ragged against the tiles
        run("ising1024_d9", "fp16x3", 1, 9, 5),
    ]


def draw(rng):
    while True:
        kind = rng.choice(["isometry", "step", "run", "run", "run"])
        if kind == "isometry":
            d = [rng.randint(2, 8) for _ in range(4)]
            mu, nu = rng.sample(range(4), 2)
            return dict(kind=kind, d0=d[0], d1=d[1], d2=d[2], d3=d[3], mu=mu, nu=nu, dcut=rng.randint(2, 10))
        if kind == "step":
            c = dict(kind=kind, precision=rng.choice(["fp16x3", "fp16x3", "tf32x3", "fp32", "fp64"]))
            c |= {"d%d" % n: rng.randint(2, 7) for n in range(4)}
            c |= dict(mu=rng.randrange(4), dcut=rng.randint(3, 8))
            dims = _dims(c)
            if math.prod(dims) > 1100 or _main_flops(dims, c["mu"], c["dcut"]) > 0.02 * RATE[c["precision"]] * 1e12:
                continue
            return c
        prec = rng.choice(["fp16x3", "fp16x3", "fp16x3", "fp16x3", "tf32x3", "fp64", "fp64oz"])
        dcut = {"fp16x3": rng.randint(3, 9), "tf32x3": rng.randint(3, 7), "fp64": rng.randint(3, 4),
                "fp64oz": rng.randint(4, 7)}[prec]
        batch = max(1, int(math.exp(rng.uniform(0.0, math.log(16.5)))))
        impure = rng.choice([0, 0, 3])
        # <sigma> near T_c takes up rounding with the volume (its susceptibility grows): few steps
        steps = rng.randint(8, 40) if dcut <= 4 and not impure else rng.randint(4, 8)
        # the impure tensors are run in a field that picks a vacuum; the pure runs mostly without
        h = rng.choice([1e-5, 1e-4]) if impure else rng.choice([0.0, 0.0, 1e-5])
        c = dict(kind="run", precision=prec, batch=batch, dcut=dcut, steps=steps, h=h, impure=impure,
                 graphs=rng.choice([False, True]))
        if _run_flops(c, dense=True) > 1.0 * RATE[prec] * 1e12 or _operand_bytes(c) > 60e9:
            continue
        return c


# ------------------------------------------------------------------ sizes


def _dims(case):
    return [case["d%d" % n] for n in range(4)]


def _main_flops(dims, mu, dcut):
    """Block-spin product, 2 flops per multiply-add, with the cheapest closing direction."""
    chi = [dims[n] if n == mu else min(dims[n] ** 2, dcut) for n in range(4)]
    best = None
    for c in range(4):
        if c == mu:
            continue
        a, b = [n for n in range(4) if n not in (mu, c)]
        rows = chi[a] * chi[b] * dims[c] ** 2 * dims[mu]
        f = 2.0 * rows * rows * dims[a] ** 2 * dims[b] ** 2 * dims[mu]
        best = f if best is None else min(best, f)
    return best


def _shapes(case):
    """(bond dimensions, direction) of every step."""
    if case["kind"] != "run":
        return [(_dims(case), case["mu"])]
    dims, out = [2, 2, 2, 2], []
    for i in range(case["steps"]):
        mu = i % 4
        out.append((list(dims), mu))
        dims = [dims[n] if n == mu else min(dims[n] ** 2, case["dcut"]) for n in range(4)]
    return out


def _products(case, k):
    return 1 if not case.get("impure") else (4 if k == 0 else 5)


def _run_flops(case, dense=False):
    # without a field the tensors conserve the Z2 charge: a quarter of the product's terms is not zero
    part = 1.0 if dense or case.get("h", 1.0) != 0.0 else 0.25
    f = sum(_main_flops(d, mu, case["dcut"]) * _products(case, k) for k, (d, mu) in enumerate(_shapes(case)))
    return f * part * case.get("batch", 1)


def _operand_bytes(case):
    d = case["dcut"]
    width = {"fp16x3": 4, "tf32x3": 8, "fp64oz": 10, "fp64": 8, "fp32": 4}[case["precision"]]
    return case["batch"] * (3 if case["impure"] else 1) * d ** 10 * (2 * width + 8)


def work(case):
    """Every tensor read once and written once per step; the block-spin product's nonzero terms."""
    if case["kind"] == "isometry":
        dims = _dims(case)
        E = math.prod(d * d for d in dims)
        Dn, Dm = dims[case["nu"]], dims[case["mu"]]
        n = Dn * Dn
        flops = 4 * Dn * Dm * E + 4 * 2.0 * n * n * Dm * Dm + 2 * 9.0 * n ** 3
        return {"bytes": 8 * (E + n * min(n, case["dcut"])), "flops": flops}
    size = 8 if case["precision"] in STORED_F64 else 4
    nt = 3 if case.get("impure") else 1
    total = 0
    for dims, mu in _shapes(case):
        new = [dims[n] if n == mu else min(dims[n] ** 2, case["dcut"]) for n in range(4)]
        total += math.prod(d * d for d in dims) + math.prod(d * d for d in new)
    return {"bytes": size * nt * case.get("batch", 1) * total, "flops": _run_flops(case)}


# ------------------------------------------------------------------ inputs


def _temperatures(case, seed):
    rng = np.random.default_rng(seed)
    return np.sort(rng.uniform(T_LO, T_HI, case["batch"]))


def _tensor(dims, seed):
    """A seeded tensor whose entries fall off with the leg indices like a coarse-grained one."""
    rng = np.random.default_rng(seed)
    t = rng.standard_normal(tuple(x for d in dims for x in (d, d)))
    for leg in range(8):
        n = t.shape[leg]
        t = t * (0.6 ** np.arange(n)).reshape([n if i == leg else 1 for i in range(8)])
    return t


_LIB = None


def _watches_x(case):
    """Pure runs read the degeneracy indicator X too. Near T_c every step doubles its sensitivity
    along one direction, so mixed runs to large volumes are compared by ln Z/V alone."""
    return not case["impure"] and case["steps"] <= (16 if case["precision"] in STORED_F64 else 8)


def _c_abi():
    global _LIB
    if _LIB is None:
        _LIB = ctypes.CDLL(library_path())
        p = ctypes.c_void_p
        _LIB.hotrg_isometry_noalloc.restype = ctypes.c_int
        _LIB.hotrg_isometry_noalloc.argtypes = [p, ctypes.POINTER(ctypes.c_int), ctypes.c_int, ctypes.c_int,
                                                ctypes.c_int, p, p, p, p]
    return _LIB


def prepare(case, seed):
    if case["kind"] == "isometry":
        dims = _dims(case)
        n = dims[case["nu"]] ** 2
        chi = min(n, case["dcut"])
        T = _device_tensor(dims, seed)
        return dict(case=case, lib=_c_abi(), T=T, dims=(ctypes.c_int * 4)(*dims),
                    U=torch.zeros(n, chi, dtype=torch.float64, device="cuda"),
                    eps=torch.zeros(2, dtype=torch.float64, device="cuda"),
                    primed=torch.zeros(1, dtype=torch.int32, device="cuda"))
    if case["kind"] == "step":
        dims = _dims(case)
        ctx = HOTRG(batch=1, dcut_max=max(dims + [case["dcut"]]), precision=case["precision"],
                    schedule=[(case["mu"], case["dcut"])], dims0=dims)
        return dict(case=case, ctx=ctx, T=_tensor(dims, seed))
    ctx = HOTRG(batch=case["batch"], dcut_max=case["dcut"], precision=case["precision"], impure=case["impure"],
                schedule=[(i % 4, case["dcut"]) for i in range(case["steps"])], graphs=case["graphs"])
    return dict(case=case, ctx=ctx, beta=1.0 / _temperatures(case, seed))


def _device_tensor(dims, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    t = torch.randn([x for d in dims for x in (d, d)], generator=g, dtype=torch.float64, device="cuda")
    for leg in range(8):
        n = t.shape[leg]
        w = 0.6 ** torch.arange(n, dtype=torch.float64, device="cuda")
        t = t * w.reshape([n if i == leg else 1 for i in range(8)])
    return (t / t.norm()).contiguous()


# ------------------------------------------------------------------ one pass


def run(state):
    case = state["case"]
    if case["kind"] == "isometry":
        st = state["lib"].hotrg_isometry_noalloc(state["T"].data_ptr(), state["dims"], case["mu"], case["nu"],
                                                 case["dcut"], state["U"].data_ptr(), state["eps"].data_ptr(),
                                                 state["primed"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if st != 0:
            raise RuntimeError("hotrg_isometry_noalloc: status %d" % st)
        return dict(U=state["U"], eps=state["eps"], primed=state["primed"])
    ctx = state["ctx"]
    stored = np.float64 if case["precision"] in STORED_F64 else np.float32
    if case["kind"] == "step":
        ctx.set_tensor(state["T"])
        ctx.step(case["mu"], case["dcut"])
        info = ctx.step_info(1)
        return dict(T=ctx.tensor().astype(stored, copy=False), ln_c=np.array([info["ln_c"]], dtype=stored))
    ctx.init_tensor(state["beta"], case["h"])
    for i in range(case["steps"]):
        ctx.step(i % 4, case["dcut"])
    out = dict(lnZ=ctx.lnZ())
    if case["impure"]:
        out["E"], out["ss"] = ctx.energy()
        out["m"] = ctx.magnetization()
    if _watches_x(case):
        out["X"] = ctx.x_indicator(0)
    return {k: v.astype(stored, copy=False) for k, v in out.items()}


# ------------------------------------------------------------------ the same in 64 bits

_DEV = "cuda" if torch.cuda.is_available() else "cpu"


def exact(case, seed):
    if case["kind"] == "isometry":
        T = _device_tensor(_dims(case), seed)
        U, eps, primed = _isometry(T, case["mu"], case["nu"], case["dcut"])
        return dict(U=U, eps=torch.tensor(eps, dtype=torch.float64), primed=None)
    # plain FP64 products: about 1 TFLOP/s
    if _run_flops(case, dense=True) > 1.2e13:
        return None
    if case["kind"] == "step":
        T = torch.from_numpy(_tensor(_dims(case), seed)).to(_DEV)
        (T,), c = _coarse([T / T.norm().item()], case["mu"], case["dcut"], 0)
        return dict(T=T.cpu(), ln_c=np.array([math.log(c)]))
    temps = _temperatures(case, seed)
    if len(temps) * case["steps"] * 0.03 > 18:
        return None
    out = dict(lnZ=[], E=[], ss=[], m=[], X=[])
    for t in temps:
        ts, lnz = _site(1.0 / t, case["h"], case["impure"])
        for k in range(case["steps"]):
            ts, c = _coarse(ts, k % 4, case["dcut"], k)
            lnz += math.log(c) / 2 ** (k + 1)
        tr = [_trace(x) for x in ts]
        out["lnZ"].append(lnz + math.log(tr[0]) / 2 ** case["steps"])
        if case["impure"]:
            out["ss"].append(tr[2] / tr[0])
            out["m"].append(tr[1] / tr[0])
            out["E"].append(-4.0 * tr[2] / tr[0] - case["h"] * tr[1] / tr[0])
        if _watches_x(case):
            M = ts[0]
            for _ in range(3):
                M = torch.diagonal(M, dim1=2, dim2=3).sum(-1)
            out["X"].append(float(torch.trace(M)) ** 2 / float(torch.trace(M @ M)))
    return {k: np.array(v) for k, v in out.items() if v}


def _site(beta, h, impure):
    """Site tensors: T = sum_s e^{beta h s} prod_j W[s, i_j], S with a further factor s."""
    W = np.array([[math.sqrt(math.cosh(beta)), s * math.sqrt(math.sinh(beta))] for s in (1.0, -1.0)])
    T = S = 0.0
    for i, s in enumerate((1.0, -1.0)):
        p = np.ones(())
        for _ in range(8):
            p = np.multiply.outer(p, W[i])
        T = T + math.exp(beta * h * s) * p
        S = S + s * math.exp(beta * h * s) * p
    c = float(np.linalg.norm(T))
    ts = [T / c, S / c] if impure else [T / c]
    return [torch.from_numpy(np.ascontiguousarray(x)).to(_DEV) for x in ts], math.log(c)


def _trace(T):
    t = T
    for _ in range(4):
        t = torch.diagonal(t, dim1=0, dim2=1).sum(-1)
    return float(t)


def _half_gram(T, leg, kleg):
    rest = [i for i in range(8) if i not in (leg, kleg)]
    M = T.permute(leg, kleg, *rest).reshape(T.shape[leg] * T.shape[kleg], -1)
    return (M @ M.T).reshape(T.shape[leg], T.shape[kleg], T.shape[leg], T.shape[kleg])


def _isometry(T, mu, nu, dcut):
    """Isometry of the HOSVD of two tensors joined along mu, from the side (nu or nu') with the
    smaller discarded weight, in the canonical gauge (clusters of 1e-10, pivot ties of 1e-8)."""
    D = T.shape[2 * nu]
    chi = min(D * D, dcut)
    cand, eps, lam0 = [], [], None
    for side in range(2):
        g1, g2 = _half_gram(T, 2 * nu + side, 2 * mu + 1), _half_gram(T, 2 * nu + side, 2 * mu)
        G = torch.einsum("akbl,ckdl->acbd", g1, g2).reshape(D * D, D * D).cpu().numpy()
        lam, V = np.linalg.eigh((G + G.T) / 2)
        lam, V = lam[::-1], V[:, ::-1]
        lam0 = lam[0] if lam0 is None else lam0
        eps.append(float(lam[chi:].sum()))
        U, start = np.zeros((D * D, chi)), 0
        while start < chi:
            end = start + 1
            while end < D * D and lam[end - 1] - lam[end] <= 1e-10 * abs(lam[0]):
                end += 1
            P = V[:, start:end] @ V[:, start:end].T
            norm = np.diag(P).copy()
            for t in range(start, min(end, chi)):
                i = int(np.argmax(norm >= (1 - 1e-8) * norm.max()))
                g = P[:, i] - U[:, start:t] @ U[i, start:t]
                U[:, t] = g / math.sqrt(norm[i])
                norm -= U[:, t] ** 2
            start = end
        q, r = np.linalg.qr(U)
        cand.append(q * np.where(np.diag(r) < 0, -1.0, 1.0))
    primed = int(eps[0] - eps[1] > 1e-9 * (abs(eps[0]) + abs(eps[1])) + 1e-13 * abs(lam0))
    return torch.from_numpy(np.ascontiguousarray(cand[primed])).to(T.device), eps, primed


def _pair(T1, T2, mu, dirs, U):
    """The block-spin contraction of T1 and T2 along mu with the isometries of the other legs."""
    a, b, c = dirs
    order = [2 * a, 2 * a + 1, 2 * b, 2 * b + 1, 2 * c, 2 * c + 1, 2 * mu, 2 * mu + 1]
    P, Q = T1.permute(order), T2.permute(order)
    A = torch.einsum("aAbBcCmM,aiX->XibBAcCmM", P, U[a])
    A = torch.einsum("XibBAcCmM,bjY->XYcCmijABM", A, U[b])
    B = torch.einsum("aAbBcCmM,pAZ->ZpaBbcCmM", Q, U[a])
    B = torch.einsum("ZpaBbcCmM,rBW->ZWcCMabprm", B, U[b])
    sa, sb = A.shape[:5], B.shape[:5]
    C = (A.reshape(math.prod(sa), -1) @ B.reshape(math.prod(sb), -1).T).reshape(*sa, *sb)
    del A, B
    C = torch.einsum("XYcCmZWdDM,cdU->XYUCmZWDM", C, U[c])
    C = torch.einsum("XYUCmZWDM,CDV->XZYWUVmM", C, U[c])
    back = [order.index(i) for i in range(8)]
    return C.permute(back).contiguous()


def _coarse(ts, mu, dcut, k):
    T = ts[0]
    dirs = [n for n in range(4) if n != mu]
    U = {}
    for n in dirs:
        u, _, _ = _isometry(T, mu, n, dcut)
        U[n] = u.reshape(T.shape[2 * n], T.shape[2 * n], -1)
    new = [_pair(T, T, mu, dirs, U)]
    if len(ts) > 1:
        S = ts[1]
        new.append((_pair(S, T, mu, dirs, U) + _pair(T, S, mu, dirs, U)) / 2)
        if k == 0:
            new.append(_pair(S, S, mu, dirs, U))
        else:
            new.append((_pair(ts[2], T, mu, dirs, U) + _pair(T, ts[2], mu, dirs, U)) / 2)
    c = new[0].norm().item()
    return [x / c for x in new], c
