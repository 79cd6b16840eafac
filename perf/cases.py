"""The work that is measured: what a program that uses this library has it do, through the
public entry points, from the smallest factorisation to a full-size coarse-graining step.

The whole calls are a run of the smallest configuration, one full-size step, a temperature
sweep and the derivatives of a run; the others are the single layers that a step is made
of (the contractions of Eqs. 6-7 in each arithmetic, the swap's product with its generated
sketch, the orthonormalisation and the core SVD), called as the building blocks they are.
"""
import math

import numpy as np
import torch

import paper_2412_14104_gb300 as tg

PREC = {"fp64": tg.FP64, "tf32x3": tg.TF32X3, "bf16x3": tg.BF16X3, "bf16x6": tg.BF16X6, "ozaki": tg.OZAKI}


def listed():
    return [
        # the smallest core SVD: a bond of 6 doubled by the oversampling, one of dozens in
        # every step of a small run (its time is launches, synchronisation and latency)
        {"name": "svd_12", "kind": "svd", "m": 12, "n": 12},
        # the core SVD of a chi = 48, r = 3 step (15 of them in each step)
        {"name": "svd_144", "kind": "svd", "m": 144, "n": 144},
        # one of the orthonormalisations of the squeezer Grams' subspace iterations at
        # chi = 48, r = 3 (rows chi^2, columns r chi; five for each of ten Grams in a step)
        {"name": "orth_tf32x3_2304x144", "kind": "orth", "m": 2304, "n": 144, "prec": "tf32x3"},
        # Eq. 6's bottleneck in float64: the plain FP64 form, here at chi = 16
        {"name": "c2_fp64_chi16", "kind": "contract", "shape": "c2", "chi": 16, "r": 2, "prec": "fp64"},
        # the same contraction in 3xTF32 at the size of the temperature sweeps (chi = 32)
        {"name": "c2_tf32x3_chi32", "kind": "contract", "shape": "c2", "chi": 32, "r": 2, "prec": "tf32x3"},
        # the second bottleneck contraction (strided in all three operands) in BF16x3
        {"name": "c4_bf16x3_chi24", "kind": "contract", "shape": "c4", "chi": 24, "r": 2, "prec": "bf16x3"},
        # the float64-grade form that the precision schedules use for the early full-size steps
        {"name": "c2_ozaki_chi24", "kind": "contract", "shape": "c2", "chi": 24, "r": 2, "prec": "ozaki"},
        # the bond swap's first product, its Gaussian sketch drawn while it is packed
        {"name": "sketch_tf32x3_chi24", "kind": "sketch", "chi": 24, "r": 2, "prec": "tf32x3"},
        # the smallest whole run: 4D Ising, chi = 6, 8 steps in float64
        {"name": "run_d4_chi6_fp64", "kind": "run", "d": 4, "chi": 6, "r": 2, "steps": 8},
        # a small temperature sweep: concurrent runs, order parameter after every step
        {"name": "sweep_chi8_fp64", "kind": "sweep", "chi": 8, "r": 2, "steps": 6, "nbeta": 8},
        # internal energy and magnetisation of a run: forward-mode derivatives
        {"name": "grad_d4_chi6", "kind": "grad", "d": 4, "chi": 6, "r": 2, "steps": 4},
        # one full-size split-precision step on a given state, as a resumed run makes it: the
        # state from host memory, then the step and its spectra
        {"name": "step_chi48_tf32x3", "kind": "step", "chi": 48, "r": 2, "prec": "tf32x3"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["svd", "svd", "orth", "contract", "contract", "contract", "contract", "sketch", "run", "step"])
    if kind == "svd":
        n = _log_int(rng, 2, 160)
        return {"kind": kind, "m": n if rng.random() < 0.5 else n + _log_int(rng, 1, 600), "n": n}
    if kind == "orth":
        n = _log_int(rng, 2, 160)
        return {"kind": kind, "m": n + _log_int(rng, 100, 100000), "n": n, "prec": rng.choice(["fp64", "tf32x3"])}
    if kind == "contract":
        prec = rng.choice(sorted(PREC))
        shape = rng.choice(["c2", "c4", "gram"])
        return {"kind": kind, "shape": shape, "chi": _log_int(rng, 4, 16 if prec == "fp64" else 28),
                "r": rng.choice([2, 2, 3]) if shape == "gram" else 2, "prec": prec}
    if kind == "sketch":
        return {"kind": kind, "chi": _log_int(rng, 12, 30), "r": rng.choice([2, 3]),
                "prec": rng.choice(["tf32x3", "bf16x3", "bf16x6"])}
    if kind == "step":
        prec = rng.choice(["fp64", "tf32x3", "bf16x3", "ozaki"])
        return {"kind": kind, "chi": _log_int(rng, 6, 14) if prec == "fp64" else _log_int(rng, 12, 32),
                "r": 2, "prec": prec}
    d = rng.choice([2, 3, 4])
    return {"kind": "run", "d": d, "chi": _log_int(rng, 3, {2: 24, 3: 12, 4: 8}[d]), "r": 2, "steps": rng.randint(3, 8)}


# --- inputs -------------------------------------------------------------------------------

def _normal(seed, shape):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)


def _empty(*shape):
    return torch.empty(shape, dtype=torch.float64, device="cuda")


def _geometry(case):
    """Modes (ext, stride, stride) and operand shapes of a contraction of the steady state,
    every leg chi and the oversampled lines r chi; einsum over the operands' own indices."""
    x, k = case["chi"], case["r"] * case["chi"]
    if case["shape"] == "c2":
        # q[(i0,kA),k,kX,g] = sum_{a,b} em[(i0,kA),a,b,k] F[a,kX,b,g]
        return dict(m=[(x * k, x * x * x, x * k * x), (x, 1, k * x)], n=[(k, x * x, x), (x, 1, 1)],
                    k=[(x, x * x, k * x * x), (x, x, x)], A=(x * k, x, x, x), B=(x, k, x, x),
                    C=(x * k, x, k, x), ein="eabk,axbg->ekxg")
    if case["shape"] == "c4":
        # out[i0,kG,k,g] = sum_{kA,kX} q[i0,kA,k,kX,g] P[kA,kX,kG]
        g = x * x
        return dict(m=[(x, k * x * k * x, g * x * x), (x, k * x, x), (x, 1, 1)], n=[(g, 1, x * x)],
                    k=[(k, x * k * x, k * g), (k, x, g)], A=(x, k, x, k, x), B=(k, k, g),
                    C=(x, g, x, x), ein="iakxg,axG->iGkg")
    # Gram of a panel of the subspace iterations: G = Y^T Y, a long sum
    return dict(m=[(k, 1, k)], n=[(k, 1, 1)], k=[(x ** 3, k, k)], A=(x ** 3, k), B=None, C=(k, k), ein="rp,rq->pq")


def _panel(case, seed):
    """Normal columns with decaying scales, as the sketched panels and cores have them."""
    m, n = case["m"], case["n"]
    decay = 0.9 if case["kind"] == "svd" else 0.98
    return _normal(seed, (m, n)) * decay ** torch.arange(n, dtype=torch.float64, device="cuda")


def _couplings(case, seed):
    """Couplings around the critical one of the dimension, with a small field."""
    u = np.random.default_rng(seed).random(2)
    beta = {2: 0.4407, 3: 0.22165, 4: 0.1497}[case.get("d", 4)]
    return beta * (0.99 + 0.02 * u[0]), 1e-3 * (0.5 + u[1])


def _state(case, seed):
    """A split site tensor (A, s, B) with orthonormal factors and a decaying spectrum, in
    host memory."""
    x = case["chi"]

    def whiten(G):  # W with W G W^T = 1
        return torch.from_numpy(np.linalg.inv(np.linalg.cholesky(G.cpu().numpy()))).cuda()

    Y = _normal(seed, (x ** 4, x))
    A = (Y @ whiten(Y.T @ Y).T).reshape((x,) * 5).cpu().numpy()
    Y = _normal(seed + (1 << 20), (x, x ** 4))
    B = (whiten(Y @ Y.T) @ Y).reshape((x,) * 5).cpu().numpy()
    s = 0.9 ** np.arange(x)
    return A, s / np.linalg.norm(s), B


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed)
    if kind == "svd":
        m, n = case["m"], case["n"]
        st.update(A=_panel(case, seed), U=_empty(m, n), S=_empty(n), V=_empty(n, n),
                  w=torch.cos(torch.arange(m, dtype=torch.float64, device="cuda")))
    elif kind == "orth":
        m, n = case["m"], case["n"]
        st.update(Y=_panel(case, seed), Q=_empty(m, n), R=_empty(n, n))
    elif kind == "contract":
        g = _geometry(case)
        A = _normal(seed, g["A"])
        st.update(g=g, A=A, B=A if g["B"] is None else _normal(seed + (1 << 20), g["B"]), C=_empty(*g["C"]))
    elif kind == "sketch":
        x = case["chi"]
        st.update(A=_normal(seed, (x * x, x ** 3)), C=_empty(x * x, x * case["r"] * x))
    elif kind == "run":
        st.update(ctx=tg.Context(case["chi"], case["r"], 2, seed=seed & 0xFFFF), at=_couplings(case, seed))
    elif kind == "sweep":
        b, h = _couplings(case, seed)
        st.update(ctx=tg.Context(case["chi"], case["r"], 2, seed=seed & 0xFFFF),
                  betas=np.linspace(0.97 * b, 1.03 * b, case["nbeta"]), h=h)
    elif kind == "grad":
        st.update(ctx=tg.Context(case["chi"], case["r"], 2, seed=seed & 0xFFFF), at=_couplings(case, seed))
    else:
        A, s, B = _state(case, seed)
        st.update(ctx=tg.Context(case["chi"], case["r"], 2, seed=seed & 0xFFFF, precision=PREC[case["prec"]]),
                  A=A, s=s, B=B)
    return st


# --- the calls ----------------------------------------------------------------------------

def _signed(U, V, w):
    """Pairs of singular vectors with w . u > 0 (an SVD leaves the sign of each pair open)."""
    sg = torch.where(w @ U < 0, -1.0, 1.0)
    return U * sg, V * sg


def _sketch_modes(case):
    x, ell = case["chi"], case["r"] * case["chi"]
    # W0[(a,k),(b,p)] = sum_j R[(a,k),j] Omega[(b,j),p]
    return [(x * x, x ** 3, x * ell)], [(x, x ** 3 * ell, ell), (ell, 1, 1)], [(x ** 3, 1, ell)]


def _spectra(ctx, d):
    return [ctx.spectrum(k) for k in range(d + 1)]


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "svd":
        tg.svd(state["A"], state["U"], state["S"], state["V"])
        U, V = _signed(state["U"], state["V"], state["w"])
        return {"U": U, "S": state["S"], "V": V}
    if kind == "orth":
        k = tg.orth(state["Y"], state["Q"], state["R"], precision=PREC[case["prec"]])
        return {"Q": state["Q"], "R": state["R"], "k": k}
    if kind == "contract":
        g = state["g"]
        return tg.contract(g["m"], g["n"], g["k"], state["A"], state["B"], state["C"], precision=PREC[case["prec"]])
    if kind == "sketch":
        m, n, k = _sketch_modes(case)
        return tg.contract_sketch(m, n, k, state["A"], state["seed"] & 0xFFFF, 0x500, state["C"],
                                  precision=PREC[case["prec"]])
    ctx = state["ctx"]
    if kind == "run":
        beta, h = state["at"]
        ctx.init_ising(beta, h, case["d"]).rg_step(case["steps"])
        return {"lnZ": ctx.lnZ(), "spectra": _spectra(ctx, case["d"]), "X": ctx.order_parameter(0),
                "state": ctx.get_state()}
    if kind == "sweep":
        lnz, X = ctx.sweep_observables(state["betas"], state["h"], 4, case["steps"])
        return {"lnZ": lnz, "X": X}
    if kind == "grad":
        beta, h = state["at"]
        ctx.init_ising(beta, h, case["d"]).rg_step(case["steps"])
        db, dh, _ = ctx.grad()
        return {"lnZ": ctx.lnZ(), "dbeta": db, "dh": dh}
    ctx.set_state(state["A"], state["s"], state["B"], 10, 0.0).rg_step(1)
    info = ctx.step_info()
    out = {"lnc": info.lnc, "partial_lnz": info.partial_lnz, "dims": np.array(list(info.dims)),
           "spectra": _spectra(ctx, 4)}
    if case["prec"] == "fp64":
        # float64 steps are checkpointed as they are; a split run's full-size state stays
        # on the device between steps
        out["state"] = ctx.get_state()
    return out


# --- what a pass cannot do without --------------------------------------------------------

def _step_flops(x, r, d):
    """Contraction and compressed bond swap of one steady-state step, 4D exponents less two
    for each missing leg direction."""
    return (8.0 * r * r + 2.0 * r + 8.0) * float(x) ** (2 * d - 1)


def work(case):
    kind = case["kind"]
    if kind in ("svd", "orth"):
        m, n = case["m"], case["n"]
        return {"bytes": 8.0 * (2 * m * n + n * n), "flops": (6.0 if kind == "svd" else 4.0) * m * n * n}
    if kind == "contract":
        g = _geometry(case)
        M, N, K = (math.prod(e[0] for e in g[i]) for i in "mnk")
        return {"bytes": 8.0 * (M * K + (0 if g["B"] is None else N * K) + M * N), "flops": 2.0 * M * N * K}
    x, r = case["chi"], case["r"]
    if kind == "sketch":
        return {"bytes": 8.0 * (x ** 5 + r * x ** 4), "flops": 2.0 * r * float(x) ** 7}
    if kind == "step":
        return {"bytes": 8.0 * 4 * x ** 5, "flops": _step_flops(x, r, 4)}
    runs = case.get("nbeta", 1) * (1 if kind != "grad" else 7)  # two passes with a tangent each
    d = case.get("d", 4)
    return {"bytes": 8.0 * 2 * x ** (d + 1) * runs, "flops": runs * case["steps"] * _step_flops(x, r, d)}


# --- the same in 64 bits ------------------------------------------------------------------

def _philox_normal(seed, sid, rows, cols):
    """The sketch as published: Philox4x32-10 (Salmon et al. 2011), 53-bit uniforms, Box-Muller."""
    n = rows * cols
    p = torch.arange((n + 1) // 2, dtype=torch.int64, device="cuda")
    mask = 0xFFFFFFFF
    c = [p & mask, p >> 32, torch.zeros_like(p), torch.full_like(p, (seed >> 32) & mask)]
    k0, k1 = seed & mask, sid

    def mulhilo(a, x):  # 32 x 32 -> 64 bits without signed overflow
        lo16, hi16 = x & 0xFFFF, x >> 16
        low = a * lo16
        mid = a * hi16 + (low >> 16)
        return (mid >> 16) & mask, ((mid << 16) | (low & 0xFFFF)) & mask

    for _ in range(10):
        h0, l0 = mulhilo(0xD2511F53, c[0])
        h1, l1 = mulhilo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask

    def u53(hi, lo):
        return (((hi >> 5) << 26) + (lo >> 6)).double().add_(0.5).mul_(2.0 ** -53)

    rad = torch.sqrt(-2.0 * torch.log(u53(c[0], c[1])))
    ang = 2.0 * math.pi * u53(c[2], c[3])
    return torch.stack([rad * torch.cos(ang), rad * torch.sin(ang)], dim=1).reshape(-1)[:n].reshape(rows, cols)


def exact(case, seed):
    kind = case["kind"]
    if kind == "svd":
        A = _panel(case, seed)
        U, S, Vh = torch.linalg.svd(A, full_matrices=False)
        U, V = _signed(U, Vh.T, torch.cos(torch.arange(case["m"], dtype=torch.float64, device="cuda")))
        return {"U": U, "S": S, "V": V}
    if kind == "orth":
        Q, R = torch.linalg.qr(_panel(case, seed))
        sg = torch.where(torch.diagonal(R) < 0, -1.0, 1.0)
        return {"Q": Q * sg, "R": sg[:, None] * R, "k": case["n"]}
    if kind == "contract":
        g = _geometry(case)
        A = _normal(seed, g["A"])
        return torch.einsum(g["ein"], A, A if g["B"] is None else _normal(seed + (1 << 20), g["B"]))
    if kind == "sketch":
        x, ell = case["chi"], case["r"] * case["chi"]
        om = _philox_normal(seed & 0xFFFF, 0x500, x * x ** 3, ell).reshape(x, x ** 3, ell)
        return torch.einsum("rj,bjp->rbp", _normal(seed, (x * x, x ** 3)), om).reshape(x * x, x * ell)
    return None  # a whole run: many steps of the method itself
