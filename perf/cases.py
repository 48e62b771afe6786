"""Workloads of this library as its users run them, for timing and for comparing outputs.

Every case goes through the Python package: a domain (or a batch of domains, or the surrogate's
network) is set up once, then a pass restarts it from a checkpoint, advances it a number of steps
and reads the fields back into device memory.  `exact` restates the scheme in plain FP64 torch.
"""
import math

import numpy as np
import torch

from paper_2310_17214_gb300 import inputs as I
from paper_2310_17214_gb300 import surrogate as S
from paper_2310_17214_gb300._native import Batch, Domain, Mlp

R_GAS = 8.314
DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _flow(name, problem, nx, ny, nz, precision, steps, **opt):
    c = {"kind": "flow", "problem": problem, "nx": nx, "ny": ny, "nz": nz, "precision": precision,
         "steps": steps, "transport": "single", "moving": False}
    c.update(opt)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the verification channel: a heated disc, FP64, 128 x 64 cells; one kernel per step and
        # little work in it, so launches and the latency of one step count
        _flow("channel2d_128x64_fp64", "channel", 128, 64, 1, "fp64", 100),
        # the wall-bounded flame held by the inlet feedback (480 x 120): a small 2-D domain that
        # runs for tens of thousands of steps
        _flow("flame2d_480x120_fp32", "flame", 480, 120, 1, "fp32", 100),
        # the 2-D reactive bed in production precision
        _flow("bed2d_1024x256_fp32", "bed", 1024, 256, 1, "fp32", 50),
        # the same bed at ragged extents in FP64, as for reference runs
        _flow("bed2d_1001x251_fp64", "bed", 1001, 251, 1, "fp64", 20),
        # FP16-stored populations with mixture-averaged transport, ragged
        _flow("bed2d_771x301_fp16_mix", "bed", 771, 301, 1, "fp32_fp16", 40, transport="mixture"),
        # the 3-D reactive bed, the headline workload
        _flow("bed3d_256x128x128_fp32", "bed", 256, 128, 128, "fp32", 16),
        # a 3-D bed with FP16-stored populations, odd extents
        _flow("bed3d_251x123x118_fp16", "bed", 251, 123, 118, "fp32_fp16", 16),
        # the 64^3 crop in FP64, the size of comparisons with the reference solution
        _flow("bed3d_64x64x64_fp64", "bed", 64, 64, 64, "fp64", 16),
        # two-step mechanism integrated implicitly in every cell
        _flow("two_step_2048x512_fp32", "two_step", 2048, 512, 1, "fp32", 4),
        # the same bed with the learned chemistry
        {"name": "surrogate_2048x512_fp32", "kind": "surrogate", "nx": 2048, "ny": 512,
         "precision": "fp32", "engine": "warp_mma", "steps": 20},
        # 48 uneven channel beds advanced together (a parameter study)
        {"name": "batch_48_beds_fp32", "kind": "batch", "domains": 48, "base": 256,
         "precision": "fp32", "steps": 50},
        # an epoch of the surrogate's training
        {"name": "train_131072_rows", "kind": "train", "rows": 131072, "batch": 8192, "steps": 16},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["flow2d", "flow2d", "flow2d", "flow3d", "flow3d", "two_step", "surrogate",
                       "batch", "train"])
    prec = rng.choice(["fp32", "fp32", "fp64", "fp32_fp16"])
    if kind == "flow2d":
        problem = rng.choice(["channel", "calibration", "flame", "bed", "bed"])
        ny = log(48, 400)
        nx = max(96, min(1400, int(ny * rng.uniform(1.3, 4.5))))
        steps = max(10, min(100, (2_500_000 if prec == "fp64" else 10_000_000) // (nx * ny)))
        mix = problem == "bed" and prec != "fp64" and rng.random() < 0.3
        return _flow("", problem, nx, ny, 1, prec, steps,
                     transport="mixture" if mix else "single",
                     moving=problem == "bed" and rng.random() < 0.15)
    if kind == "flow3d":
        hi = 70 if prec == "fp64" else 128
        nx, ny, nz = max(56, log(40, 2 * hi)), log(32, hi), log(20, hi)
        steps = max(2, min(16, (3_000_000 if prec == "fp64" else 40_000_000) // (nx * ny * nz)))
        return _flow("", "bed", nx, ny, nz, prec, steps,
                     moving=rng.random() < 0.15)
    if kind == "two_step":
        ny = log(64, 400)
        nx = max(128, int(ny * rng.uniform(1.5, 4.0)))
        return _flow("", "two_step", nx, ny, 1, "fp32" if prec == "fp32_fp16" else prec,
                     2 if prec == "fp64" else 4)
    if kind == "surrogate":
        ny = log(64, 512)
        return {"kind": "surrogate", "nx": max(128, int(ny * rng.uniform(1.5, 4.0))), "ny": ny,
                "precision": "fp32" if prec == "fp32_fp16" else prec,
                "engine": rng.choice(["warp_mma", "warp_mma", "tcgen05"]),
                "steps": 4 if prec == "fp64" else 20}
    if kind == "batch":
        return {"kind": "batch", "domains": rng.randint(5, 40), "base": log(64, 200),
                "precision": "fp32" if prec == "fp64" else prec, "steps": rng.randint(20, 50)}
    rows = log(5000, 131072)
    return {"kind": "train", "rows": rows, "batch": log(512, 16384), "steps": rng.randint(4, 16)}


# ------------------------------------------------------------------ problems and inputs
def _problem(case):
    """The problem dictionary of a flow, surrogate or (per domain) batch case."""
    nx, ny, prec = case["nx"], case["ny"], case["precision"]
    problem = case.get("problem", "two_step")
    if problem == "channel":
        p = I.config1(nx, ny)
    elif problem == "calibration":
        p = I.di_channel(L=ny - 16, H=nx)
    elif problem == "flame":
        p = I.config6(nx, ny, precision=prec)
    elif problem == "two_step":
        chem = "surrogate" if case["kind"] == "surrogate" else "implicit"
        p = I.config4(nx, ny, precision=prec, chem=chem)
    elif case["nz"] > 1:
        p = I.config3(nx, ny, case["nz"], precision=prec)
    else:
        p = I.config2(nx, ny, precision=prec)
    if case.get("transport") == "mixture":
        p = I.mixture_transport(p)
    if case.get("moving"):
        p["u_s"] = [0.004, 0.002, 0.001]
    return p


def _grid(p):
    nz = p["nz"] if p["dim"] == 3 else 1
    ax = [torch.arange(n, dtype=torch.float64, device=DEV) for n in (nz, p["ny"], p["nx"])]
    return torch.meshgrid(*ax, indexing="ij")


def _waves(p, rng, modes=3):
    """A smooth seeded field in [-1, 1]."""
    Z, Y, X = _grid(p)
    s = torch.zeros_like(X)
    for _ in range(modes):
        k = rng.integers(1, 4, size=3)
        s += torch.cos(2 * math.pi * (k[0] * X / p["nx"] + k[1] * Y / p["ny"]
                                      + (k[2] * Z / p["nz"] if p["dim"] == 3 else 0.0))
                       + rng.uniform(0, 2 * math.pi))
    return s / modes


def _particles(p, rng, x0, amin, amax):
    """Phase field of ellipses / ellipsoids with tanh interfaces on a jittered grid from x0 to the
    outlet region, kept off non-periodic walls."""
    Z, Y, X = _grid(p)
    dim, eta = p["dim"], p["eta"]
    ext = [p["nx"] - x0 - 8, p["ny"], p["nz"] if dim == 3 else 1]
    amax = max(3.0, min(amax, ext[0] / 2.8, ext[1] / 3.4, ext[2] / 3.4 if dim == 3 else 1e9))
    amin = min(amin, 0.7 * amax)
    pitch = 2.0 * amax + 1.5 * eta
    num = [max(1, int(ext[a] / pitch)) if a < dim else 1 for a in range(3)]
    phi = torch.zeros_like(X)
    for i in range(num[0]):
        for j in range(num[1]):
            for k in range(num[2]):
                jit = rng.uniform(-0.4, 0.4, size=3) * eta
                c = [x0 + (i + 0.5) * ext[0] / num[0] + jit[0], (j + 0.5) * ext[1] / num[1] + jit[1],
                     (k + 0.5) * ext[2] / num[2] + jit[2]]
                a = np.sort(rng.uniform(amin, amax, size=3))[::-1]
                th, ps = rng.uniform(0, math.pi, size=2)
                dx, dy, dz = X - c[0], Y - c[1], Z - c[2]
                u = dx * math.cos(th) + dy * math.sin(th)
                v = -dx * math.sin(th) + dy * math.cos(th)
                if dim == 3:
                    u, dz = u * math.cos(ps) + dz * math.sin(ps), -u * math.sin(ps) + dz * math.cos(ps)
                    F = (u / a[0]) ** 2 + (v / a[1]) ** 2 + (dz / a[2]) ** 2
                    m = a[2]
                else:
                    F = (u / a[0]) ** 2 + (v / a[1]) ** 2
                    m = a[1]
                d = (F.sqrt() - 1.0) * m
                phi = torch.maximum(phi, 0.5 * (1.0 - torch.tanh(2.0 * d / eta)))
    return phi


def _inlet_profile(p):
    """Inlet speed over the cross-section (uniform, or a parabola between walls)."""
    _, Y, X = _grid(p)
    u = torch.full_like(X, p["u_in"])
    if p["inlet_parabolic"] == 1:
        s = Y + 0.5
        u = u * 4.0 * s * (p["ny"] - s) / p["ny"] ** 2
    return u


def _fields(p, seed, bed=None):
    """phi, T, Y, Ts, u of the problem's initial state (FP64, flat, on the GPU)."""
    rng = np.random.default_rng([seed, p["nx"], p["ny"]])
    Z, Yg, X = _grid(p)
    n = X.numel()
    K = p["K"]
    wave = _waves(p, rng)
    lo, hi = 16.0, max(28.0, min(64.0, p["nx"] / 4.0))
    Ts = None
    if p["name"].startswith("channel_"):
        phi = torch.as_tensor(I.di_channel_fields(p)["phi"], device=DEV).reshape(X.shape)
    elif p["name"].startswith("cfg1"):
        r = min(8.0, p["ny"] / 6.0)
        cx, cy = 0.25 * p["nx"] + rng.uniform(-2, 2), 0.5 * p["ny"] + rng.uniform(-2, 2)
        phi = 0.5 * (1.0 - torch.tanh(2.0 * (torch.hypot(X - cx, Yg - cy) - r) / p["eta"]))
    elif p["name"].startswith("cfg6"):
        phi = torch.zeros_like(X)
    else:
        b = bed or p["bed"]
        x0 = p["nx"] // 8 if K == 0 else hi + 14.0
        phi = _particles(p, rng, x0, b["amin"], b["amax"])
    if K:
        Yin = torch.tensor(p["Y_in"], dtype=torch.float64, device=DEV)
        Yb = torch.tensor(I.burnt_composition(p["Y_in"], p["species"], p["M"]),
                          dtype=torch.float64, device=DEV)
        if p["name"].startswith("cfg6"):  # burnt products downstream of a wrinkled front
            w = 0.5 * (1.0 + torch.tanh((X - p["nx"] / 4.0 - 3.0 * wave) / 4.0))
            Tb = I.adiabatic_temperature(p)
        else:  # an ignited pocket in the fresh mixture
            w = 0.5 * (torch.tanh((X - lo - 2.0 * wave) / 4.0) - torch.tanh((X - hi - 2.0 * wave) / 4.0))
            Tb = p["ignite"][2]
        T = p["T_in"] + (Tb - p["T_in"]) * w
        Y = Yin[:, None] + (Yb - Yin)[:, None] * w.reshape(1, n)
    else:
        T = torch.full_like(X, p["T_in"])
        Y = None
    T = (1.0 - phi) * T + phi * p["Ts_uniform"]
    if p["Ts_field"]:
        Ts = (p["Ts_uniform"] + 20.0 * (1.0 + wave) * phi).reshape(n)
    ux = _inlet_profile(p) * (1.0 - phi) * (1.0 + 0.1 * wave)
    u = torch.cat([ux.reshape(n)] + [torch.zeros(n, dtype=torch.float64, device=DEV)] * (p["dim"] - 1))
    f = {"phi": phi.reshape(n), "T": T.reshape(n), "Y": None if Y is None else Y.reshape(-1),
         "Ts": Ts, "u": u}
    if p.get("precision", "fp64") != "fp64":  # what an FP32 domain is handed
        f = {k: None if v is None else v.float() for k, v in f.items()}
    return f


def _dtype(prec):
    return (np.float64, torch.float64) if prec == "fp64" else (np.float32, torch.float32)


def _domain(p, f, prec):
    d = Domain(p, prec)
    npd = _dtype(prec)[0]
    d.set_phase_field(f["phi"], f["Ts"], dtype=npd)
    d.set_fields(f["T"], f["Y"], f["u"], dtype=npd)
    return d


def _names(p):
    return ["T"] + (["Y"] if p["K"] else []) + (["Ts"] if p["Ts_field"] else []) + ["u"]


def _split(p, buf):
    """The packed fields of Domain.get as one view per field."""
    n = p["nx"] * p["ny"] * (p["nz"] if p["dim"] == 3 else 1)
    size = {"T": 1, "Y": p["K"], "Ts": 1, "u": p["dim"]}
    out, off = {}, 0
    for name in _names(p):
        out[name] = buf[off:off + size[name] * n]
        off += size[name] * n
    return out


def _batch_problems(case):
    ps = I.config5(n=case["domains"], precision=case["precision"],
                   base=(case["base"], case["base"] // 2))
    return [dict(p, precision=case["precision"]) for p in ps]


def _train_inputs(case, seed):
    g = np.random.default_rng(seed)
    n = case["rows"]
    X = torch.as_tensor(np.clip(g.normal(size=(n, 8)), -3, 3), dtype=torch.float32, device=DEV)
    A = torch.as_tensor(g.normal(size=(8, 6)) / math.sqrt(8), dtype=torch.float32, device=DEV)
    B = torch.as_tensor(g.normal(size=(8, 6)) / math.sqrt(8), dtype=torch.float32, device=DEV)
    return X, (torch.sin(1.5 * (X @ A)) + 0.5 * torch.tanh(X @ B)).contiguous(), S.glorot(seed)


def _surrogate_net(p, seed):
    """Parameters and record of a network fitted to the two-step chemistry: random hidden layers, the
    output layer by least squares on backward-Euler increments of random flame states."""
    rng = np.random.default_rng([seed, 77])
    m = 12000
    Yin = np.asarray(p["Y_in"])
    M = np.asarray(p["M"])
    st = np.array([r["stoich"] for r in p["reactions"]])
    e1 = rng.uniform(0, 1, m) * Yin[0] / M[0]
    e2 = e1 * (1.0 - 0.1 * rng.uniform(0, 1, m) ** 2)
    Y = Yin[:, None] + M[:, None] * (st[0][:, None] * e1 + st[1][:, None] * e2)
    q = -(np.asarray(p["hf"])[:, None] * (Y - Yin[:, None])).sum(0) / (np.asarray(p["cp"])[:, None] * Y).sum(0)
    T = np.clip(p["T_in"] + q * rng.uniform(0.7, 1.05, m), 290.0, 2000.0)
    T[:200] = np.linspace(290.0, 2000.0, 200)
    Tt, Yt = torch.tensor(T), torch.tensor(np.maximum(Y, 0.0))
    rho = p["P0"] / (R_GAS * Tt * (Yt / torch.tensor(M)[:, None]).sum(0))
    dY, _ = _backward_euler(p, Tt, Yt, rho)
    X = np.concatenate([T[:, None], Yt.numpy().T, np.full((m, 1), p["P0"])], axis=1)
    theta_s = S.theta_scale(p)
    stats, Xn, Yn = S.normalisation(X, dY.numpy().T, theta_s)
    th = S.glorot(seed).astype(np.float64)
    h, off = Xn.astype(np.float64), 0
    for a, b in ((8, 64), (64, 64), (64, 64)):
        h = np.tanh(h @ th[off:off + a * b].reshape(a, b))
        off += a * b + b
    h1 = np.concatenate([h, np.ones((m, 1))], axis=1)
    W = np.linalg.solve(h1.T @ h1 + 1e-3 * m * np.eye(65), h1.T @ Yn)
    th[off:off + 384], th[off + 384:] = W[:64].reshape(-1), W[64]
    rec = S.make_surrogate(stats, X, theta_s, p["species"], 1e-6)
    return th.astype(np.float32), rec


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        X, Y, theta = _train_inputs(case, seed)
        return {"case": case, "net": Mlp(), "X": X, "Y": Y, "theta": theta}
    npd, td = _dtype(case["precision"])
    if kind == "batch":
        ps = _batch_problems(case)
        doms = [_domain(p, _fields(p, seed + 1000 * i, bed=p["bed"]), case["precision"])
                for i, p in enumerate(ps)]
        b = Batch(doms)
        b.autotune(5)
        bufs = [torch.empty(3 * d.N, dtype=td, device=DEV) for d in doms]
        return {"case": case, "batch": b, "doms": doms, "bufs": bufs, "npd": npd}
    p = _problem(case)
    p["precision"] = case["precision"]
    d = _domain(p, _fields(p, seed), case["precision"])
    s = {"case": case, "p": p, "dom": d, "npd": npd}
    if kind == "surrogate":
        theta, rec = _surrogate_net(p, seed)
        rec.engine = {"warp_mma": 0, "tcgen05": 1}[case["engine"]]
        net = Mlp()
        net.set_params(theta)
        d.set_surrogate(net, rec)
    s["checkpoint"] = d.get_state(torch.empty(d.state_bytes(), dtype=torch.uint8, device=DEV))
    total = sum(v for k, v in d._sizes().items() if k in _names(p))
    s["out"] = torch.empty(total, dtype=td, device=DEV)
    return s


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        net = state["net"]
        net.set_params(state["theta"])
        loss = net.train(state["X"], state["Y"], case["batch"], case["steps"], 1e-3)
        return {"loss": np.float32(loss), "theta": net.get_params()}
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        for d, b in zip(state["doms"], state["bufs"]):
            d.get("T", "u", dtype=state["npd"], out=b)
        return {"T": torch.cat([b[:b.numel() // 3] for b in state["bufs"]]),
                "u": torch.cat([b[b.numel() // 3:] for b in state["bufs"]])}
    d = state["dom"]
    d.set_state(state["checkpoint"])
    d.step(case["steps"])
    d.get(*_names(state["p"]), dtype=state["npd"], out=state["out"])
    return _split(state["p"], state["out"])


# ------------------------------------------------------------------ what a pass needs
def work(case):
    """Per step every population and field is read and written once (the phase field read); the
    operations are those of the update, the integrator and the network."""
    if case["kind"] == "train":
        rows = case["steps"] * min(case["rows"], case["batch"])
        return {"bytes": rows * 56 + case["steps"] * 9286 * 28, "flops": rows * 6 * 9216}
    fp = {"fp64": (8, 8), "fp32": (4, 4), "fp32_fp16": (4, 2)}[case["precision"]]
    ps = _batch_problems(case) if case["kind"] == "batch" else [_problem(case)]
    total = {"bytes": 0, "flops": 0}
    for p in ps:
        dim, K = p["dim"], p["K"]
        n = p["nx"] * p["ny"] * (p["nz"] if dim == 3 else 1)
        Q = 9 if dim == 2 else 19
        mom = 2 * 4 * (dim + 1) if fp[1] == 2 else 0
        b = 2 * Q * fp[1] + mom + fp[0] * (2 * (1 + K + (1 if p["Ts_field"] else 0)) + 1)
        f = 20 * Q + 60 * dim + K * (8 + 9 * dim) + (60 if K else 0)
        if case.get("problem") == "two_step":
            f += 900
        if case["kind"] == "surrogate":
            f += 2 * 9216
        total["bytes"] += case["steps"] * n * b
        total["flops"] += case["steps"] * n * f
    return total


# ------------------------------------------------------------------ the scheme in FP64 torch
def _backward_euler(p, T0, Y0, rho):
    """Increments (dY [K, n], dT [n]) of one backward-Euler step of the chemistry at frozen density
    (kg/m^3).  Newton on the reactions' progress per mass x_j and on T: the species follow from x."""
    h, rx = p["dt"], p["reactions"]
    J, K = len(rx), p["K"]
    kw = {"dtype": torch.float64, "device": T0.device}
    M, cp, hf = (torch.tensor(p[k], **kw)[:, None] for k in ("M", "cp", "hf"))
    st = torch.tensor([r["stoich"] for r in rx], **kw)
    Ms = (M.T * st)  # [J, K]
    n = T0.numel()
    x = torch.zeros(J, n, **kw)
    T = T0.clone()
    hm = Ms @ hf  # [J, 1]: heat released per progress is -hm
    cm = Ms @ cp
    for _ in range(25):
        Y = Y0 + Ms.T @ x
        pos = Y > 0
        C = torch.where(pos, rho * Y / M, torch.zeros_like(Y))
        dC = torch.where(pos, rho / M, torch.zeros_like(Y))
        A = torch.zeros(n, J + 1, J + 1, **kw)
        res = torch.zeros(n, J + 1, **kw)
        for j, r in enumerate(rx):
            kf = r["A"] * torch.exp(-r["EaR"] / T) * T ** r.get("b", 0.0)
            dkf = r["EaR"] / T ** 2 + r.get("b", 0.0) / T
            terms = [(kf, dkf, r["order"])]
            if r.get("reverse"):
                v = r["reverse"]
                dn = sum(r["stoich"])
                Kc = torch.exp(v["dS"] / R_GAS - v["dH"] / (R_GAS * T)) * \
                    (p.get("p_ref", 101325.0) / (R_GAS * T)) ** dn
                terms.append((-kf / Kc, dkf - (v["dH"] / (R_GAS * T * T) - dn / T), v["order"]))
            q, qT, qY = torch.zeros(n, **kw), torch.zeros(n, **kw), torch.zeros(K, n, **kw)
            for kk, dk, order in terms:
                used = [k for k in range(K) if order[k] != 0]
                t = kk.clone()
                for k in used:
                    t = t * C[k] ** order[k]
                q = q + t
                qT = qT + t * dk
                for k in used:
                    d = kk * torch.where(C[k] > 0, order[k] * C[k].clamp_min(1e-300) ** (order[k] - 1),
                                         torch.full_like(C[k], 1.0 if order[k] == 1 else 0.0)) * dC[k]
                    for m in used:
                        if m != k:
                            d = d * C[m] ** order[m]
                    qY[k] = qY[k] + d
            hr = h / rho
            res[:, j] = -(x[j] - hr * q)
            for i in range(J):
                A[:, j, i] = -hr * (Ms[i][:, None] * qY).sum(0)
            A[:, j, j] += 1.0
            A[:, j, J] = -hr * qT
        cps, heat = (cp * Y).sum(0), (hm * x).sum(0)
        res[:, J] = -(T - T0 + heat / cps)
        for i in range(J):
            A[:, J, i] = hm[i] / cps - heat * cm[i] / cps ** 2
        A[:, J, J] = 1.0
        dlt = torch.linalg.solve(A, res)
        x, T = x + dlt[:, :J].T, T + dlt[:, J]
        if float(((Ms.T @ dlt[:, :J].T).abs().max() + (dlt[:, J] / T0).abs().max())) < 1e-14:
            break
    return Ms.T @ x, T - T0


class _Scheme:
    """The time step of one domain on [nz, ny, nx] arrays."""

    def __init__(self, p, f, surrogate=None):
        self.p, self.dim, self.K = p, p["dim"], p["K"]
        self.shape = (p["nz"] if self.dim == 3 else 1, p["ny"], p["nx"])
        r = lambda v, k=1: None if v is None else v.double().reshape(k, *self.shape) if k > 1 else v.double().reshape(self.shape)  # noqa: E731
        self.phi0 = self.phi = r(f["phi"])
        self.T, self.Ts = r(f["T"]), r(f["Ts"])
        self.Y = list(f["Y"].double().reshape(self.K, *self.shape)) if self.K else []
        u = list(f["u"].double().reshape(self.dim, *self.shape))
        self.surrogate, self.pb, self.u_in, self.n = surrogate, 0.0, p["u_in"], 0
        v = [(a, b, c) for a in (0, 1, -1) for b in (0, 1, -1) for c in (0, 1, -1)
             if abs(a) + abs(b) + abs(c) <= 2 and (self.dim == 3 or c == 0)]
        w = {2: (4 / 9, 1 / 9, 1 / 36), 3: (1 / 3, 1 / 18, 1 / 36)}[self.dim]
        self.c, self.w = v, [w[sum(map(abs, x))] for x in v]
        self.opp = [v.index(tuple(-s for s in x)) for x in v]
        rho = self.rho(self.T, self.Y)
        uu = sum(a * a for a in u)
        self.g = []
        for c, w in zip(self.c, self.w):
            cu = sum(c[a] * u[a] for a in range(self.dim))
            self.g.append(w * rho * (cu + 1.5 * cu * cu - 0.5 * uu))

    def invM(self, Y):
        return sum(y / m for y, m in zip(Y, self.p["M"])) if self.K else 1.0 / self.p["M0"]

    def cp(self, Y):
        return sum(y * c for y, c in zip(Y, self.p["cp"])) if self.K else self.p["cp0"]

    def rho(self, T, Y):
        return self.p["P0"] / (R_GAS * T * self.invM(Y) * self.p["rho_ref"])

    def props(self, T, Y):
        """mu, lambda in lattice units, and the temperature factor of the diffusivities."""
        p = self.p
        s = p["dt"] / (p["rho_ref"] * p["dx"] ** 2)
        fD = (T / p["D_Tref"]) ** p["D_exp"] if p["D_exp"] else torch.ones_like(T)
        if p.get("transport") == "mixture":
            M = p["M"]
            iM = self.invM(Y)
            X = [y / m / iM for y, m in zip(Y, M)]
            mu = [m0 * (T / t) ** 1.5 * (t + q) / (T + q) for m0, t, q in
                  zip(p["mu_k"], p["suth_Tk"], p["suth_Sk"])]
            lam = [mu[k] * (1.32 * (p["cp"][k] - R_GAS / M[k]) + 1.77 * R_GAS / M[k])
                   for k in range(self.K)]
            mm = 0.0
            for k in range(self.K):
                den = 0.0
                for j in range(self.K):
                    a = 1.0 + (mu[k] / mu[j]).sqrt() * (M[j] / M[k]) ** 0.25
                    den = den + a * a / (math.sqrt(8.0) * math.sqrt(1.0 + M[k] / M[j])) * X[j]
                mm = mm + mu[k] * X[k] / den
            l = 0.5 * (sum(x * v for x, v in zip(X, lam)) + 1.0 / sum(x / v for x, v in zip(X, lam)))
            return mm * s, l * s, fD
        mu = torch.full_like(T, p["mu_ref"] * s)
        if p["sutherland"]:
            mu = mu * (T / p["suth_T"]) ** 1.5 * (p["suth_T"] + p["suth_S"]) / (T + p["suth_S"])
        return mu, mu * self.cp(Y) / p["Pr"], fD

    def near(self, F, a, s, ghost=None):
        """F at the neighbour x + s along axis a; `ghost` (default: the cell's own value) outside."""
        d = 2 - a
        R = torch.roll(F, -s, d)
        if self.p["bc"][2 * a] != "periodic":
            at = [slice(None)] * 3
            at[d] = -1 if s > 0 else 0
            R[tuple(at)] = F[tuple(at)] if ghost is None else ghost
        return R

    def neighbour(self, a, s):
        """(T, Y, phi, Ts) of the neighbour with the ghost rules."""
        p, face = self.p, 2 * a + (s > 0)
        kind = p["bc"][face]
        gT, gY = None, [None] * self.K
        if kind == "inlet":
            gT, gY = p["T_in"], list(p["Y_in"])
        elif kind == "wall" and p["wall_T"][face] > 0:
            gT = p["wall_T"][face]
        return (self.near(self.T, a, s, gT), [self.near(y, a, s, q) for y, q in zip(self.Y, gY)],
                self.near(self.phi, a, s), None if self.Ts is None else self.near(self.Ts, a, s))

    def inlet(self):
        p = self.p
        u = torch.full(self.shape[:2], self.u_in, dtype=torch.float64, device=self.T.device)
        if p["inlet_parabolic"] == 2:
            return u * (1.0 - self.phi[:, :, 0])
        if p["inlet_parabolic"]:
            for a, n in ((1, p["ny"]), (2, p["nz"])):
                if a < self.dim and p["bc"][2 * a] == "wall":
                    s = torch.arange(n, dtype=torch.float64, device=u.device) + 0.5
                    q = 4.0 * s * (n - s) / n ** 2
                    u = u * (q[None, :] if a == 1 else q[:, None])
        return u

    def pull(self, rho, uw):
        p, out = self.p, []
        rin = p["P0"] / (R_GAS * p["T_in"] * self.invM(p.get("Y_in", [])) * p["rho_ref"])
        ui = self.inlet() if p["bc"][0] == "inlet" else None
        for i, (c, w) in enumerate(zip(self.c, self.w)):
            own = self.g[self.opp[i]]
            G = torch.roll(self.g[i], (c[2], c[1], c[0]), (0, 1, 2))
            if c[0] == -1 and p["bc"][1] == "outlet":
                cu, uu = sum(c[a] * uw[a] for a in range(self.dim)), sum(q * q for q in uw)
                G[:, :, -1] = (-own + w * (2 * self.pb + rho * (3 * cu * cu - uu)))[:, :, -1]
            if c[0] == 1 and p["bc"][0] == "inlet":
                G[:, :, 0] = own[:, :, 0] + 2 * w * rin * ui
            for a in (2, 1, 0):
                face = 2 * a + (c[a] < 0)
                if a < self.dim and c[a] and p["bc"][face] == "wall":
                    at = [slice(None)] * 3
                    at[2 - a] = 0 if c[a] > 0 else -1
                    cw = sum(c[b] * p["wall_u"][face][b] for b in range(self.dim))
                    G[tuple(at)] = (own + 2 * w * rho * cw)[tuple(at)]
            out.append(G)
        return out

    def rates(self, rho):
        """Chemistry source per lattice step: omega_k / rho_ref and omega_T / rho_ref."""
        p = self.p
        if p["chem"] == "none" or not self.K:
            return [torch.zeros_like(rho)] * self.K, torch.zeros_like(rho)
        if p["chem"] == "explicit":
            C = [rho * p["rho_ref"] * y.clamp_min(0) / m for y, m in zip(self.Y, p["M"])]
            om = [torch.zeros_like(rho)] * self.K
            for r in p["reactions"]:
                q = r["A"] * torch.exp(-r["EaR"] / self.T) * self.T ** r.get("b", 0.0)
                for k in range(self.K):
                    if r["order"][k]:
                        q = q * C[k] ** r["order"][k]
                om = [o + m * s * q * p["dt"] / p["rho_ref"] for o, m, s in
                      zip(om, p["M"], r["stoich"])]
            return om, -sum(h * o for h, o in zip(p["hf"], om))
        T, Y = self.T.reshape(-1), torch.stack([y.reshape(-1) for y in self.Y])
        r1 = rho.reshape(-1)
        if p["chem"] == "surrogate":
            dY, dT = self.surrogate(p, T, Y, r1 * p["rho_ref"])
        else:
            dY, dT = _backward_euler(p, T, Y, r1 * p["rho_ref"])
        cp = self.cp(list(Y))
        return [(r1 * d).reshape(rho.shape) for d in dY], (r1 * cp * dT).reshape(rho.shape)

    def move(self):
        p = self.p
        us = p.get("u_s")
        if not us:
            return
        phi = self.phi0
        for a in range(self.dim):
            s = self.n * us[a]
            k, f = math.floor(s), s - math.floor(s)
            n, d = phi.shape[2 - a], 2 - a
            i = torch.arange(n, device=phi.device) - k
            wrap = (lambda j: j % n) if p["bc"][2 * a] == "periodic" else (lambda j: j.clamp(0, n - 1))
            phi = (1 - f) * phi.index_select(d, wrap(i)) + f * phi.index_select(d, wrap(i - 1))
        self.phi = phi

    def moments(self):
        """Pulled populations, velocity and properties of the current state."""
        p = self.p
        rho = self.rho(self.T, self.Y)
        mu, lam, fD = self.props(self.T, self.Y)
        Kd = p["A_u"] * mu * (1 - self.phi) * self.phi ** 2 / p["eta"] ** 2
        us = p.get("u_s") or [0.0] * 3
        uw = [torch.zeros_like(rho)] * self.dim
        g = self.pull(rho, uw)
        speed = lambda g: [(3 * sum(c[a] * q for c, q in zip(self.c, g))  # noqa: E731
                            + 0.5 * (p["Fb"][a] + Kd * us[a])) / (rho + 0.5 * Kd)
                           for a in range(self.dim)]
        u = speed(g)
        if p["bc"][1] == "outlet":  # the outlet column again, with its own first velocity
            g = [torch.cat([x[:, :, :-1], y[:, :, -1:]], 2) for x, y in zip(g, self.pull(rho, u))]
            u = speed(g)
        return g, u, rho, mu, lam, fD, Kd, us

    def step(self):
        p, K = self.p, self.K
        g, u, rho, mu, lam, fD, Kd, us = self.moments()
        phi, T, Y = self.phi, self.T, self.Y
        ff = 1 - phi
        on = ff >= p["phi_min"]
        ffs = torch.where(on, ff, torch.ones_like(ff))
        iM, cp = self.invM(Y), self.cp(Y)
        SI = p["A_T"] / p["eta"] ** 2 * lam * ff * phi ** 2 * ((self.Ts if self.Ts is not None else p["Ts_uniform"]) - T)
        SI = torch.where(on & ((phi >= p["phi_min"]) if self.Ts is not None else on), SI, torch.zeros_like(T))
        om, omT = self.rates(rho)
        h2 = p["dt"] / p["dx"] ** 2
        rf = ff * rho * fD
        nb = [[self.neighbour(a, s) for s in (-1, 1)] for a in range(self.dim)]
        pr = [[(self.rho(t, y), *self.props(t, y)[1:], 1 - f) for t, y, f, _ in q] for q in nb]
        Yn, sYm = [], 0.0
        for k in range(K):
            adv, dif, cen = 0.0, 0.0, 0.0
            for a in range(self.dim):
                ym, yp = nb[a][0][1][k], nb[a][1][1][k]
                fm, fp = (0.5 * (rf + q[3] * q[0] * q[2]) for q in pr[a])
                adv = adv + u[a] * torch.where(u[a] > 0, Y[k] - ym, yp - Y[k])
                dif = dif + fp * (yp - Y[k]) - fm * (Y[k] - ym)
                cen = cen + u[a] * 0.5 * (yp - ym)
            d = (-ff * rho * adv + p["Dref"][k] * h2 * dif + ff * om[k]) / (ffs * rho)
            d = torch.where(on, d, torch.zeros_like(d))
            Yn.append(Y[k] + d)
            sYm = sYm + torch.where(on, d + cen, torch.zeros_like(d)) / p["M"][k]
        adv, dif, cen, cross = 0.0, 0.0, 0.0, 0.0
        for a in range(self.dim):
            tm, tp = nb[a][0][0], nb[a][1][0]
            km, kp = (0.5 * (ff * lam + q[3] * q[1]) for q in pr[a])
            adv = adv + u[a] * torch.where(u[a] > 0, T - tm, tp - T)
            dif = dif + kp * (tp - T) - km * (T - tm)
            cen = cen + u[a] * 0.5 * (tp - tm)
            for k in range(K):
                cross = cross + p["cp"][k] * p["Dref"][k] * h2 * fD * 0.25 * \
                    (nb[a][1][1][k] - nb[a][0][1][k]) * (tp - tm)
        dT = (-ff * rho * cp * adv + dif + ff * (rho * cross + omT + SI)) / (ffs * rho * cp)
        Tsv = self.Ts if self.Ts is not None else torch.full_like(T, p["Ts_uniform"])
        Tn = torch.where(on, T + dT, Tsv)
        D = torch.where(on, dT + cen, Tsv - T) / T + (sYm / iM if K else 0.0)
        Tsn = self.Ts
        if self.Ts is not None:
            L = p["lambda_s"] * h2 / p["rho_ref"]
            dif, ads = 0.0, 0.0
            for a in range(self.dim):
                (_, _, fm, sm), (_, _, fp, sp) = nb[a]
                dif = dif + L * (0.5 * (phi + fp) * (sp - self.Ts) - 0.5 * (phi + fm) * (self.Ts - sm))
                ads = ads + us[a] * ((self.Ts - sm) if us[a] > 0 else (sp - self.Ts))
            sol = phi >= p["phi_min"]
            ph = torch.where(sol, phi, torch.ones_like(phi))
            Tsn = torch.where(sol, self.Ts + (dif - ff * SI) / (ph * p["rhocp_s"] / p["rho_ref"]) - ads, self.Ts)
        G = [(q[1][0] - q[0][0]) / 6.0 for q in pr]
        F = [p["Fb"][a] - Kd * (u[a] - us[a]) for a in range(self.dim)]
        Ph = sum(g) + 0.5 * (rho / 3 * D + sum(a * b for a, b in zip(u, G)))
        omega = 2 * rho / (rho + 6 * mu)
        uu = sum(a * a for a in u)
        new = []
        for c, w, gi in zip(self.c, self.w, g):
            cu = sum(c[a] * u[a] for a in range(self.dim))
            e = 3 * cu + 4.5 * cu * cu - 1.5 * uu
            xi = w * (sum((c[a] - u[a]) * (G[a] * e + F[a] * (1 + e)) for a in range(self.dim)) + rho * D / 3)
            new.append(gi - omega * (gi - w * (Ph + rho * e / 3)) + (1 - 0.5 * omega) * xi)
        if p.get("outlet") == "nscbc":
            cs = math.sqrt(1 / 3)
            m = lambda v, i: float(v[:, :, i].mean())  # noqa: E731
            L5 = (m(u[0], -1) + cs) * (m(Ph, -1) - m(Ph, -2) + m(rho, -1) * cs * (m(u[0], -1) - m(u[0], -2)))
            self.pb -= 0.5 * (L5 + p.get("nscbc_sigma", 0.25) * cs / p["nx"] * self.pb)
        if p.get("inlet_feedback") is not None:
            k = int(p["inlet_feedback"])
            fuel = float((ff * -om[k])[on].sum())
            self.u_in = 1.0
            area = float(self.inlet().sum())
            rin = 1.0 / (R_GAS * p["T_in"] * self.invM(p["Y_in"]) * p["rho_ref"])
            self.u_in = min(0.3, max(0.0, fuel / (rin * p["P0"] * p["Y_in"][k] * area)))
        self.g, self.T, self.Y, self.Ts = new, Tn, Yn, Tsn
        self.n += 1
        self.move()

    def outputs(self):
        u = self.moments()[1]
        out = {"T": self.T.reshape(-1)}
        if self.K:
            out["Y"] = torch.stack(self.Y).reshape(-1)
        if self.Ts is not None:
            out["Ts"] = self.Ts.reshape(-1)
        out["u"] = torch.stack(u).reshape(-1)
        return out


def _network(theta, x):
    hs, off = [x], 0
    for a, b in ((8, 64), (64, 64), (64, 64), (64, 6)):
        z = hs[-1] @ theta[off:off + a * b].reshape(a, b) + theta[off + a * b:off + a * b + b]
        hs.append(torch.tanh(z) if b == 64 else z)
        off += a * b + b
    return hs


def _surrogate_chemistry(theta, rec):
    """The learned increments with their acceptance test, projection and implicit fallback."""
    def chem(p, T, Y, rho):
        kw = {"dtype": torch.float64, "device": T.device}
        th = torch.tensor(theta, **kw)
        v = lambda a, n: torch.tensor([a[i] for i in range(n)], **kw)  # noqa: E731
        X = torch.cat([T[:, None], Y.T, torch.full_like(T, p["P0"])[:, None]], 1)
        istd = torch.where(v(rec.x_std, 8) > 0, 1.0 / v(rec.x_std, 8).clamp_min(1e-300), torch.zeros(8, **kw))
        o = _network(th, (X - v(rec.x_mean, 8)) * istd)[-1]
        dY = torch.exp(-rec.theta_s / T)[:, None] * (o * v(rec.y_std, 6) + v(rec.y_mean, 6))
        ok = ((X >= v(rec.lo, 8)) & (X <= v(rec.hi, 8))).all(1)
        M = torch.tensor(p["M"], **kw)
        B = torch.stack([v(rec.elem[e], 6) for e in range(rec.n_elem)]) / M
        ok = ok & ((dY @ (B * v(rec.elem_mass, rec.n_elem)[:, None]).T).abs() <= rec.tol).all(1)
        dY = dY - dY @ B.T @ torch.linalg.inv(B @ B.T) @ B
        cp, hf = torch.tensor(p["cp"], **kw), torch.tensor(p["hf"], **kw)
        dT = -(dY @ hf) / ((Y.T + dY) @ cp)
        if not bool(ok.all()):
            bad = ~ok
            bY, bT = _backward_euler(p, T[bad], Y[:, bad], rho[bad])
            dY[bad], dT[bad] = bY.T, bT
        return dY.T, dT
    return chem


def exact(case, seed):
    if case["kind"] == "train":
        X, Yt, theta = _train_inputs(case, seed)
        th = torch.tensor(theta, dtype=torch.float64, device=DEV)
        m, v = torch.zeros_like(th), torch.zeros_like(th)
        nb = -(-case["rows"] // case["batch"])
        for s in range(case["steps"]):
            r0 = (s % nb) * case["batch"]
            x, y = X[r0:r0 + case["batch"]].double(), Yt[r0:r0 + case["batch"]].double()
            th = th.detach().requires_grad_(True)
            loss = ((_network(th, x)[-1] - y) ** 2).mean()
            g, = torch.autograd.grad(loss, th)
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            th = th.detach() - 1e-3 * (m / (1 - 0.9 ** (s + 1))) / ((v / (1 - 0.999 ** (s + 1))).sqrt() + 1e-8)
        return {"loss": float(loss), "theta": th}
    if case["kind"] == "batch":
        outs = []
        for i, p in enumerate(_batch_problems(case)):
            s = _Scheme(p, _fields(p, seed + 1000 * i, bed=p["bed"]))
            for _ in range(case["steps"]):
                s.step()
            outs.append(s.outputs())
        return {k: torch.cat([o[k] for o in outs]) for k in ("T", "u")}
    p = _problem(case)
    p["precision"] = case["precision"]
    chem = _surrogate_chemistry(*_surrogate_net(p, seed)) if case["kind"] == "surrogate" else None
    s = _Scheme(p, _fields(p, seed), chem)
    for _ in range(case["steps"]):
        s.step()
    return s.outputs()
