"""The work a user of this package has it do, as timed cases.

Every case goes through the public entry points of ``paper_1907_12334_gb300.msg``
on the current CUDA stream.  A case is a plain dict with a ``kind``:

  solve    one ``msg_solve_batch`` call on a batch of sampled fields (Algorithm 2
           on every grid of every sample), with its workspace and outputs kept;
  step     one estimator step: normals, KL fields, solve, multi-index differences;
  field    one ``sample_field`` call on a prepared KL basis;
  ce       one ``ce_sample_field`` call (circulant embedding);
  history  one ``msg_cycle_history`` call (the convergence study);
  normals  one ``msg_normals`` call.

Fields follow the package's Matern law (nu = 3/2, unit variance, correlation
length 0.2 along x) at aspect ratio 1/4, inside the range of the paper's
anisotropic ratio, as a truncated expansion in the cosine basis of the unit
square: lambda is the law's spectral density at the basis wavenumbers, scaled so
that the whole expansion has unit variance, and the M largest terms are kept.
Every sample of such a batch converges, so a pass times the solver and not the
cycle cap of one stray sample.
"""
import math
import random

import numpy as np
import torch

from paper_1907_12334_gb300 import inputs, msg

DEV = "cuda:0"


# --------------------------------------------------------------------- cases --

def listed():
    return [
        # the benchmark's solve at its grid size and settings, a batch of a served or memory-bound run
        dict(name="solve_256_mixed", kind="solve", shapes="same", P=8, Q=8, S=192, M=400, precision="mixed",
             qoi="integral", eps=1e-10),
        # the index set of an adaptive run in one call: every shape 4..128 cells a side, shuffled
        dict(name="solve_uneven_mixed", kind="solve", shapes="uneven", P=7, Q=7, S=180, M=64, precision="mixed",
             qoi="integral", eps=1e-10),
        # FP64 cycles, with the solutions of every grid read back (a user who wants u, not only Q)
        dict(name="solve_32_fp64_u", kind="solve", shapes="same", P=5, Q=5, S=64, M=64, precision="fp64",
             qoi="point", eps=1e-10, with_u=True),
        # one request of a served run: a few samples of one mid-size index, where latency counts
        dict(name="solve_serving_64x32", kind="solve", shapes="same", P=6, Q=5, S=6, M=64, precision="mixed",
             qoi="flux", eps=1e-8),
        # the first requests of a served run: the smallest grids, a handful of samples
        dict(name="solve_small_8x4", kind="solve", shapes="same", P=3, Q=2, S=4, M=64, precision="mixed",
             qoi="integral", eps=1e-10),
        # one estimator step over the index set 0..3 x 0..3 on base grid (3,3), finest 64 x 64
        dict(name="step_indices_64", kind="step", p0=3, q0=3, amax=3, S=256, M=64, eps=1e-10),
        # the KL contraction of a step of the benchmark: FP32 products, FP64 fields of 513 x 513 nodes
        dict(name="field_fp32_513", kind="field", mode="FP32", nx=513, ny=513, M=400, S=512, z="f64"),
        # the KL contraction on tensor cores at 1024 x 1024 points, FP32 fields
        dict(name="field_bf16x3_1024", kind="field", mode="BF16X3", nx=1024, ny=1024, M=400, S=1024, z="f32"),
        # ragged sizes on tensor cores, FP64 fields ready for the solver
        dict(name="field_tf32_257x129", kind="field", mode="TF32", nx=257, ny=129, M=300, S=777, z="f64"),
        # the served run's own fields: FP64 products, few samples of one index
        dict(name="field_fp64_129x65", kind="field", mode="FP64", nx=129, ny=65, M=64, S=24, z="f64"),
        # the paper's own field law at the benchmark's field size
        dict(name="ce_513", kind="ce", P=8, Q=8, L=9, S=8, batch=8, nu=0.5, scale=0),
        # the convergence study: MSG W(2,2) cycles from u = 0 on 64 x 64 cells
        dict(name="history_msg_64", kind="history", method="msg", P=6, Q=6, S=32, nu=2, cycles=12),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "step", "field", "field", "ce", "history", "normals"])
    if kind == "solve":
        P, Q = rng.randint(2, 8), rng.randint(2, 8)
        precision = "fp64" if P + Q <= 10 and rng.random() < 0.25 else "mixed"
        most = (64 << 20) / (P * Q << (P + Q)) * (0.02 if precision == "fp64" else 1.0)
        return dict(kind="solve", shapes="uneven" if max(P, Q) <= 6 and rng.random() < 0.3 else "same", P=P, Q=Q,
                    S=_logint(rng, 1, max(2, min(256, most))), M=rng.randint(20, 400), precision=precision,
                    qoi=rng.choice(["integral", "point", "flux"]), eps=rng.choice([1e-8, 1e-10]))
    if kind == "step":
        p0, q0 = rng.randint(2, 3), rng.randint(2, 3)
        return dict(kind="step", p0=p0, q0=q0, amax=rng.randint(1, 3), S=_logint(rng, 16, 400),
                    M=rng.randint(20, 200), eps=1e-10)
    if kind == "field":
        mode = rng.choice(["FP32", "BF16X3", "TF32", "FP64"])
        big = {"FP32": 513, "BF16X3": 1024, "TF32": 1024, "FP64": 129}[mode]
        nx, ny, M, S = _logint(rng, 9, big), _logint(rng, 9, big), _logint(rng, 20, 400), _logint(rng, 8, 1024)
        if mode == "FP32":
            S = min(S, 512)
        if mode == "FP64":
            S = min(S, 256)
        return dict(kind="field", mode=mode, nx=nx, ny=ny, M=M, S=S, z=rng.choice(["f32", "f64"]))
    if kind == "ce":
        P, Q = rng.randint(2, 8), rng.randint(2, 8)
        batch = rng.randint(1, 8)
        return dict(kind="ce", P=P, Q=Q, L=rng.choice([5, 7, 9]), S=rng.randint(batch, 8), batch=batch,
                    nu=rng.choice([0.5, 1.5, 2.5]), scale=rng.randint(0, 1))
    if kind == "history":
        P = rng.randint(3, 6)
        return dict(kind="history", method=rng.choice(["msg", "standard"]), P=P, Q=rng.randint(3, P),
                    S=rng.randint(4, 32), nu=rng.randint(2, 4), cycles=rng.randint(5, 12))
    return dict(kind="normals", S=_logint(rng, 64, 8192), M=rng.randint(20, 400))


# -------------------------------------------------------------------- inputs --

def _terms(M):
    """Wavenumbers (k, l) and sqrt(lambda) of the M largest terms of the cosine expansion."""
    law = inputs.FieldLaw(ell_y=0.05)
    k, l = np.meshgrid(np.arange(60), np.arange(400))
    # Matern nu = 3/2 in two dimensions: spectral density ~ (4 nu + |T^-1 w|^2)^-(nu + 1), w = pi (k, l)
    dens = (4 * law.nu + (math.pi * k * law.ell_x) ** 2 + (math.pi * l * law.ell_y) ** 2) ** -(law.nu + 1.0)
    order = np.argsort(-dens.ravel(), kind="stable")[:M]
    lam = dens.ravel()[order]
    return k.ravel()[order], l.ravel()[order], np.sqrt(lam / dens.sum())


def _cosines(n, wave):
    """Normalised cosines [n][len(wave)] at the nodes i / (n - 1)."""
    x = torch.arange(n, dtype=torch.float64, device=DEV) / (n - 1)
    w = torch.as_tensor(wave, dtype=torch.float64, device=DEV)
    return torch.cos(math.pi * x[:, None] * w[None, :]) * torch.where(w > 0, math.sqrt(2.0), 1.0)


def _basis(nx, ny, M):
    """(Phi [ny * nx][M], sqrt(lambda) [M]) on an nx x ny node grid, x fastest."""
    k, l, sl = _terms(M)
    cx, cy = _cosines(nx, k), _cosines(ny, l)
    return (cy[:, None, :] * cx[None, :, :]).reshape(ny * nx, M), torch.as_tensor(sl, device=DEV)


def _fields(shapes, M, gen):
    """Packed fields of a batch, one draw of the M coefficients per sample."""
    k, l, sl = _terms(M)
    xi = torch.randn(len(shapes), M, dtype=torch.float64, device=DEV, generator=gen) * torch.as_tensor(sl, device=DEV)
    kd, ld = torch.as_tensor(k, device=DEV), torch.as_tensor(l, device=DEV)
    coef = torch.zeros(len(shapes), int(l.max()) + 1, int(k.max()) + 1, dtype=torch.float64, device=DEV)
    coef[:, ld, kd] = xi
    parts = {}
    for shape in sorted(set(shapes)):
        at = [i for i, s in enumerate(shapes) if s == shape]
        cx = _cosines((2 << shape[0]) + 1, np.arange(coef.shape[2]))
        cy = _cosines((2 << shape[1]) + 1, np.arange(coef.shape[1]))
        z = torch.matmul(torch.matmul(cy, coef[at]), cx.T).reshape(len(at), -1)
        parts.update(zip(at, z))
    return torch.cat([parts[i] for i in range(len(shapes))])


def _shapes(c):
    if c["kind"] == "step":
        idx = [(a, b) for a in range(c["amax"] + 1) for b in range(c["amax"] + 1)]
        return [(c["p0"] + idx[i % len(idx)][0], c["q0"] + idx[i % len(idx)][1]) for i in range(c["S"])]
    if c["shapes"] == "same":
        return [(c["P"], c["Q"])] * c["S"]
    idx = [(p, q) for p in range(2, c["P"] + 1) for q in range(2, c["Q"] + 1)]
    shapes = [idx[i % len(idx)] for i in range(c["S"])]
    random.Random(17).shuffle(shapes)
    return shapes


def _params(c):
    precision = msg.MSG_PREC_FP64 if c.get("precision") == "fp64" else msg.MSG_PREC_MIXED
    qoi = {"integral": msg.MSG_QOI_INTEGRAL, "point": msg.MSG_QOI_POINT, "flux": msg.MSG_QOI_FLUX}
    return msg.SolverParams(eps=c["eps"], max_cycles=400, precision=precision, qoi=qoi[c.get("qoi", "integral")])


def _solver_state(s, c, shapes):
    s["PQ"] = np.array(shapes, dtype=np.int32)
    s["prm"] = _params(c)
    nq, _ = msg.packed_sizes(s["PQ"])
    s["Q"] = torch.empty(nq, dtype=torch.float64, device=DEV)
    s["status"] = torch.empty(len(shapes), dtype=torch.int32, device=DEV)
    s["ws"] = torch.empty(msg.msg_workspace_bytes(s["PQ"], s["prm"]), dtype=torch.uint8, device=DEV)


def prepare(case, seed):
    c, s = case, {"case": case, "seed": seed}
    gen = torch.Generator(device=DEV).manual_seed(seed)
    if c["kind"] == "solve":
        shapes = _shapes(c)
        _solver_state(s, c, shapes)
        s["Z"] = _fields(shapes, c["M"], gen)
        if c.get("with_u"):
            s["u"] = torch.empty(msg.msg_solution_values(s["PQ"]), dtype=torch.float64, device=DEV)
    elif c["kind"] == "step":
        shapes = _shapes(c)
        _solver_state(s, c, shapes)
        p0, q0 = c["p0"], c["q0"]
        s["L"] = s["PQ"] - np.array([p0, q0], dtype=np.int32)
        s["Z"] = torch.empty(sum(msg.field_points(P, Q) for P, Q in shapes), dtype=torch.float64, device=DEV)
        s["dQ"] = torch.empty(int(((s["L"] + 1).prod(axis=1)).sum()), dtype=torch.float64, device=DEV)
        s["Y"] = torch.empty(c["S"], dtype=torch.float64, device=DEV)
        r = 1.733  # the initial index law of the adaptive driver: P(L_j >= k) = exp(-r k)
        a = np.arange(c["amax"] + 1)
        s["ptau"] = np.exp(-r * (a[:, None] + a[None, :]))
        off = np.concatenate([[0], np.cumsum([msg.field_points(P, Q) for P, Q in shapes])])
        s["groups"] = []
        for shape in sorted(set(shapes)):
            at = [i for i, x in enumerate(shapes) if x == shape]
            Phi, sl = _basis((2 << shape[0]) + 1, (2 << shape[1]) + 1, c["M"])
            prep = torch.empty(msg.kl_prepared_bytes(Phi.shape[0], c["M"], msg.MSG_GEMM_FP64), dtype=torch.uint8,
                               device=DEV)
            msg.kl_prepare(Phi, sl, msg.MSG_GEMM_FP64, prep)
            where = torch.as_tensor(np.concatenate([np.arange(off[i], off[i + 1]) for i in at]), device=DEV)
            s["groups"].append((prep, Phi.shape[0], torch.as_tensor(at, device=DEV), where))
        s["xi"] = torch.empty(c["S"], c["M"], dtype=torch.float64, device=DEV)
    elif c["kind"] == "field":
        mode = getattr(msg, "MSG_GEMM_" + c["mode"])
        Phi, sl = _basis(c["nx"], c["ny"], c["M"])
        s["prep"] = torch.empty(msg.kl_prepared_bytes(Phi.shape[0], c["M"], mode), dtype=torch.uint8, device=DEV)
        msg.kl_prepare(Phi, sl, mode, s["prep"])
        s["xi"] = torch.randn(c["S"], c["M"], dtype=torch.float64, device=DEV, generator=gen)
        s["Z"] = torch.empty(c["S"], Phi.shape[0], dtype=torch.float32 if c["z"] == "f32" else torch.float64, device=DEV)
        s["mode"] = mode
    elif c["kind"] == "ce":
        s["law"] = msg.CeLaw(L=c["L"], batch=c["batch"], nu=c["nu"], scale=c["scale"])
        s["Z"] = torch.empty(c["S"], msg.field_points(c["P"], c["Q"]), dtype=torch.float64, device=DEV)
        s["eta_theta"] = torch.empty(c["S"], 2, dtype=torch.float64, device=DEV)
        s["status"] = torch.empty(c["S"], dtype=torch.int32, device=DEV)
        s["ws"] = torch.empty(msg.ce_workspace_bytes(c["P"], c["Q"], s["law"]), dtype=torch.uint8, device=DEV)
    elif c["kind"] == "history":
        s["prm"] = msg.SolverParams(nu1=c["nu"], nu2=c["nu"])
        s["method"] = msg.MSG_HIST_MSG if c["method"] == "msg" else msg.MSG_HIST_STANDARD
        s["Z"] = _fields([(c["P"], c["Q"])] * c["S"], 200, gen)
        s["hist"] = torch.empty(c["S"], c["cycles"] + 1, dtype=torch.float64, device=DEV)
        s["ws"] = torch.empty(msg.msg_history_workspace_bytes(c["P"], c["Q"], c["S"], s["prm"], s["method"]),
                              dtype=torch.uint8, device=DEV)
    else:
        s["xi"] = torch.empty(c["S"], c["M"], dtype=torch.float64, device=DEV)
    return s


# ----------------------------------------------------------------------- run --

def run(s):
    c = s["case"]
    if c["kind"] == "solve":
        msg.msg_solve_batch(s["PQ"], s["prm"], s["Z"], s["Q"], s["status"], workspace=s["ws"])
        out = {"Q": s["Q"], "status": s["status"]}
        if "u" in s:
            msg.msg_solution(s["PQ"], s["prm"], s["ws"], s["u"])
            out["u"] = s["u"]
        return out
    if c["kind"] == "step":
        msg.msg_normals(s["seed"], 0, c["S"], c["M"], s["xi"])
        for prep, npts, at, where in s["groups"]:
            Zg = torch.empty(at.numel(), npts, dtype=torch.float64, device=DEV)
            msg.sample_field(prep, npts, c["M"], msg.MSG_GEMM_FP64, s["xi"][at], Zg)
            s["Z"][where] = Zg.reshape(-1)
        msg.msg_solve_batch(s["PQ"], s["prm"], s["Z"], s["Q"], s["status"], workspace=s["ws"])
        msg.mimc_differences(s["L"], c["p0"], c["q0"], s["Q"], s["dQ"], ptau=s["ptau"], Y=s["Y"])
        return {"Z": s["Z"], "Q": s["Q"], "status": s["status"], "dQ": s["dQ"], "Y": s["Y"]}
    if c["kind"] == "field":
        msg.sample_field(s["prep"], c["nx"] * c["ny"], c["M"], s["mode"], s["xi"], s["Z"])
        return s["Z"]
    if c["kind"] == "ce":
        msg.ce_sample_field(c["P"], c["Q"], c["S"], s["law"], s["seed"], 0, s["Z"], s["eta_theta"], s["status"], s["ws"])
        return {"Z": s["Z"], "eta_theta": s["eta_theta"], "status": s["status"]}
    if c["kind"] == "history":
        return msg.msg_cycle_history(c["P"], c["Q"], c["S"], s["prm"], s["method"], s["Z"], c["cycles"], s["hist"],
                                     s["ws"])
    msg.msg_normals(s["seed"], 0, c["S"], c["M"], s["xi"])
    return s["xi"]


# ---------------------------------------------------------------------- work --

def _solve_flops(shapes):
    # eight cycles a grid; one W-cycle of grid (p, q) visits each of its p q grids with 2^(p+q) nodes in
    # all; a visit is four sweeps of 10 flops, a residual of 10 and 25 for the transfers
    return sum(8.0 * 75.0 * p * q * 2.0 ** (p + q) for P, Q in shapes for p in range(1, P + 1) for q in range(1, Q + 1))


def work(case):
    c = case
    if c["kind"] in ("solve", "step"):
        shapes = _shapes(c)
        nf = sum(msg.field_points(P, Q) for P, Q in shapes)
        nq = sum(P * Q for P, Q in shapes)
        b, f = 8.0 * nf + 8.0 * nq + 4.0 * len(shapes), _solve_flops(shapes)
        if c.get("with_u"):
            b += 8.0 * sum(((2 << P) - 2 + P) * ((2 << Q) - 2 + Q) for P, Q in shapes)
        if c["kind"] == "step":
            b += 8.0 * sum((P - c["p0"] + 1) * (Q - c["q0"] + 1) for P, Q in shapes)
            b += 8.0 * c["M"] * sum(msg.field_points(P, Q) for P, Q in sorted(set(shapes)))
            f += 2.0 * nf * c["M"]
        return {"bytes": b, "flops": f}
    if c["kind"] == "field":
        npts, pe = c["nx"] * c["ny"], 8.0 if c["mode"] == "FP64" else 4.0
        return {"bytes": pe * npts * c["M"] + 8.0 * c["S"] * c["M"] + (4.0 if c["z"] == "f32" else 8.0) * c["S"] * npts,
                "flops": 2.0 * npts * c["M"] * c["S"]}
    if c["kind"] == "ce":
        n = (c["L"] << (c["P"] + 1)) * (c["L"] << (c["Q"] + 1))
        # per sample a real and a complex transform of n points, the covariance and the normals
        return {"bytes": 8.0 * c["S"] * msg.field_points(c["P"], c["Q"]), "flops": c["S"] * n * (7.5 * math.log2(n) + 50.0)}
    if c["kind"] == "history":
        per = c["P"] * c["Q"] * 2.0 ** (c["P"] + c["Q"]) if c["method"] == "msg" else 4.0 * 2.0 ** (c["P"] + c["Q"])
        return {"bytes": 8.0 * c["S"] * (msg.field_points(c["P"], c["Q"]) + c["cycles"] + 1),
                "flops": c["S"] * c["cycles"] * per * (35.0 + 20.0 * c["nu"])}
    return {"bytes": 8.0 * c["S"] * c["M"], "flops": 30.0 * c["S"] * c["M"]}


# --------------------------------------------------------------------- exact --

def _normals(seed, sample, n):
    """Normals 0..n-1 of one sample's stream: numpy's Philox, the counter's second word the sample."""
    bits = np.random.Philox(key=seed, counter=((sample << 64) - 1) % (1 << 256))
    u = (bits.random_raw(-(-n // 4) * 4) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
    u = torch.as_tensor(u, device=DEV).reshape(-1, 2)
    rad, ang = torch.sqrt(-2.0 * torch.log1p(-u[:, 0])), 2.0 * math.pi * u[:, 1]
    return torch.stack([rad * torch.cos(ang), rad * torch.sin(ang)], dim=1).reshape(-1)[:n]


def _faces(Z, P, Q, p, q):
    """a / dx^2 at the x-faces [S][2^q - 1][2^p] and a / dy^2 at the y-faces [S][2^q][2^p - 1] of grid (p, q):
    series means of exp(Z) over the finest faces a face covers."""
    sx, sy = 1 << (P - p), 1 << (Q - q)
    ex = torch.exp(-Z[:, 2 * sy:-1:2 * sy, 1::2])
    ey = torch.exp(-Z[:, 1::2, 2 * sx:-1:2 * sx])
    ax = 4.0 ** p * sx / ex.reshape(Z.shape[0], (1 << q) - 1, 1 << p, sx).sum(-1)
    ay = 4.0 ** q * sy / ey.reshape(Z.shape[0], 1 << q, sy, (1 << p) - 1).sum(2)
    return ax, ay


def _direct(Z, P, Q, p, q):
    """u [S][2^q + 1][2^p + 1] of -div(a grad u) = 1 on grid (p, q) by block elimination along the longer side."""
    ax, ay = _faces(Z, P, Q, p, q)
    flip = p > q
    if flip:  # rows become the longer direction
        ax, ay = ay.transpose(1, 2), ax.transpose(1, 2)
    S, n, m = Z.shape[0], ay.shape[1] - 1, ay.shape[2]
    diag = ax[:, :, :-1] + ax[:, :, 1:] + ay[:, :-1, :] + ay[:, 1:, :]
    inv, ys, eye = [], [], torch.eye(m, dtype=torch.float64, device=DEV).expand(S, m, m)
    for j in range(n):
        T = torch.diag_embed(diag[:, j])
        if m > 1:
            off = -ax[:, j, 1:-1]
            T = T + torch.diag_embed(off, 1) + torch.diag_embed(off, -1)
        y = torch.ones(S, m, 1, dtype=torch.float64, device=DEV)
        if j:
            cpl = ay[:, j, :, None]
            T = T - cpl * inv[-1] * cpl.transpose(1, 2)
            y = y + cpl * (inv[-1] @ ys[-1])
        inv.append(torch.cholesky_solve(eye, torch.linalg.cholesky(T)))
        ys.append(y)
    u = torch.zeros(S, n + 2, m + 2, dtype=torch.float64, device=DEV)
    x = torch.zeros(S, m, 1, dtype=torch.float64, device=DEV)
    for j in range(n - 1, -1, -1):
        x = inv[j] @ (ys[j] + ay[:, j + 1, :, None] * x)
        u[:, j + 1, 1:-1] = x[:, :, 0]
    return u.transpose(1, 2) if flip else u


def _exact_solve(c, shapes, Z):
    """Q packed as msg_solve_batch writes it, and (same-shape batches) u as msg_solution does."""
    qoff = np.concatenate([[0], np.cumsum([P * Q for P, Q in shapes])])
    zoff = np.concatenate([[0], np.cumsum([msg.field_points(P, Q) for P, Q in shapes])])
    Qout, us = torch.empty(int(qoff[-1]), dtype=torch.float64, device=DEV), []
    for shape in sorted(set(shapes)):
        P, Q = shape
        at = [i for i, s in enumerate(shapes) if s == shape]
        Zs = torch.stack([Z[zoff[i]:zoff[i + 1]] for i in at]).reshape(len(at), (2 << Q) + 1, (2 << P) + 1)
        for p in range(1, P + 1):
            for q in range(1, Q + 1):
                u = _direct(Zs, P, Q, p, q)
                us.append(u.reshape(len(at), -1))
                if c.get("qoi", "integral") == "integral":
                    v = u.sum((1, 2)) / 2.0 ** (p + q)
                elif c["qoi"] == "point":
                    v = u[:, 1 << (q - 1), 1 << (p - 1)]
                else:
                    a = torch.exp(Zs[:, 2 << (Q - q):-1:2 << (Q - q), -1])
                    v = (a * u[:, 1:-1, -2]).sum(1) * 2.0 ** (p - q)
                Qout[torch.as_tensor(qoff[at] + (p - 1) * Q + q - 1, device=DEV)] = v
    return Qout, torch.cat(us, dim=1).reshape(-1) if c.get("with_u") else None


def _exact_ce(c, seed):
    law = msg.CeLaw()
    M1, M2 = c["L"] << (c["P"] + 1), c["L"] << (c["Q"] + 1)
    n1, n2 = (2 << c["P"]) + 1, (2 << c["Q"]) + 1
    Zs, ets = [], []
    for s in range(c["S"]):
        raw = np.random.Philox(key=seed, counter=((s << 64) + (1 << 128) - 1) % (1 << 256)).random_raw(4)
        u = (raw >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
        eta = law.eta_lo + (law.eta_hi - law.eta_lo) * float(u[0])
        th = math.radians(law.theta_lo + (law.theta_hi - law.theta_lo) * float(u[1]))
        tx, ty = (eta * law.lam, law.lam) if c["scale"] else (math.sqrt(eta * law.lam), math.sqrt(law.lam))

        def cov(dx, dy):
            rx, ry = math.cos(th) * dx - math.sin(th) * dy, math.sin(th) * dx + math.cos(th) * dy
            x = 2.0 * math.sqrt(c["nu"]) * torch.sqrt((rx / tx) ** 2 + (ry / ty) ** 2)
            poly = 1.0 if c["nu"] == 0.5 else 1.0 + x if c["nu"] == 1.5 else 1.0 + x + x * x / 3.0
            return poly * torch.exp(-x)

        k1, k2 = torch.arange(M1, device=DEV), torch.arange(M2, device=DEV)
        d1 = torch.where(k1 <= M1 // 2, k1, k1 - M1).double()[None, :] * 2.0 ** -(c["P"] + 1)
        d2 = torch.where(k2 <= M2 // 2, k2, k2 - M2).double()[:, None] * 2.0 ** -(c["Q"] + 1)
        arr = cov(d1, d2)
        arr[:, M1 // 2] = 0.5 * (cov(d1[:, M1 // 2], d2[:, 0]) + cov(-d1[:, M1 // 2], d2[:, 0]))
        arr[M2 // 2] = 0.5 * (cov(d1[0], d2[M2 // 2]) + cov(d1[0], -d2[M2 // 2]))
        arr[M2 // 2, M1 // 2] = 0.5 * (cov(d1[0, M1 // 2], d2[M2 // 2, 0]) + cov(d1[0, M1 // 2], -d2[M2 // 2, 0]))
        lam = torch.fft.fft2(arr).real.clamp_(min=0.0)
        xi = torch.view_as_complex(_normals(seed, s, 2 * M1 * M2).reshape(M2, M1, 2))
        Zs.append(torch.fft.fft2(torch.sqrt(lam / (M1 * M2)) * xi).real[:n2, :n1].reshape(-1))
        ets.append([eta, th])
    return {"Z": torch.stack(Zs), "eta_theta": torch.tensor(ets, dtype=torch.float64), "status": None}


def exact(case, seed):
    c = case
    gen = torch.Generator(device=DEV).manual_seed(seed)
    if c["kind"] in ("solve", "step"):
        shapes = _shapes(c)
        # block elimination costs min^3 max per grid, and as many sequential steps as the longer side
        cost = sum(2.0 ** (3 * min(p, q) + max(p, q)) for P, Q in shapes for p in range(1, P + 1) for q in range(1, Q + 1))
        steps = sum(2 ** max(p, q) for P, Q in set(shapes) for p in range(1, P + 1) for q in range(1, Q + 1))
        if cost > 1e12 or steps > 60000:
            return None
        if c["kind"] == "solve":
            Qx, u = _exact_solve(c, shapes, _fields(shapes, c["M"], gen))
            return {"Q": Qx, "status": None, **({"u": u} if c.get("with_u") else {})}
        xi = torch.stack([_normals(seed, i, c["M"]) for i in range(c["S"])])
        Z, base = [None] * c["S"], {}
        for i, (P, Q) in enumerate(shapes):
            if (P, Q) not in base:
                Phi, sl = _basis((2 << P) + 1, (2 << Q) + 1, c["M"])
                base[P, Q] = Phi * sl
            Z[i] = base[P, Q] @ xi[i]
        Z = torch.cat(Z)
        Qx, _ = _exact_solve(c, shapes, Z)
        r, dQ, Y, off = 1.733, [], [], 0
        for P, Q in shapes:
            G = Qx[off:off + P * Q].reshape(P, Q)
            off += P * Q
            pad = torch.zeros(P - c["p0"] + 2, Q - c["q0"] + 2, dtype=torch.float64, device=DEV)
            pad[1:, 1:] = G[c["p0"] - 1:, c["q0"] - 1:]
            d = pad[1:, 1:] - pad[:-1, 1:] - pad[1:, :-1] + pad[:-1, :-1]
            w = torch.exp(r * (torch.arange(d.shape[0], device=DEV)[:, None] + torch.arange(d.shape[1], device=DEV)).double())
            dQ.append(d.reshape(-1))
            Y.append((d * w).sum())
        return {"Z": Z, "Q": Qx, "status": None, "dQ": torch.cat(dQ), "Y": torch.stack(Y)}
    if c["kind"] == "field":
        Phi, sl = _basis(c["nx"], c["ny"], c["M"])
        xi = torch.randn(c["S"], c["M"], dtype=torch.float64, device=DEV, generator=gen)
        return (xi * sl) @ Phi.T
    if c["kind"] == "ce":
        return _exact_ce(c, seed)
    if c["kind"] == "history":
        return None
    return torch.stack([_normals(seed, i, c["M"]) for i in range(c["S"])])
