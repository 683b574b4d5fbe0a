"""What a program built on this package spends its time on: one pass of each case is
the calls such a program makes, through the package's public entry points.

A case is an operation ("op") on a geometry:

  block    Y = H X on a block of K images and X' = H^T R on a block of K sinograms,
           the two products of every MM-GKS step (and of any other Krylov solver)
  jac      J_theta dtheta, then J_theta^T r at the same image (its layout reused): an
           inner Gauss-Newton product
  gn       the fused per-view Gauss-Newton terms with the residual: one iteration of
           the parameter update
  train    autograd: projection and the gradients of 1/2 |H x - b|^2 in x, theta (and
           delta), as a learned reconstruction calls it
  solve    a whole reconstruction (RMM-GKS at fixed angles, or NL-RMM-GKS that also
           estimates them)

Handles run at the launch shapes they are created with, except where "plan" asks for
the shapes the autotuner picks for the benchmark workload, kept by the program.
"""
import math

import numpy as np
import torch

from paper_2605_06336_gb300 import autograd, ct

DEV = "cuda"
# launch shapes of the benchmark workload's handle (ct_set_tuning order)
PLAN = [4, 4, 1, 8, 4, 4, 1, 0, 0, 8, 2, 1]


def _bins(N):
    return int(math.ceil(math.sqrt(2.0) * N))


def listed():
    return [
        # the smallest call: one 64 x 64 image, 90 views; latency and launches
        _case("block", 64, 90, name="block_64_k1"),
        # the ordinary one-column product: every Enlarge step projects one new basis column
        _case("block", 256, 180, name="block_256_k1"),
        # the benchmark's Krylov block of 8 at the shapes its autotuned handle keeps
        _case("block", 256, 180, K=8, plan=True, name="block_256_k8_plan"),
        # dynamic CT: 16 frames with 30-120 views each, a block of 8, one launch per product
        _case("block", 256, 1200, K=8, frames=16, angles="golden", name="block_256_f16_k8"),
        # one streamed chunk of 120 views of the 2048 x 2048 problem: the largest image
        _case("block", 2048, 120, angles="chunk", name="block_2048_k1"),
        # fan beam (the paper's CT geometry), a block of 8
        _case("block", 256, 180, K=8, fan=2.0, name="fan_256_k8"),
        # the precision of the paper's arithmetic, on an odd-sized image
        _case("block", 255, 181, K=4, fp64=True, name="block_255_k4_fp64"),
        # inner Gauss-Newton products at one image
        _case("jac", 256, 180, name="jac_256"),
        # parameter update at 512 x 512 with detector offsets
        _case("gn", 512, 360, offsets=True, angles="grid", name="gn_512_offsets"),
        # learned reconstruction: a minibatch of 4, gradients in image, angles and offsets
        _case("train", 512, 360, K=4, offsets=True, angles="grid", name="train_512_k4_offsets"),
        # whole reconstruction, single precision, angles known: two outer iterations of 20 Enlarge
        # steps, enough for every part of the loop; further ones repeat it
        _case("solve", 256, 180, outer=2, name="solve_256_fp32"),
        # whole joint reconstruction in double precision: image and angles
        _case("solve", 64, 90, fp64=True, outer=2, joint=True, name="solve_64_joint_fp64"),
    ]


def _case(op, N, V, K=1, frames=1, offsets=False, fan=0.0, fp64=False, plan=False, angles="random", outer=0,
          joint=False, bins=0, name=None):
    c = {"op": op, "N": N, "V": V, "B": bins or _bins(N), "K": K, "frames": frames, "offsets": offsets, "fan": fan,
         "fp64": fp64, "plan": plan, "angles": angles, "outer": outer, "joint": joint}
    if name:
        c["name"] = name
    return c


def draw(rng):
    """One more case of the listed kinds: sides 32..2048, 8..1440 views, blocks of 1..8,
    bounded by the listed cases' cost."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["block", "block", "block", "block", "block", "jac", "gn", "train", "solve"])
    if op == "solve":
        joint = rng.random() < 0.4
        # (joint solves in double precision: small; fixed angles in single precision: up to the listed one)
        N = log(32, 64) if joint else log(64, 256)
        V = rng.randint(30, 90) if joint else rng.randint(60, 180)
        return _case(op, N, V, fp64=joint, joint=joint, outer=2, angles=rng.choice(["random", "grid"]))
    kind = rng.choice(["f32", "f32", "f32", "frames", "fan", "f64"]) if op == "block" else "f32"
    cap = {"f32": 4.0e8, "frames": 6.0e8, "fan": 9.0e7, "f64": 4.0e7}[kind]  # V N^2 K
    while True:
        K = rng.choice([1, 1, 2, 3, 4, 5, 8, 8]) if op in ("block", "train") else 1
        N = log(32, 2048)
        V = log(8, 1440)
        if V * N * N * K <= cap:
            break
    c = _case(op, N, V, K=K, offsets=rng.random() < 0.3, angles=rng.choice(["random", "grid", "golden", "chunk"]))
    if rng.random() < 0.3:  # a detector narrower or wider than the image's diagonal
        c["B"] = max(8, int(c["B"] * rng.uniform(0.7, 1.2)))
    if kind == "frames":
        c["frames"] = min(rng.randint(2, 16), V)
        c["angles"] = "golden"
    elif kind == "fan":
        c["fan"] = rng.choice([1.5, 2.0, 4.0])
    elif kind == "f64":
        c["fp64"] = True
    elif K >= 4 and op == "block" and rng.random() < 0.4:
        c["plan"] = True
    return c


# --- inputs -------------------------------------------------------------------

def _views_per_frame(c, rng):
    """Uneven view counts that add up to V (30-120 for the listed 16-frame case)."""
    F, V = c["frames"], c["V"]
    if F == 1:
        return [V]
    w = rng.uniform(0.4, 1.6, F)
    n = np.maximum(1, np.floor(V * w / w.sum()).astype(int))
    while n.sum() > V:
        n[int(np.argmax(n))] -= 1
    n[int(np.argmin(n))] += V - n.sum()
    return [int(x) for x in n]


def _angles(c, rng):
    V = c["V"]
    if c["angles"] == "grid":
        nominal = np.arange(V) * (math.pi / V)
    elif c["angles"] == "golden":
        nominal = np.mod(np.arange(V) * (math.pi * (math.sqrt(5.0) - 1.0) / 2.0), math.pi)
    elif c["angles"] == "chunk":  # a random subset of a 12 times finer grid
        nominal = np.sort(rng.permutation(12 * V)[:V]) * (math.pi / (12 * V))
    else:
        nominal = np.sort(rng.uniform(0.0, math.pi, V))
    return nominal, nominal + rng.normal(0.0, math.radians(0.5), V)


def _phantom(N, rng, count=10):
    """Overlapping random ellipses of random intensity (N x N, float64)."""
    h = 0.5 * (N - 1)
    x = torch.arange(N, dtype=torch.float64, device=DEV)[None, :] - h
    y = h - torch.arange(N, dtype=torch.float64, device=DEV)[:, None]
    img = torch.zeros(N, N, dtype=torch.float64, device=DEV)
    for _ in range(count):
        r, a = 0.35 * N * math.sqrt(rng.uniform()), rng.uniform(0.0, 2.0 * math.pi)
        cx, cy = r * math.cos(a), r * math.sin(a)
        p, q, phi, rho = rng.uniform(0.05 * N, 0.25 * N), rng.uniform(0.05 * N, 0.25 * N), rng.uniform(0, math.pi), rng.uniform()
        u = ((x - cx) * math.cos(phi) + (y - cy) * math.sin(phi)) / p
        v = ((y - cy) * math.cos(phi) - (x - cx) * math.sin(phi)) / q
        img += rho * (u * u + v * v <= 1.0)
    return img


def _inputs(c, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    N, V, B, K, F = c["N"], c["V"], c["B"], c["K"], c["frames"]
    T = torch.float64 if c["fp64"] else torch.float32
    s = {"vpf": _views_per_frame(c, rng), "T": T}
    nominal, true = _angles(c, rng)
    s["nominal"] = torch.tensor(nominal, dtype=torch.float64, device=DEV)
    s["theta"] = torch.tensor(true, dtype=torch.float64, device=DEV)
    s["delta"] = torch.tensor(rng.normal(0.0, 0.5, V), dtype=torch.float64, device=DEV) if c["offsets"] else None

    def noise(*shape):
        return torch.randn(*shape, generator=gen, dtype=T, device=DEV)

    if c["op"] == "block":  # basis columns: image structure and oscillation, unit norm
        X = torch.stack([torch.cat([_phantom(N, rng, 4).reshape(-1) for _ in range(min(F, 2))] * ((F + 1) // 2))[: F * N * N]
                         for _ in range(min(K, 2))]).to(T)
        X = X.repeat((K + 1) // 2 if K > 1 else 1, 1)[:K] + 0.3 * noise(K, F * N * N)
        s["X"] = (X / X.norm(dim=1, keepdim=True)).contiguous()
        R = noise(K, V, B)
        R = R + 2.0 * noise(K, V, 1)  # residuals: noise and per-view structure
        s["R"] = (R / R.reshape(K, -1).norm(dim=1)[:, None, None]).reshape(K, V * B).contiguous()
    else:
        img = _phantom(N, rng)
        s["true"] = img
        # the current iterate: the image blurred by one pixel, each of a minibatch with its own error
        blur = (img + torch.roll(img, 1, 0) + torch.roll(img, 1, 1) + torch.roll(img, (1, 1), (0, 1))) / 4
        X = torch.stack([blur * (1.0 - 0.05 * k) for k in range(K)]).reshape(K, N * N).to(T)
        s["X"] = (X + 0.02 * noise(K, N * N)).contiguous()
        if c["op"] == "jac":
            s["dtheta"] = torch.tensor(rng.normal(0.0, 0.01, V), dtype=torch.float64, device=DEV)
            s["r"] = noise(V * B)
        else:  # measured data: the true image at the true angles with 1 % noise
            y = torch.cat([_sum(_value, img.reshape(1, -1), w) for w in _walks(c, s["theta"], s["delta"], [V])]).reshape(-1)
            e = torch.randn(V * B, generator=gen, dtype=torch.float64, device=DEV)
            e *= 0.01 * y.norm() / e.norm()
            s["noise"] = float(e.norm())
            s["b"] = (y + e).to(T).contiguous()
            if c["op"] == "train":
                s["b"] = s["b"].expand(K, -1).contiguous()
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    s["op"] = ct.CTOperator(case["N"], case["B"], case["V"], views_per_frame=s["vpf"] if case["frames"] > 1 else None,
                            max_batch=8 if case["op"] == "solve" else case["K"], dtype=s["T"],
                            source_distance=case["fan"] * case["N"] if case["fan"] else None)
    if case["plan"]:
        s["op"].tuning = PLAN
    if case["op"] == "train":
        s["X"].requires_grad_()
        s["theta"].requires_grad_()
        if s["delta"] is not None:
            s["delta"].requires_grad_()
    return s


def run(s):
    op, c = s["op"], s["case"]
    if c["op"] == "block":
        return {"Y": op.forward(s["X"], s["theta"], s["delta"]), "X": op.adjoint(s["R"], s["theta"], s["delta"])}
    if c["op"] == "jac":
        dy = op.jac(s["X"], s["theta"], s["dtheta"], s["delta"])
        return {"dy": dy, "g": op.jacT(None, s["theta"], s["r"], s["delta"])}
    if c["op"] == "gn":
        g, j2, f, res = op.gn_terms(s["X"], s["theta"], s["b"], s["delta"], want_residual=True)
        return {"grad": g, "jnorm2": j2, "f": f, "res": res}
    if c["op"] == "train":
        y = autograd.project(s["X"], s["theta"], op, s["delta"])
        wrt = [s["X"], s["theta"]] + ([s["delta"]] if s["delta"] is not None else [])
        return {"y": y.detach(), "grads": list(torch.autograd.grad(y, wrt, y.detach() - s["b"]))}
    x, theta, _ = op.solve(s["b"], s["nominal"] if c["joint"] else s["theta"], noise_norm=s["noise"],
                           update_theta=int(c["joint"]), outer_iters=c["outer"], stop_on_convergence=0, tol1=0.0)
    return {"x": x, "theta": theta}


def work(case):
    """Each input read and each output written once; two multiply-adds for each of the
    0.9 V N^2 interpolations of a product (four in the derivative ones)."""
    e = 8 if case["fp64"] else 4
    n, m, K = case["frames"] * case["N"] ** 2, case["V"] * case["B"], case["K"]
    steps = 0.9 * case["V"] * case["N"] ** 2 * K
    ang = 8 * case["V"] * (2 if case["offsets"] else 1)
    if case["op"] == "block":
        return {"bytes": 2 * e * K * (n + m) + ang, "flops": 8 * steps}
    if case["op"] == "jac":
        return {"bytes": e * (n + 2 * m) + 3 * ang, "flops": 16 * steps}
    if case["op"] == "gn":
        return {"bytes": e * (n + 2 * m) + ang + 24 * case["V"], "flops": 8 * steps}
    if case["op"] == "train":
        return {"bytes": e * K * (2 * n + 2 * m) + 2 * ang, "flops": 16 * steps}
    # Enlarge enlarges the basis from 5 to 25 columns: H, H^T, and the column products of a step
    cols, nsteps = 25, 20 * case["outer"]
    return {"bytes": e * (n + m) + 2 * ang, "flops": nsteps * (8 * steps + 2 * cols * (6 * n + 3 * m) + 2 * n * cols * cols)}


# --- the same in 64 bits --------------------------------------------------------

def _walks(c, theta, delta, vpf):
    """The operator's rows in chunks of views: for each, the frame, pixel indices, weights and
    derivatives of every sample (views x bins x march steps)."""
    N, B = c["N"], c["B"]
    h = 0.5 * (N - 1)
    per = max(1, (1 << 23) // (N * B))
    start = 0
    for f, count in enumerate(vpf):
        for v0 in range(start, start + count, per):
            th = theta[v0:min(v0 + per, start + count)].detach()[:, None]
            d = delta[v0:min(v0 + per, start + count)].detach()[:, None] if delta is not None else 0.0
            s = torch.arange(B, dtype=torch.float64, device=DEV)[None, :] - 0.5 * (B - 1) + d
            co, si = torch.cos(th), torch.sin(th)
            if c["fan"]:
                D = c["fan"] * N
                rx, ry = s * co - D * si, s * si + D * co
                px, py = s * co, s * si
                rows = rx.abs() <= ry.abs()
                C = torch.where(rows, rx / ry, ry / rx)
                qh = torch.where(rows, h + px - py * C, h - (py - px * C))
                qr, w = -C, torch.sqrt(1 + C * C)
                dq = dw = qb = None
            else:
                t = torch.remainder(th, math.pi)
                rows = ((t <= math.pi / 4) | (t >= 3 * math.pi / 4)).expand(-1, B)
                qb = torch.where(rows, 1 / co, -1 / si)
                qr = torch.where(rows, si / co, co / si)
                qh = h + s * qb
                w = torch.where(rows, 1 / co.abs(), 1 / si.abs())
                dw = torch.where(rows, torch.sign(co) * si / co ** 2, -torch.sign(si) * co / si ** 2)
                g0 = torch.where(rows, s * si / co ** 2, s * co / si ** 2)
                gr = torch.where(rows, 1 / co ** 2, -1 / si ** 2)
                dq = (g0, gr)
            r = torch.arange(N, dtype=torch.float64, device=DEV)
            q = qh[:, :, None] + (r - h) * qr[:, :, None]
            cell = torch.floor(q)
            fr = q - cell
            cell = cell.clamp(-2, N).long()
            ri = torch.arange(N, device=DEV)

            def index(k):
                k_in = k.clamp(0, N - 1)
                i = torch.where(rows[:, :, None], ri * N + k_in, k_in * N + ri) + f * N * N
                return i, ((k >= 0) & (k < N)).double()

            i0, m0 = index(cell)
            i1, m1 = index(cell + 1)
            walk = {"i0": i0, "i1": i1, "m0": m0, "m1": m1, "fr": fr, "w": w, "dw": dw, "qb": qb,
                    "v0": v0, "v1": v0 + th.shape[0]}
            if dq is not None:
                walk["dq"] = dq[0][:, :, None] + (r - h) * dq[1][:, :, None]
            yield walk
        start += count


def _value(x, k):
    a, b = x[k["i0"]] * k["m0"], x[k["i1"]] * k["m1"]
    return k["w"] * (a + k["fr"] * (b - a)).sum(2)


def _dtheta(x, k):
    a, b = x[k["i0"]] * k["m0"], x[k["i1"]] * k["m1"]
    return k["dw"] * (a + k["fr"] * (b - a)).sum(2) + k["w"] * ((b - a) * k["dq"]).sum(2)


def _ddelta(x, k):
    a, b = x[k["i0"]] * k["m0"], x[k["i1"]] * k["m1"]
    return k["w"] * k["qb"] * (b - a).sum(2)


def _sum(what, X, k):
    return torch.stack([what(x, k) for x in X], 1)  # views x images x bins


def _all(what, X, c, s):
    return torch.cat([_sum(what, X, k) for k in _walks(c, s["theta"], s["delta"], s["vpf"])]).transpose(0, 1).reshape(len(X), -1)


def _transpose(R, c, s):
    out = torch.zeros(len(R), c["frames"] * c["N"] ** 2, dtype=torch.float64, device=DEV)
    for k in _walks(c, s["theta"], s["delta"], s["vpf"]):
        for x, r in zip(out, R):
            y = (k["w"] * r.reshape(c["V"], c["B"])[k["v0"]:k["v1"]])[:, :, None]
            x.index_add_(0, k["i0"].reshape(-1), (y * (1 - k["fr"]) * k["m0"]).reshape(-1))
            x.index_add_(0, k["i1"].reshape(-1), (y * k["fr"] * k["m1"]).reshape(-1))
    return out


def exact(case, seed):
    if case["op"] == "solve":
        return None  # an iteration, with no closed result
    c, s = case, _inputs(case, seed)
    X = s["X"].double()
    V = c["V"]
    if c["op"] == "block":
        return {"Y": _all(_value, X, c, s), "X": _transpose(s["R"].double(), c, s)}
    if c["op"] == "jac":
        J = _all(_dtheta, X, c, s)
        dy = (J.reshape(V, -1) * s["dtheta"][:, None]).reshape(-1)
        return {"dy": dy, "g": (J.reshape(V, -1) * s["r"].double().reshape(V, -1)).sum(1)}
    y = _all(_value, X, c, s)
    J = _all(_dtheta, X, c, s).reshape(len(X), V, -1)
    r = y - s["b"].double().reshape(len(X), -1)
    rv = r.reshape(len(X), V, -1)
    if c["op"] == "gn":
        return {"grad": (J * rv).sum((0, 2)), "jnorm2": (J * J).sum((0, 2)), "f": 0.5 * (rv * rv).sum((0, 2)),
                "res": r.reshape(-1)}
    grads = [_transpose(r, c, s), (J * rv).sum((0, 2))]
    if s["delta"] is not None:
        grads.append((_all(_ddelta, X, c, s).reshape(len(X), V, -1) * rv).sum((0, 2)))
    return {"y": y, "grads": grads}
