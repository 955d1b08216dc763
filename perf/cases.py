"""Cases of use of this framework: what a program that solves PDEs by probabilistic
domain decomposition asks of it, through the public API of ``paper_1705_03666_gb300.api``.

Stage one estimates the solution at interface nodes by Monte Carlo paths (or trees);
stage two interpolates the estimates and solves the subdomains.  Sizes are those of the
five workloads of ``workloads.py``, of the README and of the tests; the random seed of
every solve (and the parameters, node values and cotangents where a case has any) comes
from the case's seed.

Every family (``kind``) of case and what it stands for:

  interface  ``Context.interface_solve``: node estimates by Euler-Maruyama paths.  Small
             calls are one subdomain interface or one rank's share; the large one is the
             4096-node 3-D workload at its full path count; Robin faces take the
             reflecting scheme of the same entry point.
  train      ``interface_values`` forward and backward: fitting boundary and drift
             parameters of the Poisson problem to data.
  jacobian   ``Context.interface_grad``: the sensitivities of every node with their errors.
  batch      ``Context.batch_solve``: a mixed batch of domains with adaptive path counts.
  trees      ``Context.branching_solve``: the semilinear problem at space-time nodes.
  grid       ``Context.branching_grid_solve``: the same in a bounded domain, one tree
             per sample for all grid times.
  wos        ``Context.wos_solve``: Walk on Spheres for the Laplace problem.
  mlmc       ``Context.mlmc_solve``: the multilevel estimate.
  pdd2d      ``laplace_pdd_solve``: both stages in 2-D, FP64 paths (the API's default).
  stage2_3d  ``elliptic3d_pdd_solve``: stage two in 3-D from given node estimates.
"""
import math

import numpy as np
import torch

from paper_1705_03666_gb300 import api, workloads as W

SEED = 0x1705036660000000

# mean exit times of the node sets below (units of time; steps = time / dt), for work()
_MEAN_EXIT = {"square": 0.108, "lshape": 0.060, "cube": 0.0493, "fourier": 0.084, "robin": 0.325}
# floating-point operations of one path step (or walk jump, tree segment, grid step)
_STEP_FLOPS = {"square": 60, "lshape": 80, "cube": 105, "fourier": 106, "robin": 90}


def listed():
    return [
        # smallest calls: one interface of one subdomain at the path count of a
        # first look; launches and the longest path's latency count
        {"name": "laplace2d_small_fp32", "kind": "interface", "domain": "square", "nodes": 16,
         "paths": 2000, "dt": 1e-3, "precision": "fp32"},
        # ragged sizes on the non-convex domain (its two interfaces)
        {"name": "lshape_ragged_fp32", "kind": "interface", "domain": "lshape", "nodes": 301,
         "paths": 5003, "dt": 1e-3, "precision": "fp32"},
        # the headline workload: 4096 nodes of the cube, 1e5 paths each
        {"name": "elliptic3d_4096x1e5_fp32", "kind": "interface", "domain": "cube", "nodes": 4096,
         "paths": 100000, "dt": 1e-4, "precision": "fp32"},
        # Neumann and Robin faces (Eq. 2.4) on the 2-D nodes
        {"name": "robin2d_16x1e6_fp32", "kind": "interface", "domain": "robin", "nodes": 16,
         "paths": 1000000, "dt": 1e-3, "precision": "fp32"},
        # one training pass on the derivative workload: values and gradients
        {"name": "poisson_train_2048x1e5", "kind": "train", "nodes": 2048, "paths": 100000,
         "dt": 1e-3},
        # a tenth of the mixed batch (square, L-shape, cube; two time steps)
        {"name": "batch_mixed_2000", "kind": "batch", "nodes": 2000, "n_max": 50000,
         "target_se": 4.5e-4},
        # the KPP workload: 1024 space-time nodes, 1e5 trees each
        {"name": "kpp_trees_1024x1e5", "kind": "trees", "nodes": 1024, "trees": 100000,
         "beta": 1.0},
        # KPP on the square: 48 nodes, 16 grid times
        {"name": "kpp_grid_square_48x1e5", "kind": "grid", "nodes": 48, "times": 16,
         "trees": 100000, "dt": 1e-3},
        # Walk on Spheres on the 2-D nodes
        {"name": "wos_16x1e6_fp32", "kind": "wos", "nodes": 16, "paths": 1000000, "eps": 1e-4,
         "domain": "square", "precision": "fp32"},
        # four levels of the multilevel estimate
        {"name": "mlmc_16_4levels", "kind": "mlmc", "nodes": 16, "levels": 4, "paths": 400000,
         "dt": 4e-3},
        # the README's two-stage call: FP64 paths, spline, two 129 x 129 halves
        {"name": "pdd2d_16x1e4_129", "kind": "pdd2d", "nodes": 16, "paths": 10000, "dt": 1e-3,
         "grid": 129},
        # 3-D stage two on the 4 x 4 x 4 split: 9 plane interpolants, 64 boxes of 33^3
        {"name": "stage2_3d_4096_129", "kind": "stage2_3d", "nodes": 4096, "grid": 129,
         "split": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["interface", "interface", "interface", "interface", "train", "jacobian",
                       "batch", "trees", "grid", "wos", "mlmc", "pdd2d", "stage2_3d"])
    if kind == "interface":
        domain = rng.choice(["square", "lshape", "cube", "robin"])
        dt = rng.choice([1e-3, 1e-3, 5e-4, 1e-4])
        precision = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        nodes = _log(rng, 1, 4096)
        # up to 2e10 path steps (FP64: 2e8, its rate is 1/64)
        steps = 2e10 if precision == "fp32" else 2e8
        most = max(100, min(1000000, int(steps * dt / (_MEAN_EXIT[domain] * nodes))))
        return {"kind": kind, "domain": domain, "nodes": nodes, "paths": _log(rng, 100, most),
                "dt": dt, "precision": precision}
    if kind in ("train", "jacobian"):
        nodes = 4 * _log(rng, 1, 512)
        return {"kind": kind, "nodes": nodes,
                "paths": _log(rng, 100, max(100, min(100000, 100000000 // nodes))), "dt": 1e-3}
    if kind == "batch":
        return {"kind": kind, "nodes": _log(rng, 100, 3000), "n_max": _log(rng, 2000, 50000),
                "target_se": rng.choice([4.5e-4, 2e-3])}
    if kind == "trees":
        return {"kind": kind, "nodes": 16 * _log(rng, 1, 64), "trees": _log(rng, 1000, 200000),
                "beta": rng.choice([0.5, 1.0, 1.5])}
    if kind == "grid":
        return {"kind": kind, "nodes": 3 * _log(rng, 1, 16), "times": rng.randint(1, 16),
                "trees": _log(rng, 1000, 100000), "dt": rng.choice([1e-3, 2e-3])}
    if kind == "wos":
        return {"kind": kind, "nodes": _log(rng, 1, 200), "paths": _log(rng, 1000, 300000),
                "eps": rng.choice([1e-3, 1e-4, 1e-5]), "domain": rng.choice(["square", "lshape"]),
                "precision": rng.choice(["fp32", "fp32", "fp64"])}
    if kind == "mlmc":
        return {"kind": kind, "nodes": _log(rng, 1, 32), "levels": rng.randint(2, 5),
                "paths": _log(rng, 10000, 400000), "dt": 4e-3}
    if kind == "pdd2d":
        return {"kind": kind, "nodes": rng.randint(4, 32), "paths": _log(rng, 500, 20000),
                "dt": 1e-3, "grid": rng.randint(33, 257)}
    split = rng.choice([2, 4, 4])
    return {"kind": kind, "nodes": _log(rng, 200, 4096), "grid": split * rng.randint(8, 32) + 1,
            "split": split}


# --------------------------------------------------------------------------
# Inputs of a case (host values; shared by prepare and exact)
# --------------------------------------------------------------------------
def _problem(case, seed):
    kind = case["kind"]
    domain = case.get("domain", "square")
    if kind in ("train", "jacobian"):
        return W.poisson_fourier(seed % (1 << 31))
    if kind == "trees":
        return W.kpp("sigmoid", 4.0, case["beta"])
    if kind == "grid":
        return W.kpp("travelling", float(np.sqrt(4.0 / 3.0)), 4.0, geometry="unit_square")
    if kind == "stage2_3d" or domain == "cube":
        return W.elliptic_manufactured()
    if domain == "robin":
        return W.laplace_expcos("unit_square", reflect=[2, 1], phi=-2.0)
    return W.laplace_expcos("l_shape" if domain == "lshape" else "unit_square")


def _nodes(case):
    kind, n = case["kind"], case["nodes"]
    domain = case.get("domain", "square")
    if kind in ("train", "jacobian"):
        return W.nodes_cfg5(n // 4)
    if kind == "trees":
        return W.nodes_kpp()[:n]
    if kind == "grid":
        y = np.arange(1, n // 3 + 1, dtype=np.float64) / (n // 3 + 1)
        return np.concatenate([np.stack([np.full_like(y, x), y], 1) for x in (0.25, 0.5, 0.75)])
    if kind == "stage2_3d" or domain == "cube":
        return W.nodes_cube_planes(n)
    if domain == "lshape":
        return W.nodes_lshape_interfaces(n)
    return W.nodes_cfg1(n)


def _plane_nodes(case, seed):
    """3-D stage two: the nodes on the planes of the case's split (the 4 x 4 x 4
    recipe's planes, or the one middle plane per axis of a 2 x 2 x 2 split), the
    axis each belongs to, and stage-one estimates: the exact solution plus noise of
    the size of the workload's standard error."""
    x = W.nodes_cube_planes(case["nodes"])
    axis = np.arange(case["nodes"]) % 3
    if case["split"] == 2:
        x[np.arange(len(x)), axis] = 0.5
    u = np.sin(np.pi * x[:, 0]) * np.sin(np.pi * x[:, 1]) * np.exp(x[:, 2])
    noise = np.random.default_rng(seed).standard_normal(len(x))
    if case["split"] == 2:  # the recipe repeats its in-plane points on its three planes
        keep = (np.arange(len(x)) // 3) % 3 == 0
        x, axis, u, noise = x[keep], axis[keep], u[keep], noise[keep]
    return x, axis, u + 2.5e-3 * noise


# --------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    dev = torch.device("cuda", 0)
    s = {"kind": kind, "case": case, "seed": SEED + seed}
    if kind == "batch":
        n = case["nodes"]
        square, lshape = int(0.35 * n), int(0.35 * n)
        mix = W.batch_mix(square, lshape, n - square - lshape, seed=3)
        s["problems"] = mix["problems"]
        s["nodes"] = torch.from_numpy(mix["nodes"]).to(dev)
        s["index"] = torch.from_numpy(mix["problem_index"]).to(dev)
        s["dt"] = torch.from_numpy(mix["dt"]).to(dev)
        s["ctx"] = api.Context(mix["problems"][0])
        return s
    prob = _problem(case, seed)
    s["ctx"] = api.Context(prob)
    if kind == "pdd2d":
        return s
    if kind == "stage2_3d":
        x, axis, u = _plane_nodes(case, seed)
        s["nodes"] = torch.from_numpy(x).to(dev)
        s["axis"] = torch.from_numpy(axis).to(dev)
        s["values"] = torch.from_numpy(u).to(dev)
        return s
    s["nodes"] = torch.from_numpy(_nodes(case)).to(dev)
    if kind in ("train", "jacobian"):
        s["theta"] = torch.from_numpy(prob["params"][:64].copy()).to(dev).requires_grad_()
        s["phi"] = torch.from_numpy(prob["params"][64:].copy()).to(dev).requires_grad_()
        rng = np.random.default_rng(seed + 1)
        s["cotangent"] = torch.from_numpy(rng.standard_normal(case["nodes"])).to(dev)
    if kind == "mlmc":
        s["counts"] = [max(1, case["paths"] >> l) for l in range(case["levels"])]
    if kind == "grid":
        s["times"] = np.arange(1, case["times"] + 1, dtype=np.float64) / 16.0
    return s


def run(s):
    kind, c, ctx = s["kind"], s["case"], s["ctx"]
    if kind == "interface":
        r = ctx.interface_solve(s["nodes"], seed=s["seed"], dt=c["dt"], n_paths=c["paths"],
                                precision=c["precision"])
        return {k: r[k] for k in ("mean", "se", "n")}
    if kind == "train":
        u = api.interface_values(s["theta"], s["phi"], ctx, s["nodes"], seed=s["seed"],
                                 dt=c["dt"], n_paths=c["paths"])
        dtheta, dphi = torch.autograd.grad(u, (s["theta"], s["phi"]), s["cotangent"])
        return {"u": u.detach(), "dtheta": dtheta, "dphi": dphi}
    if kind == "jacobian":
        r = ctx.interface_grad(s["nodes"], seed=s["seed"], dt=c["dt"], n_paths=c["paths"],
                               grad_out=s["cotangent"])
        return {k: r[k] for k in ("jac", "jac_se", "dtheta", "dphi")}
    if kind == "batch":
        r = ctx.batch_solve(s["problems"], s["nodes"], s["index"], s["dt"], seed=s["seed"],
                            n_pilot=1000, n_min=1000, n_max=c["n_max"],
                            target_se=c["target_se"])
        return {k: r[k] for k in ("mean", "se", "n")}
    if kind == "trees":
        r = ctx.branching_solve(s["nodes"], seed=s["seed"], n_trees=c["trees"])
        return {k: r[k] for k in ("mean", "se", "n")}
    if kind == "grid":
        r = ctx.branching_grid_solve(s["nodes"], s["times"], seed=s["seed"], n_trees=c["trees"],
                                     dt=c["dt"])
        return {k: r[k] for k in ("mean", "se", "n")}
    if kind == "wos":
        r = ctx.wos_solve(s["nodes"], seed=s["seed"], n_paths=c["paths"], eps=c["eps"],
                          precision=c["precision"])
        return {k: r[k] for k in ("mean", "se", "n")}
    if kind == "mlmc":
        r = ctx.mlmc_solve(s["nodes"], seed=s["seed"], dt0=c["dt"], n_per_level=s["counts"])
        return {"mean": r["mean"], "se": r["se"],
                "levels": [{"mean": v["mean"], "var": v["var"]} for v in r["levels"]]}
    if kind == "pdd2d":
        r = api.laplace_pdd_solve(ctx, seed=s["seed"], n_nodes=c["nodes"], n_paths=c["paths"],
                                  dt=c["dt"], grid=(c["grid"], c["grid"]))
        return {k: r[k] for k in ("mean", "se", "left", "right")}
    r = api.elliptic3d_pdd_solve(ctx, s["nodes"], s["values"], s["axis"], grid=c["grid"],
                                 split=c["split"])
    planes = torch.stack([r["plane_values"][k] for k in sorted(r["plane_values"])])
    return {"u": r["u"], "planes": planes}


def work(case):
    """Bytes: inputs read once and outputs written once.  Operations: those of the
    method's steps (mean path lengths times the operations of a step), or of stage two's
    solves."""
    kind, n = case["kind"], case.get("nodes", 0)
    if kind == "interface":
        d = 3 if case["domain"] == "cube" else 2
        steps = n * case["paths"] * (_MEAN_EXIT[case["domain"]] / case["dt"])
        return {"bytes": n * (8 * d + 24), "flops": steps * _STEP_FLOPS[case["domain"]]}
    if kind in ("train", "jacobian"):
        steps = n * case["paths"] * (_MEAN_EXIT["fourier"] / case["dt"])
        f = _STEP_FLOPS["fourier"]
        per = (2 * f + 16) if kind == "train" else f + 16
        return {"bytes": n * (16 + 16 + (1280 if kind == "jacobian" else 0)) + 1280,
                "flops": steps * per}
    if kind == "batch":
        # half the nodes at dt = 1e-3 and half at 1e-4, most at the path cap
        per = sum(share * (_MEAN_EXIT[k] / 2) * (1e3 + 1e4) * _STEP_FLOPS[k]
                  for k, share in (("square", 0.35), ("lshape", 0.35), ("cube", 0.3)))
        var = {4.5e-4: 1.0, 2e-3: 0.3}.get(case["target_se"], 1.0)
        return {"bytes": n * (24 + 4 + 8 + 24), "flops": n * max(1000, case["n_max"] * var) * per}
    if kind == "trees":
        t = np.arange(1, 17) / 16.0
        segments = n * case["trees"] * float(np.mean(2.0 * np.exp(case["beta"] * t) - 1.0))
        return {"bytes": n * 48, "flops": segments * 60}
    if kind == "grid":
        steps = n * case["trees"] * 155.0 * (1e-3 / case["dt"]) * min(1.0, case["times"] / 4.0)
        return {"bytes": n * (24 + 16 * case["times"]), "flops": steps * 80}
    if kind == "wos":
        jumps = n * case["paths"] * (3.0 + 2.4 * -math.log10(case["eps"]))
        return {"bytes": n * 40, "flops": jumps * 45}
    if kind == "mlmc":
        steps = sum((case["paths"] >> l) * 0.108 / (case["dt"] / 2 ** l) * (1.5 if l else 1.0)
                    for l in range(case["levels"]))
        return {"bytes": n * (32 + 16 * case["levels"]), "flops": n * steps * 70}
    if kind == "pdd2d":
        steps = n * case["paths"] * (_MEAN_EXIT["square"] / case["dt"])
        p = case["grid"] - 2
        return {"bytes": n * 32 + 16 * case["grid"] ** 2, "flops": steps * 60 + 16.0 * p ** 3}
    planes = 3 * (case["split"] - 1)
    m = n / (9.0 if case["split"] == 4 else 9.0) + 131
    p = (case["grid"] - 1) // case["split"] - 1
    return {"bytes": n * 40 + 8 * case["grid"] ** 3 + planes * 8 * case["grid"] ** 2,
            "flops": planes * (2.0 / 3.0 * m ** 3 + 10.0 * m * case["grid"] ** 2)
            + case["split"] ** 3 * 12.0 * p ** 4}


# --------------------------------------------------------------------------
# Plain 64-bit values (torch only): the same discrete estimators on the same
# documented random streams, and the same discrete systems of stage two.
# --------------------------------------------------------------------------
_MASK = 0xFFFFFFFF


def _mulhilo(m, x):
    hi = (x * (m >> 16) + ((x * (m & 0xFFFF)) >> 16)) >> 16
    return hi, (x * m) & _MASK


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    k0, k1 = seed & _MASK, (seed >> 32) & _MASK
    for _ in range(10):
        h0, l0 = _mulhilo(0xD2511F53, c0)
        h1, l1 = _mulhilo(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return [c0, c1, c2, c3]


def _unif(w):
    return ((w >> 9).double() + 0.5) * 2.0 ** -23


def _normals(a, b):
    r, th = torch.sqrt(-2.0 * torch.log(_unif(a))), 2.0 * math.pi * _unif(b)
    return r * torch.cos(th), r * torch.sin(th)


def _g(domain, x):
    if domain == "cube":
        return torch.sin(math.pi * x[:, 0]) * torch.sin(math.pi * x[:, 1]) * torch.exp(x[:, 2])
    return torch.exp(x[:, 0]) * torch.cos(x[:, 1])


def _face_dists(domain, x):
    """Distances to the faces (face 2k + s on x_k = s; the L-shape's notch edges last)."""
    d = [f for k in range(x.shape[1]) for f in (x[:, k], 1.0 - x[:, k])]
    if domain == "lshape":
        for a, b in ((x[:, 0], 0.5 - x[:, 1]), (x[:, 1], 0.5 - x[:, 0])):
            d.append(torch.where(a >= 0.5, b, torch.sqrt((0.5 - a) ** 2 + b * b)))
    return torch.stack(d, 1)


def _project(domain, x, face):
    x = x.clone()
    for k in range(x.shape[1]):
        for side in (0, 1):
            x[:, k] = torch.where(face == 2 * k + side, float(side), x[:, k])
    if domain == "lshape":
        for f, k in ((4, 1), (5, 0)):
            on = face == f
            x[:, k] = torch.where(on, 0.5, x[:, k])
            x[:, 1 - k] = torch.where(on, x[:, 1 - k].clamp(min=0.5), x[:, 1 - k])
    return x


def _outside(domain, x):
    out = ((x < 0.0) | (x > 1.0)).any(1)
    return out | ((x > 0.5).all(1)) if domain == "lshape" else out


def _segment_exit(domain, x0, x1):
    d = x1 - x0
    t = torch.where(x1 < 0.0, x0 / (x0 - x1), torch.where(x1 > 1.0, (1.0 - x0) / d, 2.0))
    tb, kb = t.min(1)
    vb = (x1.gather(1, kb[:, None])[:, 0] > 1.0).double()
    if domain == "lshape":
        a = x0
        cross = (0.5 - a) / d
        tl = torch.where(d > 0, cross, torch.where(d < 0, -1.0, torch.where(a > 0.5, 0.0, 2.0)))
        th = torch.where(d > 0, 2.0, torch.where(d < 0, cross, torch.where(a > 0.5, 1.0, -1.0)))
        lo, kent = tl.max(1)
        hi = th.min(1).values
        enters = (lo < hi) & (lo <= 1.0) & (hi > 0.0) & (lo.clamp(min=0.0) < tb)
        tb = torch.where(enters, lo.clamp(min=0.0), tb)
        kb = torch.where(enters, kent, kb)
        vb = torch.where(enters, 0.5, vb)
    xe = (x0 + tb[:, None] * d).scatter(1, kb[:, None], vb[:, None])
    return xe.clamp(0.0, 1.0)


def _paths_exact(domain, nodes, seed, dt, n_paths):
    """Per-node mean and standard error of the Euler-Maruyama + Brownian-bridge scores."""
    dev = torch.device("cuda", 0)
    nodes = torch.from_numpy(nodes).to(dev)
    n, dim = nodes.shape
    total = n * n_paths
    score = torch.zeros(total, dtype=torch.float64, device=dev)
    idx = torch.arange(total, device=dev)
    x, z = nodes[idx // n_paths].clone(), torch.zeros(total, dtype=torch.float64, device=dev)
    step = 0
    c = -1.0 if domain == "cube" else 0.0
    while idx.numel():
        node, path = idx // n_paths, idx % n_paths
        zero = torch.zeros_like(idx)
        w = [v for b in range(3) for v in _philox(zero + 3 * (step // 4) + b, path, node, zero, seed)]
        if dim == 3:
            zs = [v for j in range(6) for v in _normals(w[2 * j], w[2 * j + 1])]
            us = [((w[3 * j] & 255) << 8) | ((w[3 * j + 1] & 255) << 16) | ((w[3 * j + 2] & 255) << 24)
                  for j in range(4)]
        else:
            zs = [v for j in range(4) for v in _normals(w[2 * j], w[2 * j + 1])]
            us = w[8:12]
        alive = torch.ones_like(idx, dtype=torch.bool)
        for j in range(4):
            xi = torch.stack(zs[dim * j:dim * j + dim], 1)
            y0, y1 = math.exp(c * step * dt), math.exp(c * (step + 1) * dt)
            b = torch.zeros_like(x)
            f = 0.0
            if domain == "cube":
                sx, cx = torch.sin(math.pi * x[:, 0]), torch.cos(math.pi * x[:, 0])
                sy, cy = torch.sin(math.pi * x[:, 1]), torch.cos(math.pi * x[:, 1])
                ez = torch.exp(x[:, 2])
                b[:, 0], b[:, 1] = sy * cy, 0.5 - sx * sx
                f = -((0.5 * (1.0 - 2.0 * math.pi ** 2) - 1.0) * sx * sy * ez
                      + math.pi * (b[:, 0] * cx * sy * ez + b[:, 1] * sx * cy * ez))
            xn = x + b * dt + math.sqrt(dt) * xi
            zn = z + f * y0 * dt
            hard = _outside(domain, xn)
            e = 2.0 * _face_dists(domain, x) * _face_dists(domain, xn) / dt
            p = torch.where(e < 18.0, torch.exp(-e), 0.0)
            pbest, face = p.max(1)
            cross = ~hard & (_unif(us[j]) < 1.0 - torch.prod(1.0 - p, 1)) & (pbest > 0.0)
            ends = alive & (hard | cross)
            if bool(ends.any()):
                xe = torch.where(hard[ends][:, None], _segment_exit(domain, x[ends], xn[ends]),
                                 _project(domain, xn[ends], face[ends]))
                score[idx[ends]] = _g(domain, xe) * y1 + zn[ends]
                alive &= ~ends
            x, z = xn, zn
            step += 1
        idx, x, z = idx[alive], x[alive], z[alive]
    s = score.reshape(n, n_paths)
    mean = s.mean(1)
    se = torch.sqrt(((s - mean[:, None]) ** 2).sum(1) / max(1, n_paths - 1) / n_paths)
    return {"mean": mean, "se": se,
            "n": torch.full((n,), n_paths, dtype=torch.int64, device=dev)}


def _wos_exact(domain, nodes, seed, n_paths, eps):
    dev = torch.device("cuda", 0)
    nodes = torch.from_numpy(nodes).to(dev)
    n = nodes.shape[0]
    means, ses = [], []
    for i in range(n):
        score = torch.zeros(n_paths, dtype=torch.float64, device=dev)
        idx = torch.arange(n_paths, device=dev)
        x = nodes[i].expand(n_paths, 2).clone()
        k, w = 0, None
        while idx.numel():
            d, face = _face_dists(domain, x).min(1)
            stop = d <= eps
            score[idx[stop]] = _g(domain, _project(domain, x[stop], face[stop]))
            go = ~stop
            idx, x, d = idx[go], x[go], d[go]
            if k % 4 == 0:
                zero = torch.zeros_like(idx)
                w = _philox(zero + k // 4, idx, zero + i, zero + 2, seed)
            else:
                w = [v[go] for v in w]
            th = 2.0 * math.pi * _unif(w[k % 4])
            x = x + d[:, None] * torch.stack([torch.cos(th), torch.sin(th)], 1)
            k += 1
        means.append(score.mean())
        ses.append(torch.sqrt(((score - means[-1]) ** 2).sum() / max(1, n_paths - 1) / n_paths))
    return {"mean": torch.stack(means), "se": torch.stack(ses),
            "n": torch.full((n,), n_paths, dtype=torch.int64, device=dev)}


def _spline(s, y, t):
    """Not-a-knot cubic spline through (s, y) at t (dense system for the second derivatives)."""
    K = len(s) - 1
    h = np.diff(s)
    A, r = np.zeros((K + 1, K + 1)), np.zeros(K + 1)
    for i in range(1, K):
        A[i, i - 1:i + 2] = h[i - 1], 2.0 * (h[i - 1] + h[i]), h[i]
        r[i] = 6.0 * ((y[i + 1] - y[i]) / h[i] - (y[i] - y[i - 1]) / h[i - 1])
    A[0, :3] = h[1], -(h[0] + h[1]), h[0]
    A[K, K - 2:] = h[K - 1], -(h[K - 2] + h[K - 1]), h[K - 2]
    m = np.linalg.solve(A, r)
    i = np.clip(np.searchsorted(s, t, side="right") - 1, 0, K - 1)
    a, b = s[i + 1] - t, t - s[i]
    return (m[i] * a ** 3 + m[i + 1] * b ** 3) / (6.0 * h[i]) \
        + (y[i] / h[i] - m[i] * h[i] / 6.0) * a + (y[i + 1] / h[i] - m[i + 1] * h[i] / 6.0) * b


def _sines(p):
    k = np.arange(1, p + 1)
    return torch.from_numpy(np.sin(np.pi * (np.outer(k, k) % (2 * (p + 1))) / (p + 1))).cuda()


def _laplace_half(x0, iface_x, grid, iface):
    """5-point solution on [x0, x0 + 1/2] x [0, 1] with g = e^x cos y and the interface column."""
    xs, ys = x0 + 0.5 * np.arange(grid) / (grid - 1), np.arange(grid) / (grid - 1.0)
    u = np.exp(xs)[None, :] * np.cos(ys)[:, None]
    u[1:-1, 1:-1] = 0.0
    u[:, -1 if iface_x > x0 else 0] = iface
    hx, hy, p = 0.5 / (grid - 1), 1.0 / (grid - 1), grid - 2
    f = np.zeros((p, p))
    f[:, 0] += u[1:-1, 0] / hx ** 2
    f[:, -1] += u[1:-1, -1] / hx ** 2
    f[0] += u[0, 1:-1] / hy ** 2
    f[-1] += u[-1, 1:-1] / hy ** 2
    S = _sines(p)
    lam = torch.from_numpy(4.0 * np.sin(np.pi * np.arange(1, p + 1) / (2.0 * (p + 1))) ** 2).cuda()
    F = torch.from_numpy(f).cuda()
    U = (S @ F @ S) / (lam[:, None] / hy ** 2 + lam[None, :] / hx ** 2)
    out = torch.from_numpy(u).cuda()
    out[1:-1, 1:-1] = (S @ U @ S) * (4.0 / (p + 1) ** 2)
    return out


def _pdd2d_exact(case, seed):
    n, grid = case["nodes"], case["grid"]
    y = np.arange(1, n + 1) / (n + 1.0)
    r = _paths_exact("square", np.stack([np.full(n, 0.5), y], 1), seed, case["dt"], case["paths"])
    s = np.concatenate([[0.0], y, [1.0]])
    v = np.concatenate([[math.exp(0.5)], r["mean"].cpu().numpy(), [math.exp(0.5) * math.cos(1.0)]])
    iface = _spline(s, v, np.arange(grid) / (grid - 1.0))
    g0, g1 = math.exp(0.5), math.exp(0.5) * math.cos(1.0)
    iface[0], iface[-1] = g0, g1
    return {"mean": r["mean"], "se": r["se"], "left": _laplace_half(0.0, 0.5, grid, iface),
            "right": _laplace_half(0.5, 0.5, grid, iface)}


def _plane_exact(axis, pos, x, v, grid, n_bnd=32):
    """Cubic RBF with a linear term through the plane's nodes and its perimeter."""
    o = [b for b in range(3) if b != axis]
    e = np.arange(n_bnd) / n_bnd
    one, nil = np.ones(n_bnd), np.zeros(n_bnd)
    per = np.concatenate([np.stack(p, 1) for p in ((e, nil), (one, e), (1 - e, one), (nil, 1 - e))])
    q = np.zeros((len(per), 3))
    q[:, axis], q[:, o[0]], q[:, o[1]] = pos, per[:, 0], per[:, 1]
    pts = torch.from_numpy(np.concatenate([x[:, o], per])).cuda()
    val = torch.from_numpy(np.concatenate(
        [v, np.sin(np.pi * q[:, 0]) * np.sin(np.pi * q[:, 1]) * np.exp(q[:, 2])])).cuda()
    m = len(pts)
    A = torch.zeros(m + 3, m + 3, dtype=torch.float64, device="cuda")
    A[:m, :m] = ((pts[:, None] - pts[None]) ** 2).sum(-1) ** 1.5
    A[:m, m], A[:m, m + 1:] = 1.0, pts
    A[m, :m], A[m + 1:, :m] = 1.0, pts.T
    w = torch.linalg.solve(A, torch.cat([val, val.new_zeros(3)]))
    t = torch.linspace(0.0, 1.0, grid, dtype=torch.float64, device="cuda")
    rows = []
    for t2 in t:  # slow axis o[1]
        qq = torch.stack([t, t2.expand_as(t)], 1)
        r3 = ((qq[:, None] - pts[None]) ** 2).sum(-1) ** 1.5
        rows.append(r3 @ w[:m] + w[m] + qq @ w[m + 1:])
    return torch.stack(rows)


def _stage2_3d_exact(case, seed):
    x, axis, v = _plane_nodes(case, seed)
    split, grid = case["split"], case["grid"]
    planes = {}
    for a in range(3):
        for k in range(1, split):
            sel = (x[:, a] == k / split) & (axis == a)
            planes[(a, k)] = _plane_exact(a, k / split, x[sel], v[sel], grid)
    p, m = (grid - 1) // split - 1, (grid - 1) // split + 1
    h = 1.0 / (grid - 1)
    # Dirichlet data on every box: g outside, the planes inside (lowest face index first)
    t = torch.linspace(0.0, 1.0, grid, dtype=torch.float64, device="cuda")
    Z, Y, X = torch.meshgrid(t, t, t, indexing="ij")
    g = torch.sin(math.pi * X) * torch.sin(math.pi * Y) * torch.exp(Z)
    b0, b1 = 0.5 * torch.sin(2 * math.pi * Y), 0.5 * torch.cos(2 * math.pi * X)
    f = -(0.5 * (1.0 - 2.0 * math.pi ** 2) * g - g
          + math.pi * torch.exp(Z) * (b0 * torch.cos(math.pi * X) * torch.sin(math.pi * Y)
                                      + b1 * torch.sin(math.pi * X) * torch.cos(math.pi * Y)))
    S = _sines(p)
    cm1 = torch.cos(math.pi * torch.arange(1, p + 1, dtype=torch.float64, device="cuda") / (p + 1)) - 1
    lam = (cm1[:, None, None] + cm1[None, :, None] + cm1[None, None, :]) / h ** 2 - 1.0
    scale = 8.0 / (p + 1) ** 3
    out = torch.empty_like(g)
    for kz in range(split):
        for ky in range(split):
            for kx in range(split):
                kk = (kx, ky, kz)
                sl = tuple(slice(k * (m - 1), k * (m - 1) + m) for k in kk[::-1])
                u = torch.zeros(m, m, m, dtype=torch.float64, device="cuda")
                for fc in reversed(range(6)):  # faces with interface data, lowest index last
                    a, side = fc >> 1, fc & 1
                    k = kk[a] + side
                    if 0 < k < split:
                        o = [b for b in range(3) if b != a]
                        pg = planes[(a, k)][sl[2 - o[1]], sl[2 - o[0]]]
                        u.select(2 - a, -1 if side else 0).copy_(pg)
                for fc in range(6):  # the cube's own faces carry g
                    a, side = fc >> 1, fc & 1
                    if not 0 < kk[a] + side < split:
                        u.select(2 - a, -1 if side else 0).copy_(
                            g[sl].select(2 - a, -1 if side else 0))
                i = slice(1, -1)
                bb0, bb1, ff = b0[sl][i, i, i], b1[sl][i, i, i], f[sl][i, i, i]
                for _ in range(20):
                    c = u[i, i, i]
                    lap = (u[i, i, 2:] + u[i, i, :-2] + u[i, 2:, i] + u[i, :-2, i] + u[2:, i, i]
                           + u[:-2, i, i] - 6.0 * c) / h ** 2
                    r = -ff - (0.5 * lap + bb0 * (u[i, i, 2:] - u[i, i, :-2]) / (2 * h)
                               + bb1 * (u[i, 2:, i] - u[i, :-2, i]) / (2 * h) - c)
                    r = torch.einsum("zyx,xa,yb,zc->cba", r, S, S, S) / lam * scale
                    u[i, i, i] += torch.einsum("zyx,xa,yb,zc->cba", r, S, S, S)
                out[sl] = u
    return {"u": out, "planes": torch.stack([planes[k] for k in sorted(planes)])}


def exact(case, seed):
    """None where a plain torch pass over all paths (or trees) would take too long: the
    large path solves, training, the batch and the tree solves."""
    kind, key = case["kind"], SEED + seed
    if kind == "interface" and case["domain"] != "robin":
        steps = case["nodes"] * case["paths"] * _MEAN_EXIT[case["domain"]] / case["dt"]
        if steps < 4e8 and case["nodes"] * case["paths"] < 4e6 and case["dt"] >= 5e-4:
            return _paths_exact(case["domain"], _nodes(case), key, case["dt"], case["paths"])
    if kind == "wos" and case["nodes"] * case["paths"] <= 2e7:
        return _wos_exact(case["domain"], _nodes(case), key, case["paths"], case["eps"])
    if kind == "pdd2d":
        return _pdd2d_exact(case, key)
    if kind == "stage2_3d":
        return _stage2_3d_exact(case, seed)
    return None
