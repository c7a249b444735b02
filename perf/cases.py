"""The work this library is used for, as measurable cases.

Each case is one call, or one short sequence of calls, that a planner makes
through the public binding (``paper_2310_01775_gb300.stamp``): rolling plans
out and differentiating them, the Stein update of the particles, the learned
surrogate's screening, planning and training steps, and a batched solve.
Sizes are those of the named workloads (``workloads.CONFIGS``), of the tests
and of the benchmark, and ragged ones between.

Contact constants.  At the workloads' literal constants (k = 1e4 N/m, dt =
0.01 s) the contact dynamics are chaotic: a last-bit change grows to O(1)
within a few pushes, so no two float32 programs agree there.  The rollouts
here use the softer contact of the tests (k = 1e3 N/m, c = 10 N s/m) with half
the substep and pushes of up to 0.05 m, where float32 results are reproducible
over whole plans of nearly every particle; the work per substep is the same.
"""
import math

import numpy as np
import torch

from paper_2310_01775_gb300 import stamp as S
from paper_2310_01775_gb300 import workloads as W

PHYSICS = dict(W.PHYSICS, k_contact=1e3, c_contact=10.0, dt=0.005, dist_max=0.05)
ITER = 3                       # Gumbel draws of the iteration a rollout belongs to
HIDDEN = 256                   # the surrogate network's width
ADAM_STEP, LR = 40, 1e-2       # a step in the middle of a solve


def listed():
    return [
        # one block, two short pushes, 32 particles: the smallest plan; launch and
        # latency of one forward rollout and its reverse sweep
        dict(name="rollout_1block_small", kind="rollout", nb=1, H=2, T=50, C=25, N=32, each=False),
        # one block, four pushes, 1024 particles, every substep on the tape
        dict(name="rollout_1block", kind="rollout", nb=1, H=4, T=100, C=1, N=1024, each=False),
        # three blocks with block-block contact, the benchmark's size: the
        # largest part of a solve's time
        dict(name="rollout_3block", kind="rollout", nb=3, H=6, T=100, C=25, N=2048, each=False),
        # four blocks, replanning from each particle's own start poses, a ragged count
        dict(name="rollout_4block_replan", kind="rollout", nb=4, H=5, T=100, C=25, N=613, each=True),
        # the Stein update (distances, median bandwidth, direction, Adam) of the smallest plan
        dict(name="stein_small", kind="stein", nb=1, H=2, N=32, structured=False, weighted=False),
        # ... of the benchmark's particles
        dict(name="stein_3block", kind="stein", nb=3, H=6, N=2048, structured=False, weighted=False),
        # ... of a large ragged set of wide plans
        dict(name="stein_large_ragged", kind="stein", nb=4, H=6, N=6001, structured=False, weighted=False),
        # the structured kernel with importance weights (the solver's other variants)
        dict(name="stein_structured", kind="stein", nb=1, H=4, N=1024, structured=True, weighted=True),
        # 131072 candidate plans screened down to 2048 by the surrogate
        dict(name="screen", kind="screen", nb=3, H=6, rows=131072, N=2048),
        # the surrogate's costs and gradients in an early iteration of a solve
        dict(name="surrogate_rollout", kind="surrogate", nb=3, H=6, N=2048),
        # forward and backward of one training minibatch of the surrogate's network
        dict(name="mlp_train_step", kind="mlp_step", nb=3, rows=16384),
        # batched serving: uneven problems (1-4 blocks, 2-8 pushes, 64-1024
        # particles) solved together, four iterations and the final evaluation
        dict(name="batch_solve", kind="batch", n=64, H_max=8, N_max=1024, T=100, iters=4, persistent=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rollout", "rollout", "rollout", "stein", "stein", "screen", "surrogate",
                       "mlp_step", "batch"])
    if kind == "rollout":
        nb = rng.choice([1, 2, 3, 4])
        H = rng.randint(1, 4 if nb == 1 else 6)
        T, C = rng.choice([(50, 25), (50, 1), (100, 25), (100, 1), (100, 20), (60, 12)])
        top = {1: 1024, 2: 2048, 3: 2048, 4: 1024}[nb]
        return dict(kind=kind, nb=nb, H=H, T=T, C=C, N=_log(rng, 24, top), each=rng.random() < 0.25)
    if kind == "stein":
        structured = rng.random() < 0.3
        return dict(kind=kind, nb=rng.choice([1, 2, 3, 4]), H=rng.randint(1, 4 if structured else 6),
                    N=_log(rng, 24, 1024 if structured else 6000), structured=structured,
                    weighted=rng.random() < 0.3)
    if kind == "screen":
        rows = _log(rng, 4096, 131072)
        return dict(kind=kind, nb=rng.choice([1, 2, 3]), H=rng.randint(1, 6), rows=rows,
                    N=_log(rng, 64, 2048))
    if kind == "surrogate":
        return dict(kind=kind, nb=rng.choice([1, 2, 3]), H=rng.randint(1, 8), N=_log(rng, 64, 4096))
    if kind == "mlp_step":
        return dict(kind=kind, nb=rng.choice([1, 2, 3]), rows=_log(rng, 256, 32768))
    return dict(kind=kind, n=_log(rng, 8, 64), H_max=rng.randint(2, 6), N_max=_log(rng, 80, 512),
                T=rng.choice([50, 100]), iters=rng.randint(1, 4), persistent=rng.random() < 0.5)


# ------------------------------- inputs --------------------------------------
def _params(case):
    return dict(PHYSICS, n_blocks=case["nb"], H=case["H"], T=case.get("T", 100),
                ckpt_every=case.get("C", 25))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, shape, lo=-1.0, hi=1.0):
    return torch.rand(shape, generator=g, device="cuda") * (hi - lo) + lo


def _normal(g, shape, scale):
    return torch.randn(shape, generator=g, device="cuda") * scale


def _net(g, in_dim, out_dim, head=1.0):
    """A packed network (W_l (out, in), b_l), uniform in +-1/sqrt(in); `head` scales the last layer."""
    sizes = [in_dim, HIDDEN, HIDDEN, HIDDEN, out_dim]
    parts = []
    for l, (i, o) in enumerate(zip(sizes[:-1], sizes[1:])):
        s = (head if l == 3 else 1.0) / math.sqrt(i)
        parts += [_uniform(g, o * i, -s, s), _uniform(g, o, -s, s)]
    return torch.cat(parts)


def _dims(case):
    m = 4 * case["nb"]
    return m, m + 2, case.get("H", 1) * (m + 2)


def _inputs(case, seed):
    """The arrays of a case (prepare() and exact() see the same ones)."""
    g, kind = _gen(seed), case["kind"]
    M, P, D = _dims(case) if kind != "batch" else (0, 0, 0)
    a = {}
    if kind in ("rollout", "surrogate"):
        a["init"], a["goal"] = W.scene({"n_blocks": case["nb"]}, seed)
        a["theta"] = _uniform(g, (case["N"], D))          # a solve's start distribution
        if case.get("each"):   # start poses near the scene's, as after a disturbance
            base = torch.tensor(a["init"], dtype=torch.float32, device="cuda")
            a["start"] = (base + _normal(g, (case["N"], case["nb"], 3), 0.003)).contiguous()
    if kind == "stein":
        n = case["N"]
        a["theta"] = _uniform(g, (n, D))
        a["grad"] = _normal(g, (n, D), 0.1)
        a["m"] = _normal(g, (n, D), 0.02)
        a["v"] = _normal(g, (n, D), 0.05).square() + 1e-4
        a["relaxed"], a["hard"] = _uniform(g, n, 0.0, 1.0), _uniform(g, n, 0.0, 1.0)
    if kind in ("screen", "surrogate"):
        a["init"], a["goal"] = W.scene({"n_blocks": case["nb"]}, seed)
        # pose changes of a few centimetres per push, like a trained network's
        a["net"] = _net(g, 8 * case["nb"] + 2, 3 * case["nb"], 0.25)
    if kind == "screen":
        a["theta"] = _uniform(g, (case["rows"], D))
    if kind == "mlp_step":
        a["net"] = _net(g, 8 * case["nb"] + 2, 3 * case["nb"])
        a["x"] = _uniform(g, (case["rows"], 8 * case["nb"] + 2))
        a["dy"] = _normal(g, (case["rows"], 3 * case["nb"]), 1.0 / case["rows"])
    if kind == "batch":
        a["instances"] = []
        for k, (nb, H, N, _) in enumerate(_sizes(case)):
            init, goal = W.scene({"n_blocks": nb}, 1000 * seed + k)
            a["instances"].append(dict(n_blocks=nb, H=H, N=N, seed=1000 * seed + k, init=init, goal=goal))
    return a


def prepare(case, seed):
    st = torch.cuda.current_stream().cuda_stream
    kind, a = case["kind"], _inputs(case, seed)
    s = {"case": dict(case), "seed": int(seed), **a}
    new = lambda *shape: torch.empty(shape, device="cuda")  # noqa: E731
    if kind == "rollout":
        p = s["problem"] = S.Problem(_params(case), a["init"], a["goal"], case["N"], st)
        s["cost"], s["final"], s["out"] = new(case["N"]), new(case["N"], p.S), new(case["N"], p.D)
    elif kind == "stein":
        init, goal = W.scene({"n_blocks": case["nb"]}, seed)
        p = s["problem"] = S.Problem(_params(case), init, goal, case["N"], st)
        if case["structured"]:
            p.set_svgd_kernel(1)
        s["h"], s["phi"] = new(1), new(case["N"], p.D)
    elif kind in ("screen", "surrogate"):
        P, n = _params(case), case["N"]
        p = s["problem"] = S.Problem(P, a["init"], a["goal"], n, st)
        sur = s["surrogate"] = S.Surrogate(P, case.get("rows", n), n, st)
        sur.set_params(a["net"])
        s["cost"], s["out"] = new(n), new(n, p.D)
        s["index"] = torch.empty(n, dtype=torch.int32, device="cuda")
    elif kind == "mlp_step":
        i, o, n = 8 * case["nb"] + 2, 3 * case["nb"], case["rows"]
        net = s["mlp"] = S.MLP(i, o, n, n, st)
        net.set_params(a["net"])
        s["y"], s["dx"], s["dparams"] = new(n, o), new(n, i), new(net.n_params)
    else:
        b = s["batch"] = S.Batch(dict(PHYSICS, T=case["T"]), a["instances"], st)
        b.set_persistent(case["persistent"])
        s["thetas"] = torch.empty(sum(d["N"] * d["H"] * (4 * d["n_blocks"] + 2) for d in a["instances"]),
                                  device="cuda")
        s["views"], at = [], 0
        for d in a["instances"]:
            n = d["N"] * d["H"] * (4 * d["n_blocks"] + 2)
            s["views"].append(s["thetas"][at:at + n])
            at += n
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "rollout":
        p, n, seed = s["problem"], case["N"], s["seed"]
        if case["each"]:
            p.rollout_fwd_from(s["theta"], s["start"], n, seed, ITER, 0, s["cost"], s["final"])
        else:
            p.rollout_fwd(s["theta"], n, seed, ITER, 0, s["cost"], s["final"])
        p.rollout_adjoint(s["theta"], n, seed, ITER, s["out"])
        return {"cost": s["cost"], "final": s["final"], "grad": s["out"]}
    if kind == "stein":
        p, n = s["problem"], case["N"]
        if case["weighted"]:
            p.svgd_step_weighted(s["theta"], s["grad"], s["relaxed"], s["hard"], n, s["m"], s["v"],
                                 ADAM_STEP, LR, s["h"], s["phi"])
        else:
            p.svgd_step(s["theta"], s["grad"], n, s["m"], s["v"], ADAM_STEP, LR, 0, s["h"], s["phi"])
        return {"theta": s["theta"], "m": s["m"], "v": s["v"], "h": s["h"], "phi": s["phi"]}
    if kind == "screen":
        s["surrogate"].screen(s["problem"], s["theta"], case["rows"], case["N"], s["out"], s["index"])
        return {"theta": s["out"], "index": s["index"]}
    if kind == "surrogate":
        s["surrogate"].rollout(s["problem"], s["theta"], case["N"], s["seed"], ITER, s["cost"], s["out"])
        return {"cost": s["cost"], "grad": s["out"]}
    if kind == "mlp_step":
        s["mlp"].forward_saved(s["x"], case["rows"], s["y"], 0)
        s["mlp"].backward(s["dy"], case["rows"], 0, s["dx"], s["dparams"])
        return {"y": s["y"], "dx": s["dx"], "dparams": s["dparams"]}
    # the particles and the best hard cost of every instance (not the indices of
    # the best plans: where two costs tie to rounding, either may come first)
    s["batch"].solve(case["iters"], 1e-3)
    for k, v in enumerate(s["views"]):
        s["batch"].read_theta(k, v)
    return {"theta": s["thetas"], "best_cost": s["batch"].results()["best_cost"]}


# ------------------------------- work ----------------------------------------
def _rollout_flops(nb):
    """Forward FLOP per particle and substep: every pusher's contact with its own
    block (75), the reach tests of the other (pusher, block) and corner pairs
    (8 and 12), trigonometry, friction and integration (60 per block)."""
    return 4 * nb * 75 + 4 * nb * (nb - 1) * (8 + 12) + 60 * nb


def work(case):
    kind = case["kind"]
    if kind == "batch":
        fl = by = 0
        for nb, H, N, D in _sizes(case):
            fl += case["iters"] * (3 * _rollout_flops(nb) * H * case["T"] * N + N * N * (3 * D + D))
            by += 4 * (2 * N * D)
        return {"bytes": by, "flops": fl}
    M, P, D = _dims(case)
    if kind == "rollout":   # the reverse sweep does about twice the forward's arithmetic
        n = case["N"]
        return {"bytes": 4 * (2 * n * D + n * (1 + 6 * case["nb"])),
                "flops": 3 * _rollout_flops(case["nb"]) * n * case["H"] * case["T"]}
    if kind == "stein":     # distances (half the pairs), k g and k (theta_i - theta_j), Adam
        n = case["N"]
        return {"bytes": 4 * 8 * n * D, "flops": n * n * (1.5 * D + 4 * D) + 12 * n * D}
    F, O = 8 * case["nb"] + 2, 3 * case["nb"]
    net = 2 * (F * HIDDEN + 2 * HIDDEN * HIDDEN + HIDDEN * O)   # one row through the network
    if kind == "screen":
        return {"bytes": 4 * (case["rows"] + case["N"]) * D + 4 * case["N"],
                "flops": net * case["rows"] * case["H"]}
    if kind == "surrogate":
        return {"bytes": 4 * (2 * case["N"] * D + case["N"]), "flops": 2 * net * case["N"] * case["H"]}
    n_params = net // 2 + 3 * HIDDEN + O
    return {"bytes": 4 * (case["rows"] * (2 * F + 2 * O) + n_params), "flops": 3 * net * case["rows"]}


def _sizes(case):
    """The instances of a batch: (blocks, pushes, particles, D) of each."""
    rng = np.random.default_rng(case["n"])
    out = []
    for _ in range(case["n"]):
        nb, H = int(rng.integers(1, 5)), int(rng.integers(2, case["H_max"] + 1))
        N = int(math.exp(rng.uniform(math.log(64), math.log(case["N_max"]))))
        out.append((nb, H, N, H * (4 * nb + 2)))
    return out


# --------------------- the same results in 64 bits ---------------------------
def _sm64(key, ctr):
    """SplitMix64: output ctr + 1 of the generator started at `key`."""
    with np.errstate(over="ignore"):
        z = np.uint64(key) + (np.asarray(ctr, dtype=np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _relax(theta, case, seed, noise):
    """Choice weights (N, H, M), tangential offsets and push distances (N, H)."""
    M, P, _ = _dims(case)
    H, n = case["H"], theta.shape[0]
    f = lambda k: float(np.float32(PHYSICS[k]))  # noqa: E731
    th = theta.reshape(n, H, P)
    a = th[:, :, :M]
    if noise:
        key = _sm64(_sm64(np.uint64(seed), 0), ITER)
        u = ((_sm64(key, np.arange(n * H * M)) >> np.uint64(41)).astype(np.float64) + 0.5) / 2.0 ** 23
        a = a + torch.tensor(-np.log(-np.log(u)), device="cuda").reshape(n, H, M)
    return (torch.softmax(a / f("tau"), -1), f("offset_max") * torch.tanh(th[:, :, M]),
            f("dist_max") * torch.sigmoid(th[:, :, M + 1]))


def _cost(q, dist, goal):
    f = lambda k: float(np.float32(PHYSICS[k]))  # noqa: E731
    goal = torch.tensor(np.asarray(goal, dtype=np.float32).astype(np.float64), device="cuda")
    e = q - goal
    yaw = torch.atan2(torch.sin(e[..., 2]), torch.cos(e[..., 2]))
    return ((e[..., :2] ** 2).sum((1, 2)) + f("w_yaw") * (yaw ** 2).sum(1) + f("w_push") * (dist ** 2).sum(1))


def _square(px, py, bx, by, c, s, hs):
    """Signed distance of points to squares and the outward unit normals."""
    dx, dy = px - bx, py - by
    lx, ly = c * dx + s * dy, -s * dx + c * dy
    qx, qy = lx.abs() - hs, ly.abs() - hs
    one, zero = torch.ones_like(lx), torch.zeros_like(lx)
    sx, sy = torch.where(lx >= 0, one, -one), torch.where(ly >= 0, one, -one)
    out = (qx > 0) | (qy > 0)
    mx, my = qx.clamp(min=0), qy.clamp(min=0)
    ln = torch.sqrt(torch.where(out, mx * mx + my * my, one))
    xa = qx >= qy
    nlx = torch.where(out, sx * mx / ln, torch.where(xa, sx, zero))
    nly = torch.where(out, sy * my / ln, torch.where(xa, zero, sy))
    return torch.where(out, ln, torch.maximum(qx, qy)), c * nlx - s * nly, s * nlx + c * nly


def _simulate(theta, case, seed, start, goal):
    """Cost and final state of every plan, in the dtype of theta."""
    from torch.utils.checkpoint import checkpoint
    f = lambda k: float(np.float32(PHYSICS[k]))  # noqa: E731
    nb, T, n = case["nb"], case["T"], theta.shape[0]
    hs, r, dt, m = f("half_size"), f("pusher_r"), f("dt"), f("mass")
    inertia = m * (2 * (2 * hs) ** 2) / 12
    weight = f("mu") * m * f("g")
    lever = 2 * hs / 6 * (math.sqrt(2) + math.log(1 + math.sqrt(2)))
    z, off, dist = _relax(theta, case, seed, True)
    normals = theta.new_tensor([[0, 1], [1, 0], [0, -1], [-1, 0]]).repeat(nb, 1)
    obj = torch.arange(nb, device="cuda").repeat_interleave(4)
    pairs = [(a, b) for a in range(nb) for b in range(nb) if a != b]
    own = torch.tensor([a for a, b in pairs for _ in range(4)], device="cuda", dtype=torch.long)
    oth = torch.tensor([b for a, b in pairs for _ in range(4)], device="cuda", dtype=torch.long)
    corner = theta.new_tensor([[1, 1], [-1, 1], [-1, -1], [1, -1]]).repeat(len(pairs), 1) * hs

    def contact(delta, nx, ny, wx, wy):
        vn = wx * nx + wy * ny
        fn = torch.where(delta > 0, (f("k_contact") * delta - f("c_contact") * vn).clamp(min=0),
                         torch.zeros_like(delta))
        tx, ty = wx - vn * nx, wy - vn * ny
        return fn, f("mu_c") * fn / torch.sqrt(tx * tx + ty * ty + f("eps_t") ** 2), tx, ty

    def push(q, v, w, offset, length):
        c0, s0 = torch.cos(q[:, obj, 2]), torch.sin(q[:, obj, 2])
        lx = normals[:, 0] * (hs + r) - normals[:, 1] * offset[:, None]
        ly = normals[:, 1] * (hs + r) + normals[:, 0] * offset[:, None]
        p0x, p0y = q[:, obj, 0] + c0 * lx - s0 * ly, q[:, obj, 1] + s0 * lx + c0 * ly
        step = (length / T)[:, None]
        ddx, ddy = -(c0 * normals[:, 0] - s0 * normals[:, 1]) * step, -(s0 * normals[:, 0] + c0 * normals[:, 1]) * step
        for j in range(T):
            x, y, vx, vy, om = q[..., 0], q[..., 1], v[..., 0], v[..., 1], v[..., 2]
            c, s = torch.cos(q[..., 2]), torch.sin(q[..., 2])
            px, py = (p0x + (j + 1) * ddx)[:, :, None], (p0y + (j + 1) * ddy)[:, :, None]
            b = lambda t: t[:, None, :]  # noqa: E731
            sd, nx, ny = _square(px, py, b(x), b(y), b(c), b(s), hs)
            rx, ry = px - r * nx - b(x), py - r * ny - b(y)
            fn, gt, tx, ty = contact(r - sd, nx, ny, (ddx / dt)[:, :, None] - (b(vx) - b(om) * ry),
                                     (ddy / dt)[:, :, None] - (b(vy) + b(om) * rx))
            fx, fy = -fn * nx + gt * tx, -fn * ny + gt * ty
            ww = w[:, :, None]
            F = torch.stack([(ww * fx).sum(1), (ww * fy).sum(1), (ww * (rx * fy - ry * fx)).sum(1)], -1)
            if pairs:
                g = lambda t, k: t[:, k]  # noqa: E731
                rlx = g(c, own) * corner[:, 0] - g(s, own) * corner[:, 1]
                rly = g(s, own) * corner[:, 0] + g(c, own) * corner[:, 1]
                kx, ky = g(x, own) + rlx, g(y, own) + rly
                sd, nx, ny = _square(kx, ky, g(x, oth), g(y, oth), g(c, oth), g(s, oth), hs)
                dx, dy = kx - g(x, oth), ky - g(y, oth)
                fn, gt, tx, ty = contact(-sd, nx, ny,
                                         g(vx, own) - g(om, own) * rly - (g(vx, oth) - g(om, oth) * dy),
                                         g(vy, own) + g(om, own) * rlx - (g(vy, oth) + g(om, oth) * dx))
                fx, fy = fn * nx - gt * tx, fn * ny - gt * ty
                F = F.index_add(1, own, torch.stack([fx, fy, rlx * fy - rly * fx], -1))
                F = F.index_add(1, oth, torch.stack([-fx, -fy, -(dx * fy - dy * fx)], -1))
            sv = torch.sqrt(vx * vx + vy * vy + f("eps_v") ** 2)
            so = torch.sqrt(om * om + f("eps_w") ** 2)
            F = F - weight * torch.stack([vx / sv, vy / sv, lever * om / so], -1)
            v = v + dt * F / F.new_tensor([m, m, inertia])
            q = q + dt * v
        return q, v

    q = start.expand(n, nb, 3)
    v = torch.zeros_like(q)
    for k in range(case["H"]):
        q, v = checkpoint(push, q, v, z[:, k], off[:, k], dist[:, k], use_reentrant=False)
    return _cost(q, dist, goal), torch.cat([q, v], -1).reshape(n, 6 * nb)


def _mlp64(net, in_dim, out_dim, x):
    sizes, at, h = [in_dim, HIDDEN, HIDDEN, HIDDEN, out_dim], 0, x
    for l, (i, o) in enumerate(zip(sizes[:-1], sizes[1:])):
        w, b = net[at:at + i * o].reshape(o, i), net[at + i * o:at + i * o + o]
        at += i * o + o
        h = h @ w.T + b
        h = torch.nn.functional.silu(h) if l < 3 else h
    return h


def _median_h(x):
    """Median heuristic: lower median of the squared pair distances over ln(N + 1)."""
    n = x.shape[0]
    d2 = torch.cdist(x, x, compute_mode="donot_use_mm_for_euclid_dist").square()
    i = torch.triu_indices(n, n, 1, device="cuda")
    d = d2[i[0], i[1]]
    return torch.kthvalue(d, (d.numel() - 1) // 2 + 1).values / math.log(n + 1), d2


def _stein64(case, a):
    n, H = case["N"], case["H"]
    M, P, D = _dims(case)
    th, g = a["theta"].double(), a["grad"].double()
    w = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    if case["weighted"]:
        w = torch.softmax(a["hard"].double() - a["relaxed"].double(), 0)
    if not case["structured"]:
        h, d2 = _median_h(th)
        K = torch.exp(-d2 / h) * w[None, :]
        phi = K @ g + (2 / h) * (th * K.sum(1, keepdim=True) - K @ th)
    else:
        t3 = th.reshape(n, H, P)
        sft, uv = torch.softmax(t3[:, :, :M], -1), t3[:, :, M:]
        hc, hz = _median_h(uv.reshape(n, -1))[0] / H, _median_h(sft.reshape(n, -1))[0] / H
        h, K, rep = hc, torch.zeros(n, n, dtype=torch.float64, device="cuda"), torch.zeros_like(t3)
        for k in range(H):
            c, z = uv[:, k], sft[:, k]
            ec = torch.exp(-torch.cdist(c, c, compute_mode="donot_use_mm_for_euclid_dist").square() / hc)
            ez = torch.exp(-torch.cdist(z, z, compute_mode="donot_use_mm_for_euclid_dist").square() / hz)
            K += ec + ez
            rep[:, k, M:] = (2 / hc) * (c * (ec @ w)[:, None] - ec @ (w[:, None] * c))
            x = z[:, None, :] - z[None, :, :]                    # s_i - s_j
            jx = z[None, :, :] * (x - (z[None, :, :] * x).sum(-1, keepdim=True))
            rep[:, k, :M] = (2 / hz) * torch.einsum("ij,ijc->ic", ez * w[None, :], jx)
        phi = ((K * w[None, :]) @ g + rep.reshape(n, D)) / (2 * H)
    m = 0.9 * a["m"].double() - 0.1 * phi
    v = 0.999 * a["v"].double() + 0.001 * phi * phi
    th = th - LR * (m / (1 - 0.9 ** ADAM_STEP)) / (torch.sqrt(v / (1 - 0.999 ** ADAM_STEP)) + 1e-8)
    return {"theta": th, "m": m, "v": v, "h": h.reshape(1), "phi": phi}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("screen", "batch"):
        # a choice among near-equal costs; four iterations of many solves
        return None
    a = _inputs(case, seed)
    if kind == "stein":
        return _stein64(case, a)
    if kind == "mlp_step":
        x = a["x"].double().requires_grad_(True)
        net = a["net"].double().requires_grad_(True)
        y = _mlp64(net, x.shape[1], a["dy"].shape[1], x)
        dx, dp = torch.autograd.grad(y, (x, net), a["dy"].double())
        return {"y": y.detach(), "dx": dx, "dparams": dp}
    start = torch.tensor(np.asarray(a["init"], dtype=np.float32).astype(np.float64), device="cuda")
    theta = a["theta"].double().requires_grad_(True)
    if kind == "rollout":
        start = a["start"].double() if case["each"] else start
        cost, final = _simulate(theta, case, seed, start, a["goal"])
        (g,) = torch.autograd.grad(cost.sum(), theta)
        return {"cost": cost.detach(), "final": final.detach(), "grad": -g}
    z, off, dist = _relax(theta, case, seed, True)
    q, nb, n = start.expand(case["N"], case["nb"], 3), case["nb"], case["N"]
    net = a["net"].double()
    for k in range(case["H"]):
        pose = torch.stack([q[..., 0], q[..., 1], torch.cos(q[..., 2]), torch.sin(q[..., 2])], -1)
        x = torch.cat([pose.reshape(n, -1), z[:, k], (off[:, k] / float(np.float32(PHYSICS["offset_max"])))[:, None],
                       (dist[:, k] / float(np.float32(PHYSICS["dist_max"])))[:, None]], -1)
        q = q + _mlp64(net, 8 * nb + 2, 3 * nb, x).reshape(n, nb, 3)
    cost = _cost(q, dist, a["goal"])
    (g,) = torch.autograd.grad(cost.sum(), theta)
    return {"cost": cost.detach(), "grad": -g}
