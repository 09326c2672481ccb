"""Performance cases of the multiresolution step, through the package's public calls.

Families (a case's "family"):
  restart   a run that restarts from a checkpoint on the host (set_blocks), advances it by full
            multiresolution steps (refine all, RK4, the shock filter where it is on, coarsening rounds) and
            writes the grid and its fields back to the host (get_blocks)
  go-on     an advection run on an equidistant grid (Jmin = Jmax) that goes on from where it stands: full steps,
            then the fields to the host
  network   the refinement proposal's network: forward, loss and gradient on host samples (cnn_eval)

Sizes are those of the benchmark's workloads, of the tests and of the paper's studies (Sec. 3 and 4).
"""
import math
import random

import numpy as np
import torch

import paper_1902_00088_gb300 as mr


def _flow(name, family, rhs, dim, Bs, precision, Jmin, Jmax, eps, steps, **kw):
    c = dict(name=name, family=family, rhs=rhs, dim=dim, Bs=Bs, precision=precision, detail_fp64=False, Jmin=Jmin,
             Jmax=Jmax, eps=eps, steps=steps, ntrees=1, width=0.05, spin=2, eager=False, mu=0.0, filtered=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest run: a 2D pulse on a few tens of 17^2 blocks in plain FP64, host-driven steps
        # (kernel latency, launches and the host's round trips)
        _flow("adv2d-fp64-small", "restart", "adv", 2, 17, "fp64", 2, 5, 1e-3, 12, eager=True),
        # the swirl test of Sec. 3 in the single-precision form: few hundred blocks, captured steps
        _flow("swirl2d-fp32", "restart", "swirl", 2, 17, "fp32", 1, 8, 1e-4, 25, detail_fp64=True,
              width=math.sqrt(0.005), spin=4000),
        # the paper's own study case of the swirl: 33^2 blocks, plain FP64
        _flow("swirl2d-33-fp64", "restart", "swirl", 2, 33, "fp64", 1, 6, 1e-5, 15, width=math.sqrt(0.005), spin=3000),
        # many independent 2D problems advanced together (a parameter sweep)
        _flow("forest-64-trees", "restart", "adv", 2, 17, "fp32", 2, 8, 1e-4, 25, detail_fp64=True, ntrees=64),
        # a 3D pulse in a few hundred 17^3 blocks, the benchmark's default
        _flow("adv3d-fp32", "restart", "adv", 3, 17, "fp32", 2, 6, 1e-4, 20, detail_fp64=True, width=0.04),
        # the same method in plain FP64 with a smaller threshold
        _flow("adv3d-fp64", "restart", "adv", 3, 17, "fp64", 2, 5, 1e-5, 10, width=0.06),
        # equidistant grids (the paper's comparison runs): 2D, 65536 blocks of 17^2 ...
        _flow("fixed2d-fp32", "go-on", "adv", 2, 17, "fp32", 8, 8, 1e-3, 60, detail_fp64=True),
        # ... and 3D, 32768 blocks of 17^3: the largest case
        _flow("fixed3d-fp32", "go-on", "adv", 3, 17, "fp32", 5, 5, 1e-4, 20, detail_fp64=True, width=0.04),
        # Navier-Stokes in flux form: a thin temporal mixing layer on 33^2 blocks, FP32 stages, FP64 state
        _flow("mixing-thin-33", "restart", "ns", 2, 33, "fp32_acc64", 2, 7, 1e-3, 12, width=1.0 / 240.0,
              mu=0.5 / 240.0 / 1000.0, spin=20),
        # Navier-Stokes in the skew-symmetric form with the shock filter (the double shear layer of Sec. 4):
        # early in the run on an adaptive grid ...
        _flow("shear-adaptive", "restart", "ns_skew", 2, 17, "fp32_acc64", 2, 7, 1e-3, 25, width=8.0 / 240.0, mu=1e-6,
              filtered=True, spin=400),
        # ... and the fixed grid that it is compared with, which is also where the adaptive grid ends
        _flow("shear-fixed", "restart", "ns_skew", 2, 17, "fp32_acc64", 7, 7, 1e-3, 20, width=8.0 / 240.0, mu=1e-6,
              filtered=True),
        # training of the proposal network: forward and backward on a few thousand block tiles
        dict(name="network-17", family="network", Bs=17, samples=3000),
    ]


def draw(rng):
    """One more case of the same families and ranges."""
    f = rng.choice(["2d", "2d", "forest", "3d", "fixed2d", "fixed3d", "ns", "ns", "nsfixed", "network"])
    loguni = lambda a, b: math.exp(rng.uniform(math.log(a), math.log(b)))
    form = lambda: rng.choice([("fp32", True), ("fp32", False), ("fp64", False), ("fp32_acc64", False)])
    eps = float("%.3g" % loguni(1e-5, 1e-3))
    steps = rng.randint(5, 25)
    if f == "network":
        c = dict(family="network", Bs=rng.choice([17, 33]), samples=int(loguni(7, 4500)))
    elif f in ("2d", "forest"):
        p, d64 = form()
        rhs = "adv" if f == "forest" else rng.choice(["adv", "swirl"])
        B = rng.choice([17, 17, 33])
        c = _flow("", "restart", rhs, 2, B, p, 2 if f == "forest" else rng.randint(1, 3),
                  rng.randint(4, 8 if B == 17 else 7), eps, steps, detail_fp64=d64,
                  ntrees=int(loguni(2, 100)) if f == "forest" else 1, width=rng.uniform(0.03, 0.1),
                  spin=rng.randint(2, 300), eager=rng.random() < 0.2)
    elif f == "3d":
        p, d64 = form()
        c = _flow("", "restart", "adv", 3, 17, p, rng.randint(1, 2), rng.randint(3, 6 if p == "fp32" else 5),
                  max(eps, 2e-5), rng.randint(4, 15), detail_fp64=d64, width=rng.uniform(0.04, 0.1),
                  spin=rng.randint(2, 20))
    elif f == "fixed2d":
        p, d64 = form()
        J = rng.randint(3, 8)
        c = _flow("", "go-on", rng.choice(["adv", "swirl"]), 2, 17 if J == 8 else rng.choice([17, 33]), p, J, J, eps,
                  rng.randint(5, 40), detail_fp64=d64, width=rng.uniform(0.04, 0.1))
    elif f == "fixed3d":
        p, d64 = form()
        J = rng.randint(2, 4)
        c = _flow("", "go-on", "adv", 3, 17, p, J, J, eps, rng.randint(3, 20), detail_fp64=d64,
                  width=rng.uniform(0.04, 0.1))
    else:
        B = rng.choice([17, 33])
        skew = rng.random() < 0.6
        p = rng.choice(["fp32_acc64", "fp32_acc64", "fp32", "fp64"])
        J = rng.randint(4, 6 if p == "fp64" or B == 33 else 7)
        fixed = f == "nsfixed"
        if fixed:
            J = min(J, 5 if B == 33 else 6)
        c = _flow("", "restart", "ns_skew" if skew else "ns", 2, B, p, J if fixed else 2, J,
                  1e-3, rng.randint(4, 15), spin=2 if fixed else rng.randint(2, 100),
                  width=loguni(1.0 / 240.0, 0.1), mu=2e-6)
        if skew:  # without the filter only a layer that the grid resolves
            c.update(filtered=rng.random() < 0.7, mu=1e-6)
            c["width"] = 8.0 / 240.0 if c["filtered"] else 8.0 / 30.0
    c.pop("name", None)
    return c


# --------------------------------------------------------------------------- inputs
def _trees(case, seed):
    """Tree descriptions: initial fields and parameters from the seed."""
    r = random.Random(seed * 7919 + 13)
    out = []
    for k in range(case["ntrees"]):
        t = dict(Jmin=case["Jmin"], Jmax=case["Jmax"], eps=case["eps"])
        if case["rhs"] in ("adv", "swirl"):
            sigma = case["width"]
            c = [r.random(), r.random(), r.random() if case["dim"] == 3 else 0.0]
            if case["rhs"] == "swirl":  # the blob of Sec. 3, shifted a little
                c[0], c[1] = 0.5 + r.uniform(-0.02, 0.02), 0.75 + r.uniform(-0.02, 0.02)
                t["rhs_params"] = (5.0,)
            elif case["ntrees"] > 1:  # a sweep: widths, velocities, levels and thresholds differ
                sigma = r.uniform(0.02, 0.1)
                t["Jmax"] = r.randint(min(4, case["Jmax"]), case["Jmax"])
                t["eps"] = 10.0 ** r.uniform(-5.0, -3.0)
                t["rhs_params"] = (r.uniform(-1.0, 1.0), r.uniform(-1.0, 1.0), 0.0)
            else:
                t["rhs_params"] = (r.uniform(0.5, 1.0), r.uniform(-1.0, 1.0),
                                   r.uniform(0.5, 1.0) if case["dim"] == 3 else 0.0)
            t.update(ic="gauss", ic_params=(c[0], c[1], c[2], sigma))
        elif case["rhs"] == "ns":  # temporal mixing layer, mirrored so that it is periodic
            a = [r.uniform(-1.0, 1.0) for _ in range(8)]
            phi = [r.uniform(0.0, 2.0 * math.pi) for _ in range(8)]
            t.update(ic="mixing", ic_params=(case["width"], 0.5, 0.3, 1.4, 1e-3) + tuple(a) + tuple(phi),
                     rhs_params=(1.4, case["mu"], 0.71, 1e-5 if case["filtered"] else 0.0), x0=(0.0, -0.5, 0.0))
        else:  # double shear layer of Sec. 4 (L = 8)
            t.update(ic="shear_layer", ic_params=(2.0, 1.0, 1.0, -1.0, case["width"], 2.5, r.uniform(0.08, 0.12), 0.25,
                                                  4.0, r.uniform(0.0, 8.0)),
                     rhs_params=(1.4, case["mu"], 0.71, 1e-5 if case["filtered"] else 0.0))
        out.append(t)
    return out


def _domain(case):
    return 8.0 if case["rhs"] == "ns_skew" else 1.0


def _dts(case, trees):
    """CFL 0.5 with the fastest signal of each tree on its finest level."""
    out = []
    for t in trees:
        if case["rhs"] == "adv":
            u = math.sqrt(sum(v * v for v in t["rhs_params"][:3])) or 1.0
        else:
            u = {"swirl": 1.0, "ns": 0.5 + 0.5 / 0.3, "ns_skew": 1.0 + math.sqrt(1.4 * 2.5)}[case["rhs"]]
        out.append(0.5 * _domain(case) / ((case["Bs"] - 1) << t["Jmax"]) / u)
    return np.array(out)


def _capacity(case):
    if case["Jmin"] == case["Jmax"]:
        return (1 << (case["dim"] * case["Jmax"])) + 64
    if case["dim"] == 3:
        return 30_000
    if case["ntrees"] > 1:
        return 600_000 if case["Bs"] == 17 else 200_000
    return 60_000


def _room(case):
    """Blocks that the program's host buffers hold: the whole grid, or what an adaptive one can reach here."""
    full = case["ntrees"] << (case["dim"] * case["Jmax"])
    if case["Jmin"] == case["Jmax"]:
        return full
    return min(full, 3000 if case["dim"] == 3 else 20_000 if case["ntrees"] > 1 else 6000)


def _pinned(shape, dtype):
    return torch.zeros(shape, dtype=dtype, pin_memory=True).numpy()


def prepare(case, seed):
    if case["family"] == "network":
        g = torch.Generator().manual_seed(seed)
        T = case["Bs"] + 8
        n = case["samples"]
        f = mr.Forest(dim=2, Bs=case["Bs"], precision="fp32", rhs="adv", capacity=64,
                      trees=[dict(Jmin=1, Jmax=2, eps=1e-3, ic="gauss", ic_params=(0.5, 0.5, 0.0, 0.1),
                                  rhs_params=(1.0, 0.0, 0.0))])
        # channel 0: a field's deviation from its centre value over the largest one; channel 1: log10 details
        x = torch.empty(n, 2, T, T)
        x[:, 0] = torch.rand(n, T, T, generator=g) * 2 - 1
        x[:, 1] = torch.rand(n, T, T, generator=g) * 3 - 3
        y = (torch.rand(n, generator=g) < 0.1).float()
        w = []
        for k, s in enumerate(mr.Forest.CNN_SHAPES):
            m = int(np.prod(s))
            if len(s) == 4:
                w.append(torch.randn(m, generator=g) * math.sqrt(2.0 / (s[1] * 9)))
            elif k == 6:
                w.append(torch.randn(m, generator=g) * 0.25)
            else:
                w.append(torch.randn(m, generator=g) * 0.05)
        return dict(case=case, g=f, params=torch.cat(w).numpy(), x=x.numpy(), y=y.numpy())
    trees = _trees(case, seed)
    ns = case["rhs"] in ("ns", "ns_skew")
    g = mr.Forest(dim=case["dim"], Bs=case["Bs"], nvar=4 if ns else 1, precision=case["precision"],
                  detail_fp64=case["detail_fp64"], rhs=case["rhs"], trees=trees, capacity=_capacity(case),
                  norm_kind=1 if ns else 0, L=_domain(case))
    dts = _dts(case, trees)
    t = np.zeros(case["ntrees"])
    g.init_tree()
    g.set_time(t, dts)
    g.step_graph(case["spin"])
    t = t + case["spin"] * dts
    s = dict(case=case, g=g, t=t, dts=dts)
    room = _room(case)
    per = (4 if ns else 1) * case["Bs"] ** case["dim"]
    s["info"] = _pinned((room * mr.BLOCK_INFO_DTYPE.itemsize,), torch.uint8).view(mr.BLOCK_INFO_DTYPE)
    s["fields"] = _pinned((room * per,), torch.float64).reshape((room, 4 if ns else 1) + (case["Bs"],) * case["dim"])
    if case["family"] == "restart":  # the checkpoint that every pass starts from
        info, f = g.get_blocks(out=(s["info"], s["fields"]))
        s["start"] = (info["level"].copy(), info["coords"].copy(), info["tree"].copy())
        s["start_fields"] = _pinned(f.shape, torch.float64)
        s["start_fields"][:] = f
    return s


# ----------------------------------------------------------------------------- pass
def run(s):
    case, g = s["case"], s["g"]
    if case["family"] == "network":
        prob, grad, loss = g.cnn_eval(s["params"], s["x"], s["y"], w_pos=4.0)
        return dict(prob=prob, grad=grad, loss=float(loss))
    if case["family"] == "restart":
        level, coords, tree = s["start"]
        g.set_blocks(level, coords, s["start_fields"], tree=tree)
        if case["eager"]:
            t = s["t"]
            for _ in range(case["steps"]):
                g.step(t, s["dts"])
                t = t + s["dts"]
        else:
            g.set_time(s["t"], s["dts"])
            g.step_graph(case["steps"])
    else:
        g.step_graph(case["steps"])
    info, _ = g.get_blocks(out=(s["info"], s["fields"]))
    # the program's own buffers; the first n blocks are this pass's
    b = s["info"]
    return dict(n=len(info), level=b["level"], tree=b["tree"], coords=b["coords"], fields=s["fields"])


# ----------------------------------------------------------------------------- work
def work(case):
    """Each step reads the state of the grid that it evolves (all blocks refined for safety) once and writes it
    once; the checkpoint and the result cross once more as doubles.  Operations: four RK stages over that grid."""
    if case["family"] == "network":
        T = case["Bs"] + 8
        T2 = (T - 1) // 2 + 1
        T3 = (T2 - 1) // 2 + 1
        mac = 16 * 9 * (2 * T * T + 16 * T2 * T2 + 16 * T3 * T3)
        return dict(bytes=case["samples"] * (2 * T * T + 2) * 4 + 2 * 4961 * 4, flops=case["samples"] * 3 * 2 * mac)
    ns = case["rhs"] in ("ns", "ns_skew")
    pts = case["Bs"] ** case["dim"]
    vals = pts * (4 if ns else 1)
    size = 4 if case["precision"] == "fp32" else 8
    ops = {"adv": 7 * case["dim"] + 3, "swirl": 21, "ns": 160, "ns_skew": 230}[case["rhs"]] + 6 * (4 if ns else 1)
    if case["Jmin"] == case["Jmax"]:
        n = 1 << (case["dim"] * case["Jmax"])
        return dict(bytes=case["steps"] * n * vals * 2 * size + n * vals * 8, flops=case["steps"] * 4 * n * pts * ops)
    # adaptive: the blocks advanced by these steps, counted on the device
    s = prepare(case, 1)
    s["g"].reset_stats()
    out = run(s)
    advanced = s["g"].stats()["stage_blocks"] / 4
    n = out["n"] + len(s["start"][0])
    return dict(bytes=advanced * vals * 2 * size + n * vals * 8, flops=advanced * 4 * pts * ops)


# ---------------------------------------------------------------------------- exact
def _hilbert(cells, bits):
    """Hilbert index of integer cells (n x d) by J. Skilling's transform (AIP Conf. Proc. 707, 381)."""
    X = [cells[:, a].astype(np.int64).copy() for a in range(cells.shape[1])]
    d = len(X)
    q = 1 << (bits - 1)
    while q > 1:
        p = q - 1
        for i in range(d):
            on = (X[i] & q) != 0
            t = np.where(on, 0, (X[0] ^ X[i]) & p)
            X[0] = np.where(on, X[0] ^ p, X[0] ^ t)
            X[i] = X[i] ^ t if i else X[0]
        q >>= 1
    for i in range(1, d):
        X[i] = X[i] ^ X[i - 1]
    t = np.zeros_like(X[0])
    q = 1 << (bits - 1)
    while q > 1:
        t = np.where((X[d - 1] & q) != 0, t ^ (q - 1), t)
        q >>= 1
    for i in range(d):
        X[i] = X[i] ^ t
    h = np.zeros_like(X[0])
    for b in range(bits - 1, -1, -1):
        for i in range(d):
            h = (h << 1) | ((X[i] >> b) & 1)
    return h


def _blocks_of(grid, B, J):
    """Blocks, in Hilbert order, of a periodic node grid (nvar, [z,] y, x)."""
    d = grid.dim() - 1
    n = 1 << J
    ax = np.meshgrid(*([np.arange(n)] * d), indexing="ij")
    c = np.stack([a.ravel() for a in ax[::-1]], 1)  # x, y[, z]
    c = c[np.argsort(_hilbert(c, J), kind="stable")]
    out = torch.empty((len(c), grid.shape[0]) + (B,) * d, dtype=grid.dtype, device=grid.device)
    N = grid.shape[-1]
    i = torch.arange(B, device=grid.device)
    cc = torch.from_numpy(c).to(grid.device)
    for k in range(0, len(c), 2048):
        q = cc[k:k + 2048]
        ix = (q[:, 0, None] * (B - 1) + i) % N
        iy = (q[:, 1, None] * (B - 1) + i) % N
        if d == 2:
            out[k:k + 2048] = grid[:, iy[:, :, None], ix[:, None, :]].transpose(0, 1)
        else:
            iz = (q[:, 2, None] * (B - 1) + i) % N
            out[k:k + 2048] = grid[:, iz[:, :, None, None], iy[:, None, :, None], ix[:, None, None, :]].transpose(0, 1)
    return out


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["family"] == "network":
        s = prepare(case, seed)
        x = torch.from_numpy(s["x"]).to(dev).double()
        y = torch.from_numpy(s["y"]).to(dev).double()
        p, w, o = torch.from_numpy(s["params"]).to(dev).double().requires_grad_(), [], 0
        for sh in mr.Forest.CNN_SHAPES:
            m = int(np.prod(sh))
            w.append(p[o:o + m].reshape(sh))
            o += m
        conv = torch.nn.functional.conv2d
        h = torch.relu(conv(x, w[0], w[1], padding=1))
        h = torch.relu(conv(h, w[2], w[3], stride=2, padding=1))
        h = torch.relu(conv(h, w[4], w[5], stride=2, padding=1))
        z = h.amax((2, 3)) @ w[6] + w[7]
        prob = torch.sigmoid(z)
        ls = torch.nn.functional.logsigmoid
        loss = -(4.0 * y * ls(z) + (1 - y) * ls(-z)).mean()
        loss.backward()
        return dict(prob=prob.detach(), grad=p.grad, loss=loss.detach())
    if case["Jmin"] != case["Jmax"] or case["rhs"] == "ns":
        return None  # an adaptive grid's evolution has no short closed form
    t0 = _trees(case, seed)[0]
    dt = float(_dts(case, [t0])[0])
    B, J, d, L = case["Bs"], case["Jmax"], case["dim"], _domain(case)
    N = (B - 1) << J
    h = L / N
    x = torch.arange(N, dtype=torch.float64, device=dev) * h
    total = case["spin"] + case["steps"]

    def dif(f, a):  # 4th-order central difference along axis -1 - a
        r = lambda k: torch.roll(f, -k, -1 - a)
        return ((r(-2) - r(2)) + 8.0 * (r(1) - r(-1))) / (12.0 * h)

    if case["rhs"] in ("adv", "swirl"):
        f = None
        for a in range(d):
            r = x - t0["ic_params"][a]
            r = r - L * torch.floor(r / L + 0.5)
            e = torch.exp(-r * r / (2 * t0["ic_params"][3] ** 2)).reshape([-1] + [1] * a)
            f = e if f is None else f * e
        q = f.expand([N] * d).clone()[None]
        if case["rhs"] == "adv":
            u = t0["rhs_params"]

            def rate(q, t):
                k = -u[0] * dif(q, 0) - u[1] * dif(q, 1)
                return k - u[2] * dif(q, 2) if d == 3 else k
        else:
            A, S = torch.sin(math.pi * x) ** 2, torch.sin(2 * math.pi * x)

            def rate(q, t):
                ct = math.cos(math.pi * t / t0["rhs_params"][0])
                return -(ct * A[None, :] * S[:, None]) * dif(q, 0) + (ct * A[:, None] * S[None, :]) * dif(q, 1)
    else:  # skew-symmetric Navier-Stokes on (sqrt(rho), sqrt(rho) u, sqrt(rho) v, p)
        rho1, rho0, v1, v0, lw, p0, amp, hw, xc, yc = t0["ic_params"]
        gam, mu, Pr, rth = t0["rhs_params"]
        kap = mu * gam / ((gam - 1.0) * Pr)
        prof = (0.5 * (torch.tanh((x - (xc - hw)) / lw) - torch.tanh((x - (xc + hw)) / lw)))[None, :]
        rho = (rho0 + (rho1 - rho0) * prof).expand(N, N)
        u = (amp * torch.sin(2 * math.pi * (x - yc)))[:, None].expand(N, N)
        v = (v0 + (v1 - v0) * prof).expand(N, N)
        q = torch.stack([rho.sqrt(), rho.sqrt() * u, rho.sqrt() * v, torch.full_like(rho, p0)])

        def rate(q, t):
            f, sx, sy, p = q
            u, v, th = sx / f, sy / f, p / (f * f)
            ux, uy, vx, vy = dif(u, 0), dif(u, 1), dif(v, 0), dif(v, 1)
            txx, tyy = mu * (2 * ux - 2 / 3 * (ux + vy)), mu * (2 * vy - 2 / 3 * (ux + vy))
            txy = mu * (uy + vx)
            px, py = dif(p, 0), dif(p, 1)
            k0 = -0.5 * (dif(sx, 0) + u * dif(f, 0) + dif(sy, 1) + v * dif(f, 1))
            con = lambda m: dif(m * u, 0) + u * dif(m, 0) + dif(m * v, 1) + v * dif(m, 1)
            k1 = -0.5 * con(sx) - (px - dif(txx, 0) - dif(txy, 1)) / f
            k2 = -0.5 * con(sy) - (py - dif(txy, 0) - dif(tyy, 1)) / f
            heat = dif(kap * dif(th, 0), 0) + dif(kap * dif(th, 1), 1)
            k3 = (-gam * (dif(p * u, 0) + dif(p * v, 1)) + (gam - 1) * (u * px + v * py)
                  + (gam - 1) * (txx * ux + txy * (uy + vx) + tyy * vy + heat))
            return torch.stack([k0, k1, k2, k3])

        def shock_filter(q):
            f, sx, sy, p = q
            r = lambda g, k, a: torch.roll(g, -k, -1 - a)
            u, v = sx / f, sy / f
            th = (r(u, 1, 0) - r(u, -1, 0)) / (2 * h) + (r(v, 1, 1) - r(v, -1, 1)) / (2 * h)
            c2 = gam * p / (f * f)
            out = q
            for a in (0, 1):
                D = (-r(th, 1, a) + 2 * th - r(th, -1, a)) / 4
                M = ((D - r(D, 1, a)) ** 2 + (D - r(D, -1, a)) ** 2) / 2
                s = torch.clamp(1 - rth / (M / (c2 / (h * h)) + 1e-16), min=0.0)
                flux = 0.5 * (s + r(s, 1, a)) * (-0.25) * (r(q, 1, a) - q)
                out = out - (flux - r(flux, -1, a))
            return out
    t = 0.0
    for _ in range(total):
        k = rate(q, t)
        acc = q + dt / 6 * k
        k = rate(q + dt / 2 * k, t + dt / 2)
        acc = acc + dt / 3 * k
        k = rate(q + dt / 2 * k, t + dt / 2)
        acc = acc + dt / 3 * k
        q = acc + dt / 6 * rate(q + dt * k, t + dt)
        if case["filtered"]:
            q = shock_filter(q)
        t += dt
    return dict(n=None, level=None, tree=None, coords=None, fields=_blocks_of(q, B, J))
