"""What this framework is used for, as calls that can be timed: the l1-ball
projection, whole solves of Algorithm 1 (float32 and 16-bit iterates, from
device and from host memory), a batch of uneven cubes, the unrolled solve with
its gradient, and one transposed pass.

A case is a dict of plain values; prepare() makes the inputs from a seed and
the handle a user's program keeps, run() is one call through the public entry
points, work() the bytes and operations that call cannot do without, exact()
the same result in float64 by plain torch.
"""
import math

import numpy as np
import torch

from paper_2510_00562_gb300.autograd import unrolled_geosstv
from paper_2510_00562_gb300.solver import (GRAD_PARAMS, STATE_KEYS, STATE_LEAD, GeoSSTVBatch, GeoSSTVSolver,
                                           make_params, project_l1ball)

SIDES = (32, 48, 96, 128, 256)          # spatial sides and band counts of the uneven batch
BANDS = (31, 64, 128)


def listed():
    return [
        # the projection as an operator of its own: a small vector (a call that
        # is all latency) and one the size of the largest cube
        {"name": "project_4096", "kind": "project", "n": 4096},
        {"name": "project_58m", "kind": "project", "n": 512 * 512 * 224},
        # a patch-sized cube
        {"name": "solve_64x64x32", "kind": "solve", "n1": 64, "n2": 64, "n3": 32, "passes": 200, "storage": "fp32",
         "tol": 0.0},
        # a scene cropped to odd sides, with the stopping rule on (it does not
        # stop within the cap)
        {"name": "solve_157x203x61_tol", "kind": "solve", "n1": 157, "n2": 203, "n3": 61, "passes": 100,
         "storage": "fp32", "tol": 1e-7},
        {"name": "solve_128x128x64", "kind": "solve", "n1": 128, "n2": 128, "n3": 64, "passes": 200,
         "storage": "fp32", "tol": 0.0},
        # scenes of the usual benchmark size
        {"name": "solve_256x256x128", "kind": "solve", "n1": 256, "n2": 256, "n3": 128, "passes": 100,
         "storage": "fp32", "tol": 0.0},
        # the largest scene, end to end from pinned host memory
        {"name": "host_512x512x224", "kind": "host", "n1": 512, "n2": 512, "n3": 224, "passes": 40,
         "storage": "fp32", "tol": 0.0},
        # the 16-bit phase of the precision form
        {"name": "solve_bf16_512x512x224", "kind": "solve", "n1": 512, "n2": 512, "n3": 224, "passes": 16,
         "storage": "bf16", "tol": 0.0},
        {"name": "solve_fp16_256x256x200", "kind": "solve", "n1": 256, "n2": 256, "n3": 200, "passes": 32,
         "storage": "fp16", "tol": 0.0},
        # many scenes at once
        {"name": "batch_8_uneven", "kind": "batch", "passes": 64,
         "cubes": "32x48x31,96x128x64,128x32x128,256x96x64,48x256x31,128x128x128,256x256x64,96x96x31"},
        # learning the radii: an unrolled solve and its gradient
        {"name": "grad_128x128x64", "kind": "grad", "n1": 128, "n2": 128, "n3": 64, "passes": 40, "ckpt": 0},
        # the transpose of one pass, as a reverse mode of a user's own calls it
        {"name": "vjp_512x256x64", "kind": "vjp", "n1": 512, "n2": 256, "n3": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["project", "project", "solve", "solve", "solve", "solve16", "host", "batch", "grad", "vjp"])
    if kind == "project":
        return {"kind": "project", "n": _log_int(rng, 256, 56_000_000)}
    if kind == "batch":
        cubes = ",".join("%dx%dx%d" % (rng.choice(SIDES), rng.choice(SIDES), rng.choice(BANDS))
                         for _ in range(rng.randint(2, 12)))
        return {"kind": "batch", "passes": rng.choice([32, 48, 50, 64]), "cubes": cubes}
    top = {"solve": 12_000_000, "solve16": 20_000_000, "host": 20_000_000, "grad": 2_000_000, "vjp": 12_000_000}[kind]
    low = {"host": 1_000_000, "solve16": 500_000}.get(kind, 30_000)
    n = math.exp(rng.uniform(math.log(low), math.log(top)))
    # sides about as unequal as scenes are: bands a quarter to all of the mean side
    side = n ** (1.0 / 3.0)
    n3 = max(4, int(side * rng.uniform(0.35, 1.2)))
    n1 = max(8, int(math.sqrt(n / n3) * rng.uniform(0.7, 1.4)))
    n2 = max(8, int(n / n3 / n1))
    if rng.random() < 0.4:
        n1, n2 = (n1 + 7) // 8 * 8, (n2 + 7) // 8 * 8
    c = {"kind": kind if kind != "solve16" else "solve", "n1": n1, "n2": n2, "n3": n3}
    if kind == "vjp":
        return c
    if kind == "grad":
        return dict(c, passes=rng.randint(8, 40), ckpt=rng.choice([0, 0, 1]))
    small = n1 * n2 * n3 < 2_000_000
    c["passes"] = rng.randint(50, 200) if small else rng.randint(16, 60)
    c["storage"] = rng.choice(["bf16", "fp16"]) if kind == "solve16" else "fp32"
    if kind == "solve16":
        c["passes"] = rng.randint(12, 32)
    c["tol"] = rng.choice([0.0, 0.0, 1e-7])
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _problem(n1, n2, n3, seed):
    """An observation with Gaussian noise, salt and pepper and stripes over a
    piecewise-smooth scene, and the radii of the constraints."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    h = np.random.default_rng(seed)
    sigma, sp_rate, stripe_rate, amp = 0.1, 0.05, 0.05, 0.25
    # Voronoi regions with spectra of three Gaussians each
    at = h.uniform(size=(6, 2)) * np.array([n1, n2])
    band = np.arange(n3)
    spectra = np.zeros((6, n3))
    for r in range(6):
        for _ in range(3):
            c, w, a = h.uniform(0, n3), h.uniform(n3 / 12, n3 / 3), h.uniform(0.2, 1)
            spectra[r] += a * np.exp(-0.5 * ((band - c) / w) ** 2)
    spectra = (spectra - spectra.min()) / max(spectra.max() - spectra.min(), 1e-9)
    ii = torch.arange(n1, device="cuda")[:, None] + 0.5
    jj = torch.arange(n2, device="cuda")[None, :] + 0.5
    d2 = torch.stack([(ii - float(a)) ** 2 + (jj - float(b)) ** 2 for a, b in at])
    clean = torch.from_numpy(spectra.T.astype(np.float32)).cuda()[:, d2.argmin(0)]
    rand = lambda *s: torch.rand(*s, device="cuda", generator=g)  # noqa: E731
    t = torch.where(rand(n3, 1, n2) < stripe_rate, (rand(n3, 1, n2) - 0.5) * 2 * amp, torch.zeros(1, device="cuda"))
    v = clean + t
    v += sigma * torch.randn(n3, n1, n2, device="cuda", generator=g)
    k = rand(n3, n1, n2)
    sp = k < sp_rate
    val = (k < 0.5 * sp_rate).float()
    alpha = 0.9 * float(((val - clean - t).abs() * sp).sum(dtype=torch.float64))
    beta = 0.9 * n1 * float(t.abs().sum(dtype=torch.float64))
    v = torch.where(sp, val, v).contiguous()
    eps = 0.95 * sigma * math.sqrt(n1 * n2 * n3 * (1 - sp_rate))
    return v, dict(eps=eps, alpha=alpha, beta=beta)


def _state(n1, n2, n3, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (n3, n1, n2)
    st = {k: 0.1 * torch.randn(STATE_LEAD[k] + shape, device="cuda", generator=g) for k in STATE_KEYS}
    st["u"] = torch.rand(shape, device="cuda", generator=g) * 1.2 - 0.1
    return st


def _shapes(case):
    return [tuple(int(x) for x in c.split("x")) for c in case["cubes"].split(",")]


def _vector(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = case["n"]
    # the residual of an observation: mostly Gaussian, a few large outliers
    x = 0.1 * torch.randn(n, device="cuda", generator=g)
    x = torch.where(torch.rand(n, device="cuda", generator=g) < 0.05, x + 0.6, x)
    return x, 0.25 * float(x.abs().sum(dtype=torch.float64))


def _params(case, radii):
    return make_params(max_iter=case["passes"], tol=case.get("tol", 0.0), check_every=25,
                       storage=case.get("storage", "fp32"), **radii)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "project":
        x, r = _vector(case, seed)
        return {"kind": kind, "x": x, "r": r}
    if kind == "batch":
        got = [_problem(*s, seed + 101 * k) for k, s in enumerate(_shapes(case))]
        prm = [make_params(max_iter=case["passes"], **r) for _, r in got]
        return {"kind": kind, "v": [v for v, _ in got], "batch": GeoSSTVBatch(_shapes(case), prm)}
    n1, n2, n3 = case["n1"], case["n2"], case["n3"]
    v, radii = _problem(n1, n2, n3, seed)
    if kind == "grad":
        target = _problem(n1, n2, n3, seed + 1)[0]
        return {"kind": kind, "v": v.requires_grad_(), "radii": {k: torch.tensor(x, dtype=torch.float64, requires_grad=True)
                                                                 for k, x in dict(radii, omega=0.03).items()},
                "target": target, "passes": case["passes"], "ckpt": case["ckpt"],
                "solver": GeoSSTVSolver(n1, n2, n3, make_params(max_iter=case["passes"], **radii))}
    if kind == "vjp":
        sol = GeoSSTVSolver(n1, n2, n3, make_params(max_iter=1, **_vjp_radii(n1 * n2 * n3)))
        x = _state(n1, n2, n3, seed + 7)
        sol.load(v, reset=False)
        sol.set_state(x)
        sol.iterate(1)
        return {"kind": kind, "x": x, "x1": sol.get_state(), "bar": _state(n1, n2, n3, seed + 8), "solver": sol}
    sol = GeoSSTVSolver(n1, n2, n3, _params(case, radii))
    if kind == "host":
        pin = lambda: torch.empty((n3, n1, n2), dtype=torch.float32, pin_memory=True)  # noqa: E731
        hv = pin()
        hv.copy_(v)
        return {"kind": kind, "solver": sol, "v": hv, "out": [pin(), pin(), pin()]}
    return {"kind": kind, "solver": sol, "v": v}


def _vjp_radii(n):
    # radii at which both l1 balls and the l2 ball are active for a random state
    return dict(eps=0.2 * math.sqrt(n), alpha=0.05 * n, beta=0.05 * n)


def run(state):
    kind = state["kind"]
    if kind == "project":
        out, tau = project_l1ball(state["x"], state["r"])
        return {"out": out, "tau": tau}
    if kind == "batch":
        u, s, t, done = state["batch"].solve(state["v"])
        return {"u": u, "s": s, "t": t, "passes": done}
    if kind == "grad":
        v, r = state["v"], state["radii"]
        u = unrolled_geosstv(v, r["eps"], r["alpha"], r["beta"], r["omega"], iters=state["passes"],
                             solver=state["solver"], ckpt_every=state["ckpt"])
        loss = ((u - state["target"]) ** 2).mean()
        grads = torch.autograd.grad(loss, [v] + [r[k] for k in GRAD_PARAMS])
        return {"u": u.detach(), "v_bar": grads[0], **{k: g for k, g in zip(GRAD_PARAMS, grads[1:])}}
    if kind == "vjp":
        bar, vbar, pbar = state["solver"].vjp_step(state["x"], state["x1"], state["bar"])
        return {"bar": bar, "v_bar": vbar, "params": pbar}
    if kind == "host":
        u, s, t = state["out"]
        n = state["solver"].solve_host(state["v"], u, s, t)
        return {"u": u, "s": s, "t": t, "passes": n}
    u, s, t, n = state["solver"].solve(state["v"])
    return {"u": u, "s": s, "t": t, "passes": n}


def work(case):
    """A pass of Algorithm 1 reads and writes its 21 state cubes once and reads
    v; its transpose reads the state and the adjoint, writes the adjoint, reads
    v and adds to the adjoint of v.  About 300 operations a voxel and pass."""
    kind = case["kind"]
    if kind == "project":
        return {"bytes": 8 * case["n"], "flops": 4 * case["n"]}
    if kind == "batch":
        n = sum(a * b * c for a, b, c in _shapes(case)) * case["passes"]
        return {"bytes": 43 * 4 * n, "flops": 300 * n}
    n = case["n1"] * case["n2"] * case["n3"]
    if kind == "vjp":
        return {"bytes": 4 * n * (21 + 6 + 42 + 2), "flops": 400 * n}
    if kind == "grad":
        return {"bytes": 4 * n * (43 + 66) * case["passes"], "flops": 700 * n * case["passes"]}
    word = 4 if case["storage"] == "fp32" else 2
    return {"bytes": (42 * word + 4) * n * case["passes"], "flops": 300 * n * case["passes"]}


# ---------------------------------------------------------------------------
# the same in float64
# ---------------------------------------------------------------------------
GU, GW, GS, GT, GY = 1 / 13, 0.25, 1.0, 1 / 3, 0.2          # the default step sizes


def _d(x, axis):
    return torch.cat([x.diff(dim=axis), torch.zeros_like(x.narrow(axis, 0, 1))], axis)


def _dt(y, axis):
    z = y.narrow(axis, 0, y.shape[axis] - 1)
    zero = torch.zeros_like(y.narrow(axis, 0, 1))
    return torch.cat([zero, z], axis) - torch.cat([z, zero], axis)


def _shift(x, di, dj):
    """x[..., i + di, j + dj], zero outside."""
    n1, n2 = x.shape[-2:]
    p = torch.nn.functional.pad(x, (max(0, -dj), max(0, dj), max(0, -di), max(0, di)))
    return p[..., max(0, di):max(0, di) + n1, max(0, dj):max(0, dj) + n2]


def _masks(x):
    mv, mh = torch.ones_like(x[0, :, :1]), torch.ones_like(x[0, :1, :])
    mv[-1], mh[:, -1] = 0, 0
    return mv, mh


def _L(yv, yh):
    mv, mh = _masks(yv)
    yv, yh = mv * yv, mh * yh
    return [yv, mv * 0.25 * (yh + _shift(yh, 0, -1) + _shift(yh, 1, 0) + _shift(yh, 1, -1)),
            mh * 0.25 * (yv + _shift(yv, -1, 0) + _shift(yv, 0, 1) + _shift(yv, -1, 1)), yh,
            0.5 * (yv + _shift(yv, -1, 0)), 0.5 * (yh + _shift(yh, 0, -1))]


def _Lt(w):
    mv, mh = _masks(w[0])
    a, b = mv * w[1], mh * w[2]
    gv = w[0] + 0.25 * (b + _shift(b, 1, 0) + _shift(b, 0, -1) + _shift(b, 1, -1)) + 0.5 * (w[4] + _shift(w[4], 1, 0))
    gh = w[3] + 0.25 * (a + _shift(a, 0, 1) + _shift(a, -1, 0) + _shift(a, -1, 1)) + 0.5 * (w[5] + _shift(w[5], 0, 1))
    return mv * gv, mh * gh


def _shrink(w, thr):
    out = []
    for k in (0, 2, 4):
        n2 = w[k] ** 2 + w[k + 1] ** 2
        on = n2 > thr * thr
        f = torch.where(on, 1 - thr / torch.sqrt(torch.where(on, n2, torch.ones_like(n2))), torch.zeros_like(n2))
        out += [f * w[k], f * w[k + 1]]
    return out


def _l1ball(x, r):
    """The projection, differentiable in x and r; returns (projection, tau)."""
    with torch.no_grad():
        a = x.detach().abs().flatten()
        if float(a.sum()) <= float(r):
            tau = None
        else:
            srt = a.sort(descending=True).values
            cs = srt.cumsum(0)
            on = srt - (cs - float(r)) / torch.arange(1, srt.numel() + 1, device=x.device) > 0
            m = int(on.sum())
            tau = float((cs[m - 1] - float(r)) / m)
            del srt, cs, on
    if tau is None:
        return x, 0.0
    if x.requires_grad or isinstance(r, torch.Tensor):
        on = x.detach().abs() > tau
        tau = ((x.abs() * on).sum() - r) / on.sum()
    return x.sign() * (x.abs() - tau).clamp_min(0), tau


def _box(x):
    return torch.where((x > 0) & (x < 1), x, x.detach().clamp(0, 1))


def _pass(st, v, p):
    """One pass of Algorithm 1 on float64 cubes."""
    u, s, t, w1, w2, y1, y2, y3, y4 = st
    zero = torch.zeros_like(u)
    au = u - GU * (_dt(y1[0], 1) + _dt(y1[1], 2) + _dt(_dt(y2[0], 1) + _dt(y2[1], 2), 0) + y4)
    un = _box(au)
    w1n = _shrink([w + GW * x for w, x in zip(w1, _L(*y1))], GW * p["omega"])
    w2n = _shrink([w + GW * x for w, x in zip(w2, _L(*y2))], GW)
    sn = _l1ball(s - GS * y4, p["alpha"])[0]
    tn = _l1ball(t - GT * (_dt(y3, 1) + y4), p["beta"])[0]
    ub, sb, tb = 2 * un - u, 2 * sn - s, 2 * tn - t
    lv, lh = _Lt([2 * a - b for a, b in zip(w1n, w1)])
    y1n = [y1[0] + GY * (_d(ub, 1) - lv), y1[1] + GY * (_d(ub, 2) - lh)]
    lv, lh = _Lt([2 * a - b for a, b in zip(w2n, w2)])
    ds = _d(ub, 0)
    y2n = [y2[0] + GY * (_d(ds, 1) - lv), y2[1] + GY * (_d(ds, 2) - lh)]
    y3n = y3 + GY * _d(tb, 1)
    q = y4 + GY * (ub + sb + tb) - GY * v
    nq = torch.sqrt((q * q).sum())
    lim = p["eps"] * GY
    y4n = (1 - lim / nq) * q if float(nq.detach()) > float(lim) else zero
    return [un, sn, tn, w1n, w2n, y1n, y2n, y3n, y4n]


def _start(v):
    z = torch.zeros_like(v)
    return [v, z, z, [z] * 6, [z] * 6, [z] * 2, [z] * 2, z, z]


def _solve(v, p, passes):
    with torch.no_grad():
        st = _start(v.double())
        for _ in range(passes):
            st = _pass(st, v, p)
    return st


def _flat(st):
    """float64 lists of cubes from the dense state of the framework."""
    w = lambda x: list(x.double().reshape((6,) + x.shape[2:]))  # noqa: E731
    d = {k: st[k].double() for k in STATE_KEYS}
    return [d["u"], d["s"], d["t"], w(st["w1"]), w(st["w2"]), list(d["y1"]), list(d["y2"]), d["y3"], d["y4"]]


def exact(case, seed):
    kind = case["kind"]
    if kind == "project":
        x, r = _vector(case, seed)
        out, tau = _l1ball(x.double(), r)
        return {"out": out, "tau": tau}
    if kind == "batch":
        got = []
        for k, s in enumerate(_shapes(case)):
            v, radii = _problem(*s, seed + 101 * k)
            got.append(_solve(v, dict(radii, omega=0.03), case["passes"])[:3])
        return {"u": [g[0] for g in got], "s": [g[1] for g in got], "t": [g[2] for g in got], "passes": None}
    n1, n2, n3 = case["n1"], case["n2"], case["n3"]
    v, radii = _problem(n1, n2, n3, seed)
    p = dict(radii, omega=0.03)
    if kind == "vjp":
        return None                 # the state after the pass is the framework's own
    if kind == "grad":
        if n1 * n2 * n3 * case["passes"] > 60_000_000:
            return None
        target = _problem(n1, n2, n3, seed + 1)[0].double()
        v = v.double().requires_grad_()
        prm = {k: torch.tensor(x, dtype=torch.float64, device="cuda", requires_grad=True) for k, x in p.items()}
        st = _start(v)
        for _ in range(case["passes"]):
            st = _pass(st, v, prm)
        grads = torch.autograd.grad(((st[0] - target) ** 2).mean(), [v] + [prm[k] for k in GRAD_PARAMS],
                                    allow_unused=True)
        return {"u": st[0].detach(), "v_bar": grads[0], **{k: g for k, g in zip(GRAD_PARAMS, grads[1:])}}
    u, s, t = _solve(v, p, case["passes"])[:3]
    return {"u": u, "s": s, "t": t, "passes": None}
