"""What the performance of this framework is measured on.

Each case is one call pattern of a user's program, through the package's
public classes: a single grid advanced by a number of time steps and read back
(``Sim``), a batch of instances advanced and read back (``Batch``), and the
surrogate network trained or evaluated (``Mlp``).  The sizes are those of the
repository's own workloads, studies and tests.

``listed()`` gives the fixed cases, ``draw(rng)`` one more of the same ranges,
``prepare`` what the program has in hand before the call (the handle with its
initial state, the pinned arrays its results are read into, the training
data), ``run`` the call, ``work`` the bytes and operations that it cannot do
without, and ``exact`` the same results in 64 bits from plain torch.
"""
import math

import numpy as np
import torch

import paper_1301_5058_gb300 as cx

SWEEP_SIDES = "512,1024,1536,2048"
# the algorithmic operations of one forward-Euler cell update and of one Heun
# step of a cell (two faces at 14 and an update at 15; a multiply-add is two)
EULER_FLOPS, HEUN_FLOPS = 43, 90


def _grid(name, nx, ny, steps, **kw):
    """One simulation handle: `steps` time steps, the diagnostics, b and n."""
    case = dict(kind="grid", nx=nx, ny=ny, dx=1.0, steps=steps, f64=False, heun=False,
                per_step=False, triangular=False, constant=False, upwind=False, n0=0.35, chi0=1.0,
                sigma0=4.0, a=0.8, bM=0.71, r0sq=1024.0)
    case.update(kw)
    return dict(case, name=name) if name else case


def _batch(name, count, sides, steps, **kw):
    """`count` instances, the i-th with side i of the list (taken cyclically),
    square or strips of height 1, its parameters drawn from the seed."""
    case = dict(kind="batch", count=count, sides=sides, strip=False, dx=1.0, steps=steps,
                f64=False, heun=False, per_step=False, triangular=False, constant=False,
                upwind=False, a=0.5, bM=0.71, r0sq=1024.0)
    case.update(kw)
    return dict(case, name=name) if name else case


def _net(name, kind, members, rows, batch=0, steps=0):
    case = dict(kind=kind, members=members, rows=rows, batch=batch, steps=steps)
    return dict(case, name=name) if name else case


def listed():
    return [
        # a few steps at a time, looking at the fields in between: the smallest call
        _grid("peek_256", 256, 256, 10, n0=0.7, chi0=0.5, a=0.5, bM=0.5, r0sq=16.0),
        # the plain-method case of the tests and of the smoke check: 256^2, 2000 steps
        _grid("config_256", 256, 256, 2000, n0=0.7, chi0=0.5, a=0.5, bM=0.5, r0sq=16.0),
        # one point of the parameter sweep stepped alone, between two of its 40 readings
        _grid("point_512", 512, 512, 500, n0=0.5, chi0=2.0, sigma0=3.0, a=0.5),
        # a grid that fits no tile, with the donor-cell mobility and an odd number of steps
        _grid("ragged_upwind", 1501, 1037, 301, n0=0.71, chi0=2.0, sigma0=2.0, upwind=True),
        # the 2D runs of the paper (N = 2048, L = 680): Heun, sigma redrawn every
        # step from the triangular law
        _grid("paper_2048", 2048, 2048, 200, dx=680.0 / 2048, n0=0.71, chi0=5.0, sigma0=1.0, a=1.0,
              r0sq=6.25, heun=True, per_step=True, triangular=True),
        # the radial colony in 64 bits, as it is checked against the 32-bit one
        _grid("radial_f64", 1024, 1024, 200, f64=True),
        # the benchmark's grid: 16384^2, dense branching regime
        _grid("large_16384", 16384, 16384, 200),
        # the 1D front-speed study: one strip per (n0, chi0), constant chemotaxis
        # law, 64 bits, no noise
        _batch("strips_f64", 20, "400", 1000, strip=True, dx=0.1, f64=True, constant=True, a=0.0,
               r0sq=6.25),
        # the labels of a small sweep (256^2 instances), between two readings
        _batch("labels_256", 96, "256", 500, r0sq=64.0),
        # the parameter sweep's mix of sides
        _batch("sweep_mix", 24, SWEEP_SIDES, 500),
        # the screen's networks: Adam steps of 8 members on minibatches of 256
        _net("train_8", "train", 8, 8192, 256, 100),
        # screening candidates: one forward pass of the 8 members over 8192 points
        _net("screen_8", "screen", 8, 8192),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["grid"] * 6 + ["batch"] * 3 + ["strips", "train", "screen"])
    if what == "train":
        return _net("", "train", rng.randint(1, 16), _log(rng, 1024, 8192), _log(rng, 50, 1000),
                    _log(rng, 20, 200))
    if what == "screen":
        return _net("", "screen", rng.randint(1, 16), _log(rng, 100, 8192))
    if what == "strips":
        return _batch("", rng.randint(2, 30), "%d" % _log(rng, 200, 1600), _log(rng, 50, 2000),
                      strip=True, dx=round(rng.uniform(0.05, 0.2), 3), f64=rng.random() < 0.8,
                      constant=True, upwind=rng.random() < 0.3, a=0.0, r0sq=6.25)
    opt = dict(heun=rng.random() < 0.3, per_step=rng.random() < 0.3, triangular=rng.random() < 0.5,
               constant=rng.random() < 0.15, upwind=rng.random() < 0.2, f64=rng.random() < 0.2)
    # cell-steps a drawn case may take, well below the largest listed case
    room = 2e8 if opt["f64"] else 1e10
    if what == "batch":
        lo = _log(rng, 64, 1500)
        sides = [_log(rng, lo, min(2048, 2 * lo)) for _ in range(rng.randint(1, 4))]
        mean = sum(s * s for s in sides) / len(sides)
        # the instances together at most as large as the listed mix, or in 64 bits a quarter
        count = max(2, min(_log(rng, 4, 96), int((1.2e7 if opt["f64"] else 5e7) / mean)))
        steps = max(1, min(_log(rng, 10, 1000), int(room / (mean * count))))
        return _batch("", count, ",".join(str(s) for s in sides), steps,
                      a=round(rng.uniform(0.1, 1.0), 2), r0sq=64.0, **opt)
    nx = _log(rng, 32, 8192)
    ny = max(16, min(8192, int(nx * math.exp(rng.uniform(-0.7, 0.7)))))
    steps = max(1, min(_log(rng, 2, 2000), int(room / (nx * ny))))
    return _grid("", nx, ny, steps, n0=round(rng.uniform(0.2, 1.4), 3),
                 chi0=rng.choice([0.0, round(rng.uniform(0.05, 5.0), 3)]),
                 sigma0=round(rng.uniform(1.0, 6.0), 3), a=round(rng.uniform(0.1, 1.0), 2),
                 r0sq=rng.choice([16.0, 64.0, 1024.0]), **opt)


def _options(case):
    """The parameter fields that a case's switches stand for."""
    return dict(precision=cx.CX_PREC_F64 if case["f64"] else cx.CX_PREC_F32,
                scheme=cx.CX_SCHEME_HEUN if case["heun"] else cx.CX_SCHEME_EULER,
                noise_mode=cx.CX_NOISE_PER_STEP if case["per_step"] else cx.CX_NOISE_STATIC,
                noise_dist=cx.CX_NOISE_TRIANGULAR if case["triangular"] else cx.CX_NOISE_UNIFORM,
                chemo_law=cx.CX_CHEMO_CONSTANT if case["constant"] else cx.CX_CHEMO_RECEPTOR,
                mobility=cx.CX_MOBILITY_UPWIND if case["upwind"] else cx.CX_MOBILITY_CENTRAL)


def _instances(case, seed):
    """(nx, ny, n0, chi0, sigma0, a, seed) of every instance of a batch case:
    the sweep's log-uniform box, or the front-speed study's range for strips."""
    r = np.random.default_rng(seed)
    sides = [int(s) for s in case["sides"].split(",")]
    out = []
    for i in range(case["count"]):
        s = sides[i % len(sides)]
        if case["strip"]:
            n0, chi0, sigma0 = r.uniform(0.35, 4.0), r.uniform(0.0, 10.0), 1.0
        else:
            n0 = math.exp(r.uniform(math.log(0.1), math.log(1.5)))
            chi0 = math.exp(r.uniform(math.log(0.05), math.log(4.0)))
            chi0 = 0.0 if r.uniform() < 0.1 else chi0
            sigma0 = math.exp(r.uniform(0.0, math.log(8.0)))
        out.append((s, 1 if case["strip"] else s, n0, chi0, sigma0, case["a"], seed + i))
    return out


def _net_data(case, seed):
    """(inputs, targets, parameters) of a network case: points of the unit box,
    labels that are a smooth function of them, Glorot-uniform weights."""
    r = np.random.default_rng(seed)
    e, n = case["members"], case["rows"]
    x = r.uniform(-1, 1, (n, 4)).astype(np.float32)
    t = np.stack([np.sin(2 * x[:, 0]) * x[:, 2] + 0.5 * x[:, 1], np.tanh(2 * x[:, 1] - x[:, 3])], 1)
    t = (t + 0.02 * r.normal(size=t.shape)).astype(np.float32)
    theta = []
    for _ in range(e):
        for rows, cols in ((256, 4), (256, 256), (2, 256)):
            lim = math.sqrt(6.0 / (rows + cols))
            theta += [r.uniform(-lim, lim, rows * cols), np.zeros(rows)]
    theta = np.concatenate(theta).astype(np.float32).reshape(e, -1)
    if case["kind"] == "train":  # every member takes the rows in its own order
        order = [r.permutation(n) for _ in range(e)]
        x, t = np.stack([x[p] for p in order]), np.stack([t[p] for p in order])
    return x, t, theta


def _host(shape, f64):
    """A pinned host array that results are read into."""
    return torch.empty(shape, dtype=torch.float64 if f64 else torch.float32, pin_memory=True).numpy()


def prepare(case, seed):
    if case["kind"] == "grid":
        sim = cx.Sim(case["nx"], case["ny"], case["dx"], seed=seed, n0=case["n0"],
                     chi0=case["chi0"], sigma0=case["sigma0"], noise_amp=case["a"], bM=case["bM"],
                     r0sq=case["r0sq"], **_options(case))
        shape = (case["ny"], case["nx"])
        return dict(case=case, sim=sim, b=_host(shape, case["f64"]), n=_host(shape, case["f64"]))
    if case["kind"] == "batch":
        inst = _instances(case, seed)
        batch = cx.Batch([dict(nx=nx, ny=ny, dx=case["dx"], seed=s, n0=n0, chi0=chi0, sigma0=s0,
                               noise_amp=a, bM=case["bM"], r0sq=case["r0sq"],
                               b_threshold=0.5 * n0 if case["strip"] else 0.0, **_options(case))
                          for nx, ny, n0, chi0, s0, a, s in inst])
        # the fields of all instances one after the other in one array each
        at = np.cumsum([0] + [nx * ny for nx, ny, *_ in inst])
        out = [_host(int(at[-1]), case["f64"]) for _ in range(2)]
        views = [[o[at[i]:at[i + 1]].reshape(inst[i][1], inst[i][0]) for i in range(len(inst))]
                 for o in out]
        return dict(case=case, batch=batch, out=out, views=views)
    x, t, theta = _net_data(case, seed)
    net = cx.Mlp(case["rows"], theta, members=case["members"])
    return dict(case=case, net=net, x=x, t=t)


def _masses(d):
    return [d["mass_b"], d["mass_n"], d["invariant"]]


def run(state):
    case = state["case"]
    if case["kind"] == "grid":
        sim = state["sim"]
        sim.step(case["steps"])
        d = sim.diagnostics(check=False)
        cx.cx_get_field(sim.h, cx.CX_FIELD_B, state["b"])
        cx.cx_get_field(sim.h, cx.CX_FIELD_N, state["n"])
        return dict(b=state["b"], n=state["n"], masses=np.array(_masses(d)))
    if case["kind"] == "batch":
        batch = state["batch"]
        batch.step(case["steps"])
        d = batch.diagnostics(check=False)
        for which, views in zip((cx.CX_FIELD_B, cx.CX_FIELD_N), state["views"]):
            for i, v in enumerate(views):
                cx.cx_batch_get_field(batch.h, i, which, v)
        return dict(b=state["out"][0], n=state["out"][1], masses=np.array([_masses(x) for x in d]))
    if case["kind"] == "train":
        losses = state["net"].train(state["x"], state["t"], case["batch"], case["steps"], 1e-3)
        return dict(losses=losses, params=state["net"].params())
    return dict(y=state["net"].forward(state["x"]))


def work(case):
    if case["kind"] in ("grid", "batch"):
        if case["kind"] == "grid":
            cells = case["nx"] * case["ny"]
        else:
            cells = sum(nx * ny for nx, ny, *_ in _instances(case, 0))
        # b and n read and written once, a static sigma field read once
        size = (8 if case["f64"] else 4) * (4 if case["per_step"] else 5)
        return {"bytes": size * cells,
                "flops": cells * case["steps"] * (HEUN_FLOPS if case["heun"] else EULER_FLOPS)}
    e, n = case["members"], case["rows"]
    params = 256 * 4 + 256 + 256 * 256 + 256 + 2 * 256 + 2
    macs = 256 * 4 + 256 * 256 + 2 * 256
    if case["kind"] == "screen":
        return {"bytes": 4 * (4 * n + e * params + 2 * e * n), "flops": 2 * macs * e * n}
    return {"bytes": 4 * e * (6 * n + 6 * params) + 8 * e * case["steps"],
            "flops": case["steps"] * e * (6 * macs * case["batch"] + 12 * params)}


# ---- the same results in 64 bits from plain torch ----------------------------

def _philox(c, k):
    """Philox4x32-10 (Salmon et al., SC'11) of four counter words (int64 tensors
    holding 32 bits) under the key words k (numbers or tensors that broadcast)."""
    mask = 0xFFFFFFFF

    def product(m, x):  # the high and low words of a 32 x 32 bit product
        lo, hi = m * (x & 0xFFFF), m * (x >> 16)
        low = lo + ((hi & 0xFFFF) << 16)
        return ((hi >> 16) + (low >> 32)) & mask, low & mask

    k0, k1 = k
    for _ in range(10):
        h0, l0 = product(0xD2511F53, c[0])
        h1, l1 = product(0xCD9E8D57, c[2])
        c = (h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0)
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _delta(cells, seeds, step, triangular, words32):
    """Delta of cells 0 .. cells - 1 of every instance at a time step, (instances,
    cells).  words32: the recipe of a 32-bit state whose sigma is redrawn every
    step (one block per four cells, two 16-bit numbers a cell)."""
    mask = 0xFFFFFFFF
    k = tuple(torch.tensor([(s >> sh) & mask for s in seeds], device="cuda").reshape(-1, 1)
              for sh in (0, 32))
    out = torch.empty(len(seeds), cells, dtype=torch.float64, device="cuda")
    per = 4 if words32 else 1
    chunk = (1 << 25) // len(seeds) // 4 * 4 + 4
    for c0 in range(0, cells, chunk):
        c1 = min(cells, c0 + chunk)
        i = torch.arange(c0 // per, -(-c1 // per), device="cuda").reshape(1, -1)
        w = _philox((i & mask, i >> 32, torch.full_like(i, step & mask),
                     torch.full_like(i, step >> 32)), k)
        if words32:
            w = torch.stack(w, -1).reshape(len(seeds), -1)[:, :c1 - c0]
            ja, jb = w >> 16, w & 0xFFFF
            d = (ja + jb if triangular else 2 * ja).double() / 2.0 ** 16 - 1.0
        else:
            ka, kb = (w[0] << 21) | (w[1] >> 11), (w[2] << 21) | (w[3] >> 11)
            d = ((ka + kb if triangular else 2 * ka) - (1 << 53)).double() / 2.0 ** 53
        out[:, c0:c1] = d
    return out


def _solve(case, nx, ny, n0, chi0, sigma0, a, seeds):
    """(b, n, masses) of the instances of one size after the case's steps; n0, chi0,
    sigma0 lists.  Fluxes with face means on the faces between cells, none at
    the walls; forward Euler or Heun."""
    dx, bM = case["dx"], case["bM"]
    col = [torch.tensor(v, dtype=torch.float64, device="cuda").reshape(-1, 1, 1)
           for v in (n0, chi0, sigma0)]
    N0, X0, S0 = col
    B = bM + N0
    dmax = torch.clamp(S0 * (1 + a) * N0 * B * (1 + X0 * B), min=1.0)
    dt = 0.2 * torch.minimum(dx * dx / (4 * dmax), 1 / (4 / dx ** 2 + B))

    def sigma(step):
        d = _delta(nx * ny, seeds, step, case["triangular"], case["per_step"] and not case["f64"])
        return d.mul_(a).add_(1.0).reshape(-1, ny, nx).mul_(S0)

    x = (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5 - nx / 2) * dx
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5 - ny / 2) * dx
    q = (x * x + (y * y)[:, None]) / case["r0sq"]
    b = torch.where(q <= 40.0, bM * torch.exp(-q), 0.0 * q).expand(len(seeds), ny, nx).clone()
    n = N0.expand(len(seeds), ny, nx).clone()
    del q

    def fluxes(s, b, n, rb, rn, axis):
        m = b.shape[axis]
        if m < 2:
            return
        L, R = (lambda f: f.narrow(axis, 0, m - 1)), (lambda f: f.narrow(axis, 1, m - 1))
        bL, bR, nf = L(b), R(b), (L(n) + R(n)).mul_(0.5)
        dn = (R(n) - L(n)).div_(dx)
        bf = (bL + bR).mul_(0.5)
        b2 = torch.where(dn >= 0, bL, bR).square_() if case["upwind"] else bf * bf
        chi = X0 if case["constant"] else X0 / (nf + 1).square_()
        f = (bR - bL).div_(dx).mul_(bf).sub_(b2.mul_(chi).mul_(dn))
        f.mul_(nf).mul_((L(s) + R(s)).mul_(0.5)).div_(dx)
        L(rb).add_(f)
        R(rb).sub_(f)
        dn.div_(dx)
        L(rn).add_(dn)
        R(rn).sub_(dn)

    def rate(s, b, n):
        rb = n * b
        rn = -rb
        fluxes(s, b, n, rb, rn, 1)
        fluxes(s, b, n, rb, rn, 2)
        return rb.mul_(dt), rn.mul_(dt)

    s = None if case["per_step"] else sigma(0)
    for step in range(case["steps"]):
        if case["per_step"]:
            s = sigma(step)
        rb, rn = rate(s, b, n)
        if case["heun"]:
            rb2, rn2 = rate(s, b + rb, n + rn)
            rb, rn = rb.add_(rb2).mul_(0.5), rn.add_(rn2).mul_(0.5)
        b.add_(rb)
        n.add_(rn)
    mb, mn = (f.sum((1, 2)) * dx * dx for f in (b, n))
    return b, n, torch.stack([mb, mn, mb + mn], 1)


def _network(theta, x):
    """The layers' values of every member, x (members, n, 4)."""
    e = theta.shape[0]
    cut = np.cumsum([0, 1024, 256, 65536, 256, 512, 2])
    w1, b1, w2, b2, w3, b3 = (theta[:, i:j] for i, j in zip(cut[:-1], cut[1:]))
    h1 = torch.tanh(x @ w1.reshape(e, 256, 4).mT + b1[:, None])
    h2 = torch.tanh(h1 @ w2.reshape(e, 256, 256).mT + b2[:, None])
    return h1, h2, h2 @ w3.reshape(e, 2, 256).mT + b3[:, None]


def _exact_train(case, x, t, theta):
    e, nb, lr = case["members"], case["batch"], 1e-3
    m, v, losses = torch.zeros_like(theta), torch.zeros_like(theta), []
    for k in range(case["steps"]):
        i = k % (case["rows"] // nb) * nb
        xs, ts = x[:, i:i + nb], t[:, i:i + nb]
        h1, h2, y = _network(theta, xs)
        losses.append((y - ts).square().sum((1, 2)) / (2 * nb))
        w2 = theta[:, 1280:1280 + 65536].reshape(e, 256, 256)
        w3 = theta[:, 1280 + 65536 + 256:-2].reshape(e, 2, 256)
        dy = (y - ts) / nb
        d2 = (dy @ w3) * (1 - h2 * h2)
        d1 = (d2 @ w2) * (1 - h1 * h1)
        g = torch.cat([(d1.mT @ xs).reshape(e, -1), d1.sum(1), (d2.mT @ h1).reshape(e, -1),
                       d2.sum(1), (dy.mT @ h2).reshape(e, -1), dy.sum(1)], 1)
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        theta = theta - lr * (m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    return torch.stack(losses, 1), theta


def exact(case, seed):
    if case["kind"] == "grid":
        b, n, masses = _solve(case, case["nx"], case["ny"], [case["n0"]], [case["chi0"]],
                              [case["sigma0"]], case["a"], [seed])
        return dict(b=b[0], n=n[0], masses=masses[0])
    if case["kind"] == "batch":
        inst = _instances(case, seed)
        b, n, masses = ([None] * len(inst) for _ in range(3))
        for size in sorted({(i[0], i[1]) for i in inst}):
            at = [k for k, i in enumerate(inst) if (i[0], i[1]) == size]
            got = _solve(case, *size, [inst[k][2] for k in at], [inst[k][3] for k in at],
                         [inst[k][4] for k in at], case["a"], [inst[k][6] for k in at])
            for j, k in enumerate(at):
                b[k], n[k], masses[k] = got[0][j].reshape(-1), got[1][j].reshape(-1), got[2][j]
        return dict(b=torch.cat(b), n=torch.cat(n), masses=torch.stack(masses))
    x, t, theta = (torch.tensor(v, device="cuda").double() for v in _net_data(case, seed))
    if case["kind"] == "train":
        losses, params = _exact_train(case, x, t, theta)
    else:
        y = _network(theta, x.expand(case["members"], -1, -1))[2]
    one = (lambda v: v[0]) if case["members"] == 1 else (lambda v: v)
    return dict(losses=one(losses), params=one(params)) if case["kind"] == "train" else dict(y=one(y))
