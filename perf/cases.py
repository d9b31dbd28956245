"""Performance cases of the dynamic optimal-transport framework.

Each case is one piece of work that a user of the package has it do, through the
public entry points: solves of Algorithm 1 on image grids and hue histograms
(single pairs, batches of one size, batches of mixed sizes, FP32 and FP64
plans), the periodic histogram specification of the hue image pipeline, and one
layer of the warm-start network in training.

Solves run a fixed number of iterations (no tolerance), with the residual
checks at the plan's default spacing of 10 iterations.  They return the energy of
the last check and what the caller takes home: the packed path (m, f) in solver
units, as a warm start or a training target takes it ("path"), or the
interpolated densities f, as a morph takes its frames ("frames").  ``exact``
repeats them in 64 bits with plain torch: dense transform matrices, Newton to
convergence.
"""
import math

import torch

import paper_1501_04840_gb300 as ot
from paper_1501_04840_gb300 import huepipe
from paper_1501_04840_gb300 import nn as net

SIGMA, TAU_SIGMA = 0.3, 0.99          # the grid defaults

RGB = "neumann,neumann,periodic"


def _image(name, n1, n2, C, P, iters, bc=RGB, batch=1, prec="mixed", take="path"):
    return {"name": name, "kind": "image", "n1": n1, "n2": n2, "C": C, "P": P, "iters": iters, "bc": bc,
            "batch": batch, "prec": prec, "take": take}


def _hue(name, bins, P, batch, iters):
    return {"name": name, "kind": "hue", "bins": bins, "P": P, "batch": batch, "iters": iters, "take": "frames"}


def listed():
    return [
        # the smallest image pair of the tests and the smoke run: latency and launches count
        _image("rgb 32x32x3x16", 32, 32, 3, 16, 100),
        # the warm-start network's image size
        _image("rgb 128x128x3x32", 128, 128, 3, 32, 100),
        # the benchmark's headline workload (the paper's image size and time steps)
        _image("rgb 256x256x3x32", 256, 256, 3, 32, 100),
        # the largest grid of the precision study
        _image("rgb 512x512x3x64", 512, 512, 3, 64, 20),
        # a photograph's thumbnail: 4:3, no power of two on any axis
        _image("rgb 180x135x3x24", 180, 135, 3, 24, 20, take="frames"),
        # a grey image of odd sides and odd P, Neumann on both axes
        _image("grey 225x151x17", 225, 151, 1, 17, 20, bc="neumann,neumann", take="frames"),
        # the FP64 plan, the precision study's reference arm
        _image("rgb 128x128x3x32 fp64", 128, 128, 3, 32, 20, prec="fp64"),
        # one pair of hue histograms (section 5 of the paper)
        _hue("hue 360x64", 360, 64, 1, 50),
        # the same sizes, 64 pairs in one plan
        _hue("hue 360x64 batch 64", 360, 64, 64, 50),
        # a batch of mixed sizes, as the batch benchmark's (image sides 64..256, hue histograms)
        {"name": "mixed batch", "kind": "mixed", "images": "64x96x16;128x96x24;192x128x20;100x75x18",
         "hues": "360x64;101x20;256x32;400x40;288x48;64x16;333x27;180x36", "iters": 50},
        # specification of an image's hues to a transported histogram (every frame of a hue morph)
        {"name": "hue specify 256x256", "kind": "specify", "npix": 65536, "bins": 360},
        # forward and backward of one convolution of the warm-start network's finest level, batch 4
        {"name": "conv 16-16 128x128x32", "kind": "conv", "N": 4, "T": 32, "Y": 128, "X": 128, "cin": 16, "cout": 16},
    ]


def _side(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.3:                       # sides of camera and screen images are often such lengths
        n = min((m for m in (32, 48, 64, 96, 128, 160, 192, 240, 256, 320, 384, 480, 512) if lo <= m <= hi),
                key=lambda m: abs(math.log(m / n)), default=n)
    return n


def _unnamed(case):
    return {k: v for k, v in case.items() if k != "name"}


def draw(rng):
    kind = rng.choice(["rgb", "rgb", "rgb", "rgb", "grey", "other", "fp64", "hue", "huebatch", "mixed", "specify",
                       "conv"])
    if kind in ("rgb", "grey", "other", "fp64"):
        hi = 160 if kind == "fp64" else 320
        n1 = _side(rng, 32, hi)
        n2 = min(hi, max(24, int(n1 * rng.uniform(0.6, 1.5))))
        if rng.random() < 0.3:
            n2 = _side(rng, max(24, n2 // 2), min(hi, 2 * n2))
        take = "path" if kind == "fp64" else "frames"
        if kind != "fp64" and rng.random() < 0.3:                # sides of a power of two
            n1, n2, take = rng.choice([64, 128, 256, 512]), rng.choice([64, 128, 256, 512]), "path"
        C = 1 if kind == "grey" else 3
        P = rng.choice([16, 32, 32, 64, rng.randint(9, 48)])
        cells = n1 * n2 * C * P
        iters = max(10, min(100 if take == "path" else 20, int((2e7 if kind == "fp64" else 4e8) / cells)))
        bc = {"grey": "neumann,neumann", "rgb": RGB, "fp64": RGB}.get(kind) or rng.choice(
            ["neumann,neumann,neumann", "periodic,periodic,periodic", "periodic,neumann,periodic"])
        return _unnamed(_image("", n1, n2, C, P, iters, bc, 1, "fp64" if kind == "fp64" else "mixed", take))
    if kind == "hue":
        return _unnamed(_hue("", _side(rng, 64, 420), rng.randint(16, 64), 1, rng.randint(20, 50)))
    if kind == "huebatch":
        return _unnamed(_hue("", _side(rng, 64, 480), rng.randint(16, 64), rng.randint(4, 96), rng.randint(20, 60)))
    if kind == "mixed":
        im = ";".join("%dx%dx%d" % (_side(rng, 48, 192), _side(rng, 48, 192), rng.randint(12, 40))
                      for _ in range(rng.randint(2, 4)))
        hu = ";".join("%dx%d" % (_side(rng, 64, 400), rng.randint(16, 64)) for _ in range(rng.randint(3, 8)))
        return {"kind": "mixed", "images": im, "hues": hu, "iters": rng.randint(15, 50)}
    if kind == "specify":
        return {"kind": "specify", "npix": int(round(4 ** rng.uniform(6, 8.5))),
                "bins": rng.choice([180, 256, 360, rng.randint(64, 720)])}
    lvl = rng.randint(0, 3)                      # a level of the network: 16/32/48/64 channels
    ch = (16, 32, 48, 64)
    side = 128 >> lvl
    cin = rng.choice([ch[lvl], ch[max(0, lvl - 1)], ch[lvl] + ch[min(3, lvl + 1)]])
    return {"kind": "conv", "N": rng.randint(1, 4), "T": 32, "Y": side, "X": side, "cin": cin,
            "cout": ch[lvl]}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _blobs(n1, n2, C, gen):
    """Gaussian blobs per channel (centres uniform, deviation 3..6 pixels, amplitude 0.5..1), a floor, mass 1."""
    nb = max(8, n1 * n2 // 2048)
    u = torch.rand((C, 4, nb), generator=gen, dtype=torch.float64)
    sd = 3 + 3 * u[:, 2]
    amp = 0.5 + 0.5 * u[:, 3]
    x = torch.arange(n1, dtype=torch.float64) + 0.5
    y = torch.arange(n2, dtype=torch.float64) + 0.5
    gx = torch.exp(-(x[None, :, None] - n1 * u[:, 0, None, :]) ** 2 / (2 * sd[:, None, :] ** 2))
    gy = torch.exp(-(y[None, :, None] - n2 * u[:, 1, None, :]) ** 2 / (2 * sd[:, None, :] ** 2)) * amp[:, None, :]
    out = gy @ gx.transpose(1, 2) + 1e-3
    return out / out.sum()


def _bumps(n, gen):
    """Three von Mises bumps on n periodic bins, mass 1."""
    u = torch.rand((3, 3), generator=gen, dtype=torch.float64)
    th = (torch.arange(n, dtype=torch.float64) + 0.5) * (2 * math.pi / n)
    w = -torch.log(u[2] + 1e-12)
    h = (w[:, None] * torch.exp((2 + 18 * u[0])[:, None] * (torch.cos(th[None] - 2 * math.pi * u[1][:, None]) - 1)))
    h = h.sum(0)
    return h / h.sum()


def _sizes(text):
    return [tuple(int(v) for v in s.split("x")) for s in text.split(";")]


def _densities(case, seed):
    """(f0, f1) of every problem of a solve, float32 on the GPU (a list of pairs for a mixed batch)."""
    gen = torch.Generator().manual_seed(int(seed))
    if case["kind"] == "image":
        f = [torch.stack([_blobs(case["n1"], case["n2"], case["C"], gen) for _ in range(case["batch"])])
             for _ in range(2)]
        return [a.float().cuda() for a in f]
    if case["kind"] == "hue":
        f = [torch.stack([_bumps(case["bins"], gen) for _ in range(case["batch"])]) for _ in range(2)]
        return [a.float().cuda() for a in f]
    pairs = [tuple(_blobs(n1, n2, 3, gen).float().cuda() for _ in range(2)) for n1, n2, _ in _sizes(case["images"])]
    return pairs + [tuple(_bumps(n, gen).float().cuda() for _ in range(2)) for n, _ in _sizes(case["hues"])]


def _specify_inputs(case, seed):
    """Hues of a flower on its background (two clusters, 8-bit image noise) and a transported histogram."""
    gen = torch.Generator().manual_seed(int(seed))
    n, bins = case["npix"], case["bins"]
    u = torch.rand(n, generator=gen, dtype=torch.float64)
    g = torch.randn(n, generator=gen, dtype=torch.float64)
    h = torch.where(u < 0.35, 0.13 + 0.02 * g, 0.38 + 0.03 * g) % 1.0
    return h.float().clamp(0, 1 - 2.0 ** -24).cuda(), _bumps(bins, gen).float().cuda()


def _conv_inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    vol = (case["N"], case["T"], case["Y"], case["X"])

    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda")

    cin, cout = case["cin"], case["cout"]
    x = normal(*vol, cin).relu().bfloat16()
    w = (normal(cout, 27, cin) * math.sqrt(2.0 / (27 * cin))).bfloat16()
    return vol, x, w, 0.1 * normal(cout), (1e-2 * normal(*vol, cout)).bfloat16()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "image":
        bc = case["bc"].split(",")
        n = (case["n1"], case["n2"], case["C"])[:len(bc)]
        g = ot.grid(n, bc, case["P"], precision=ot.PREC_FP64 if case["prec"] == "fp64" else ot.PREC_MIXED)
        return {"case": case, "plan": ot.Plan(g, batch=case["batch"]), "f": _densities(case, seed)}
    if kind == "hue":
        return {"case": case, "plan": ot.Plan(ot.hue_grid(case["bins"], case["P"]), batch=case["batch"]),
                "f": _densities(case, seed)}
    if kind == "mixed":
        grids = [ot.rgb_grid(*s) for s in _sizes(case["images"])] + [ot.hue_grid(*s) for s in _sizes(case["hues"])]
        return {"case": case, "batch": ot.Batch(grids), "f": _densities(case, seed)}
    if kind == "specify":
        h, target = _specify_inputs(case, seed)
        return {"case": case, "h": h, "target": target}
    vol, x, w, bias, dy = _conv_inputs(case, seed)
    cin, cout = case["cin"], case["cout"]
    bf = dict(dtype=torch.bfloat16, device="cuda")
    return {"case": case, "vol": vol, "x": x, "w": w, "bias": bias, "dy": dy, "g": torch.empty_like(dy),
            "y": torch.empty(vol + (cout,), **bf), "dx": torch.empty(vol + (cin,), **bf),
            "wr": torch.empty(cout * 27 * cin, **bf), "dw": torch.empty((cout, 27, cin), device="cuda"),
            "db": torch.empty(cout, device="cuda")}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("image", "hue"):
        plan = s["plan"]
        st = plan.solve(s["f"][0], s["f"][1], case["iters"])
        if case["take"] == "path":
            x = torch.empty(plan.path_size, dtype=torch.float32, device="cuda")
            plan.x_into(x)
        else:
            x = torch.empty((plan.batch,) + plan.f_shape(), dtype=torch.float32, device="cuda")
            plan.path_into(x)
        return {"x": x, "energy": st.energy}
    if kind == "mixed":
        st = s["batch"].solve([a for a, _ in s["f"]], [b for _, b in s["f"]], case["iters"])
        return [{"x": s["batch"].path(i)["f"], "energy": q.energy} for i, q in enumerate(st)]
    if kind == "specify":
        return huepipe.specify(s["h"], case["bins"], s["target"])
    x, y, g, dx = (net.whole(s[k]) for k in ("x", "y", "g", "dx"))
    net.conv3d(s["vol"], x, s["w"], s["bias"], y, True)
    s["g"].copy_(s["dy"])
    net.relu_grad(g, y)
    s["dw"].zero_()
    s["db"].zero_()
    net.conv3d_wgrad(s["vol"], x, g, s["dw"], s["db"])
    net.rotate_weights(case["cin"], case["cout"], s["w"], s["wr"])
    net.conv3d(s["vol"], g, s["wr"], None, dx, False)
    return {"y": s["y"], "dx": s["dx"], "dw": s["dw"], "db": s["db"]}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------

def _solve_work(n1, n2, C, P, batch, iters, size=4):
    """An iteration reads and writes its state (x and b: four values each per cell), forms the stencils and the prox
    (about 150 operations a cell) and transforms every axis forth and back (2.5 log2 n operations per cell each);
    the solve reads the densities once and writes the densities of its path once."""
    cells = n1 * n2 * C * P * batch
    lg = sum(math.log2(max(n, 2)) for n in (n1, n2, P)) + 6
    return {"bytes": cells * 16.0 * size * iters + cells * 4.0 + 8.0 * n1 * n2 * C * batch,
            "flops": cells * (150.0 + 5.0 * lg) * iters}


def work(case):
    kind = case["kind"]
    if kind == "image":
        return _solve_work(case["n1"], case["n2"], case["C"], case["P"], case["batch"], case["iters"],
                           8 if case["prec"] == "fp64" else 4)
    if kind == "hue":
        return _solve_work(case["bins"], 1, 1, case["P"], case["batch"], case["iters"])
    if kind == "mixed":
        w = [_solve_work(a, b, 3, P, 1, case["iters"]) for a, b, P in _sizes(case["images"])]
        w += [_solve_work(n, 1, 1, P, 1, case["iters"]) for n, P in _sizes(case["hues"])]
        return {k: sum(v[k] for v in w) for k in ("bytes", "flops")}
    if kind == "specify":
        n = case["npix"]      # the hues read and written once; a sort and a search over the cyclic shifts
        return {"bytes": 8.0 * n + 4.0 * case["bins"], "flops": 40.0 * n * math.log2(n)}
    vox = case["N"] * case["T"] * case["Y"] * case["X"]
    ci, co = case["cin"], case["cout"]
    # x, dy read; y, dx written; weights and their gradients; three products of 27 taps
    return {"bytes": 2.0 * vox * 2 * (ci + co) + 27.0 * ci * co * 6, "flops": 3 * 2.0 * vox * 27 * ci * co}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

def _basis(n, periodic):
    """Orthonormal eigenvectors (rows) of the axis's Laplacian and 4 sin^2 of their half angle."""
    i = torch.arange(n, dtype=torch.float64, device="cuda")
    if not periodic:
        M = torch.cos(math.pi / n * i[:, None] * (i[None, :] + 0.5)) * math.sqrt(2.0 / n)
        M[0] = math.sqrt(1.0 / n)
        return M, 4 * torch.sin(math.pi * i / (2 * n)) ** 2
    fr = (i + 1).div(2, rounding_mode="floor")
    ang = 2 * math.pi / n * ((fr[:, None] * i[None, :]) % n)
    M = torch.where((torch.arange(n, device="cuda") % 2 == 1)[:, None], torch.cos(ang), torch.sin(ang)) * math.sqrt(2.0 / n)
    M[0] = math.sqrt(1.0 / n)
    if n % 2 == 0 and n > 1:
        M[n - 1] = torch.cos(math.pi * i) * math.sqrt(1.0 / n)
    return M, 4 * torch.sin(math.pi * fr / n) ** 2


def _along(M, v, dim):
    return torch.movedim(torch.tensordot(v, M, dims=([dim], [1])), -1, dim)


def _prox(am, af):
    """argmin |u|^2/(2v) + sigma/2 |u - am|^2 + sigma/2 (v - af)^2 per cell, by Newton from an upper bound."""
    e = SIGMA * af
    d = 0.5 * SIGMA ** 2 * sum(a * a for a in am)
    live = e + d > 0
    z = torch.where(live, e + d, torch.zeros_like(e)).clamp_min(0)
    for _ in range(80):
        w = 1 + z
        step = (w * w * (z - e) - d) / (w * (2 * (z - e) + w))
        step = torch.where(live, step, torch.zeros_like(step))
        z = z - step
        if float((step.abs() / (1e-300 + z.abs() + e.abs() + d)).max()) < 1e-15:
            break
    z = torch.where(live, z.clamp_min(0), torch.zeros_like(z))
    r = z / (1 + z)
    return [r * a for a in am], z / SIGMA


def _exact_solve(f0, f1, P, periodic, iters, take="frames"):
    """Algorithm 1 in 64 bits for densities [B][c][y][x] (or [B][bin]) on axes listed x first."""
    d = len(periodic)
    B = f0.shape[0]
    f0, f1 = (a.double().reshape((B,) + tuple(a.shape[1 + (a.dim() - 1 - d):])) for a in (f0, f1))
    n = [f0.shape[d - k] for k in range(d)]                      # axis k lies in dimension d - k of [B][..]
    ax = [1 + d - k for k in range(d)]                           # its dimension in [B][t][..]
    S = f0[0].numel()
    dims = tuple(range(1, 1 + d))
    m0, m1 = f0.sum(dims), f1.sum(dims)
    shape = (B,) + (1,) * d
    f0, f1 = f0 * (S / m0).view(shape), f1 * (S / m1).view(shape)
    scale = 0.5 * (m0 + m1) / S
    mats = [_basis(n[k], periodic[k]) for k in range(d)] + [_basis(P, False)]
    axes, fac = ax + [1], [float(v) for v in n] + [float(P)]
    lam = torch.zeros((1,) * (2 + d), dtype=torch.float64, device="cuda")
    for (_, ev), a, s in zip(mats, axes, fac):
        lam = lam + (s * s * ev).view([-1 if q == a else 1 for q in range(2 + d)])
    inv = torch.where(lam > 1e-9, 1 / lam.clamp_min(1e-9), torch.zeros_like(lam))

    def edge(v, k):                                              # zero on the absent last face of a Neumann axis
        if not periodic[k]:
            v.narrow(ax[k], n[k] - 1, 1).zero_()
        return v

    full = (B, P) + tuple(f0.shape[1:])
    am = [torch.zeros(full, dtype=torch.float64, device="cuda") for _ in range(d)]
    af = torch.zeros(full, dtype=torch.float64, device="cuda")    # slot t: f at time (t + 1) / P
    b = [torch.zeros_like(af) for _ in range(d + 1)]
    en = None
    for it in range(iters):
        fn = torch.cat([af[:, :-1], f1[:, None]], 1)
        r = P * (fn - torch.cat([f0[:, None], af[:, :-1]], 1))
        for k in range(d):
            r += fac[k] * (am[k] - am[k].roll(1, ax[k]))         # the absent face is zero: rolling it in is harmless
        for (M, _), a in zip(mats, axes):
            r = _along(M, r, a)
        r = r * inv
        for (M, _), a in zip(mats, axes):
            r = _along(M.T, r, a)
        xm = [edge(am[k] + fac[k] * (r.roll(-1, ax[k]) - r), k) for k in range(d)]
        xf = af[:, :-1] + P * (r[:, 1:] - r[:, :-1])
        y = [0.5 * (v + v.roll(1, ax[k])) for k, v in enumerate(xm)]
        y.append(0.5 * (torch.cat([f0[:, None], xf], 1) + torch.cat([xf, f1[:, None]], 1)))
        q = [v + w for v, w in zip(y, b)]
        u, v = _prox(q[:-1], q[-1])
        bn = [p - w for p, w in zip(q, u + [v])]
        if it == iters - 1:
            uu = sum(p * p for p in u)
            en = torch.where(v > 0, uu / (2 * v.clamp_min(1e-300)), torch.zeros_like(v)).flatten(1).sum(1) / (S * P) * scale
        bb = [2 * p - w for p, w in zip(bn, b)]
        am = [edge(xm[k] - TAU_SIGMA * 0.5 * (bb[k] + bb[k].roll(-1, ax[k])), k) for k in range(d)]
        an = torch.zeros_like(af)
        an[:, :-1] = xf - TAU_SIGMA * 0.5 * (bb[-1][:, :-1] + bb[-1][:, 1:])
        af, b = an, bn
    if take == "path":                                           # (m_0, ..., f) per problem, in solver units
        m = [v.roll(1, ax[k]) if periodic[k] else v.narrow(ax[k], 0, n[k] - 1) for k, v in enumerate(xm)]
        x = torch.cat([v.flatten(1) for v in m + [xf]], 1).flatten()
    else:
        x = xf * scale.view((B,) + (1,) * (d + 1))
    return {"x": x, "energy": float(en.mean())}


def _exact_specify(h, bins, target):
    """Exact counts, strict order by (hue, index), the cyclic shift of least squared circular distance."""
    n = h.numel()
    t = target.double().clamp_min(0)
    xb = t / t.sum() * n
    cnt = xb.floor()
    short = n - int(cnt.sum())
    cnt[torch.sort(xb - cnt, descending=True, stable=True).indices[:short]] += 1
    cnt = cnt.long()
    start = torch.cumsum(cnt, 0) - cnt
    bin_of = torch.repeat_interleave(torch.arange(bins, device="cuda"), cnt)
    q = torch.arange(n, device="cuda")
    y = (bin_of + (q - start[bin_of] + 0.5) / cnt[bin_of]) / bins
    x, idx = torch.sort(h.double(), stable=True)
    yy = torch.cat([y, y])
    cost = torch.empty(n, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 27) // n)
    for s0 in range(0, n, step):
        s = torch.arange(s0, min(n, s0 + step), device="cuda")
        win = yy.as_strided((n + 1, n), (1, 1))[n - s]           # row s: y at (r - s) mod n
        e = (x[None] - win).abs()
        cost[s] = torch.minimum(e, 1 - e).square().sum(1)
    out = torch.empty_like(y)
    out[idx] = y[(q - int(cost.argmin())) % n]
    return out.reshape(h.shape)


def _taps(x, w):
    """3 x 3 x 3 correlation with zero padding: x [N][T][Y][X][ci], w [co][27][ci]."""
    N, T, Y, X, _ = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    out = torch.zeros((N, T, Y, X, w.shape[0]), dtype=x.dtype, device=x.device)
    for k in range(27):
        t, y, c = k // 9, k // 3 % 3, k % 3
        out += xp[:, t:t + T, y:y + Y, c:c + X] @ w[:, k].T
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "image":
        f = _densities(case, seed)
        per = [v == "periodic" for v in case["bc"].split(",")]
        return _exact_solve(f[0], f[1], case["P"], per, case["iters"], case["take"])
    if kind == "hue":
        f = _densities(case, seed)
        return _exact_solve(f[0], f[1], case["P"], [True], case["iters"])
    if kind == "mixed":
        f = _densities(case, seed)
        im, hu = _sizes(case["images"]), _sizes(case["hues"])
        out = [_exact_solve(f[i][0][None], f[i][1][None], P, [False, False, True], case["iters"])
               for i, (_, _, P) in enumerate(im)]
        out += [_exact_solve(f[len(im) + i][0][None], f[len(im) + i][1][None], P, [True], case["iters"])
                for i, (_, P) in enumerate(hu)]
        return [dict(r, x=r["x"][0]) for r in out]
    if kind == "specify":
        h, target = _specify_inputs(case, seed)
        return _exact_specify(h, case["bins"], target)
    vol, x, w, bias, dy = _conv_inputs(case, seed)
    x, w, dy = x.double(), w.double(), dy.double()
    y = (_taps(x, w) + bias.double()).relu()
    g = torch.where(y > 0, dy, torch.zeros_like(dy))
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    N, T, Y, X = vol
    dw = torch.stack([g.flatten(0, 3).T @ xp[:, k // 9:k // 9 + T, k // 3 % 3:k // 3 % 3 + Y, k % 3:k % 3 + X]
                      .flatten(0, 3) for k in range(27)], 1)
    dx = _taps(g, w.flip(1).permute(2, 1, 0).contiguous())
    return {"y": y, "dx": dx, "dw": dw, "db": g.flatten(0, 3).sum(0)}
