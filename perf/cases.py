"""Cases for timing the library: the calls a user of this package makes.

Each case is one pass through the public entry points (``Plan``'s methods,
``reconstruct``) at a size of this repository's own workloads, batch, tests or
a generic one; ``draw`` gives more cases of the same ranges.  Inputs are cone-beam
projections of random balls with 1 % noise (the workloads' recipe with balls in
place of ellipsoids), made on the GPU from the seed alone; calls that start
from filtered projections get them from an FFT in torch.  ``exact`` restates
every path in 64 bits in plain torch and numpy.

Kinds of case:

* ``scan``: filter, then FDK-OD backprojection, from device projections to a
  device volume -- the library's main path.
* ``plain``: filter, then plain FDK, the baseline the method is compared with.
* ``decompose``: the decomposition stage alone (shift and angular decimation).
* ``net``: the decomposition with the learned decimation.
* ``train``: the gradient step of the learned decimation's trainer.
* ``slab``: one slab of a piecemeal reconstruction (the detector rows it needs,
  filtered, decomposed and backprojected on the device).
* ``host``: whole reconstruction from page-locked host projections to a
  page-locked host volume.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1708_07515_gb300 as fd

NOISE = 0.01        # standard deviation over the largest line integral
BALLS = 10
NET_SIZE = 1440
_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _case(kind, N, P, s, D, Nu=0, Nv=0, r=4.0, q="f32", taps="triangle", nz=0, name=None):
    c = {"kind": kind, "N": N, "Nu": Nu or N, "Nv": Nv or N, "P": P, "s": s, "D": D, "r": r, "q": q, "taps": taps,
         "nz": nz}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the batch's smallest volume: a preview or a small specimen, where launches and latency count
        _case("scan", 64, 90, 1, 2, name="scan_64"),
        # the small whole-volume workload
        _case("scan", 128, 128, 2, 2, name="scan_128"),
        # a batch volume whose view count is prime: no decimation, the squares only crop
        _case("scan", 192, 269, 2, 1, name="scan_192_crop"),
        # odd and ragged everything: squares of 62 and 63 voxels, odd detector, a nearer source
        _case("scan", 250, 363, 2, 3, Nu=253, Nv=247, r=2.5, name="scan_250_odd"),
        # the benchmark's workload: a 512^3 scan in float32
        _case("scan", 512, 720, 3, 4, name="scan_512"),
        # the precision form's workload: 1024^3 from bfloat16-stored projections
        _case("scan", 1024, 720, 4, 8, q="bf16", name="scan_1024_bf16"),
        # plain FDK on the 256^3 workload with float16 storage: the yardstick the method's error is judged by
        _case("plain", 256, 360, 2, 4, q="f16", name="plain_256_f16"),
        # the windowed-sinc low-pass (better quality), decomposition stage of the 512^3 scan
        _case("decompose", 512, 720, 3, 4, taps="sinc", name="sinc_512"),
        # the learned decimation at inference, 256^3 workload
        _case("net", 256, 360, 2, 4, name="net_256"),
        # one gradient step of its training on four slices
        _case("train", 256, 360, 2, 4, nz=4, name="train_256"),
        # the paper's scale, piecemeal: one 64-slice slab of 2000^3 from bfloat16-stored rows
        _case("slab", 2000, 720, 5, 16, q="bf16", nz=64, name="slab_2000_bf16"),
        # end to end from page-locked host memory, as a scanner's pipeline calls it
        _case("host", 512, 720, 3, 4, name="host_512"),
    ]


def draw(rng: random.Random):
    """One more case of the ranges above (sizes log-uniform, odd ones among them)."""
    kind = rng.choice(["scan", "scan", "scan", "plain", "decompose", "net", "train", "slab", "host"])
    lo, hi = {"scan": (48, 1024), "plain": (48, 400), "decompose": (64, 640), "net": (48, 300), "train": (48, 300),
              "slab": (300, 2000), "host": (64, 512)}[kind]
    N = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    s = max(0, int(round(math.log2(N / 64.0))) + (1 if rng.random() < 0.3 else 0))
    D = rng.choice([d for d in (1, 2, 3, 4, 6, 8, 16) if d <= 2 * 2 ** s])
    if kind in ("decompose", "net", "train"):
        D = rng.choice([2, 3, 4, 8])
    if kind in ("scan", "slab") and N > 400:
        D = rng.choice([4, 8, 16])
    cap = {"net": 400, "train": 400}.get(kind, 720)
    P = max(1, min(int(round(rng.uniform(0.7, 1.6) * N)), cap) // D) * D
    if N > 700:
        D = max(D, 8)
        P = max(1, P // D) * D
    Nu, Nv = N, N
    if rng.random() < 0.5:
        Nu, Nv = N + rng.randint(-6, 12), N + rng.randint(-6, 12)
    q = "f32" if kind in ("train", "host") else rng.choice(["f32", "f32", "bf16", "f16"])
    taps = "sinc" if kind in ("scan", "decompose", "slab") and D > 1 and rng.random() < 0.3 else "triangle"
    nz = {"train": 4, "slab": rng.choice([17, 32, 48, 64])}.get(kind, 0)
    return _case(kind, N, P, s, D, Nu, Nv, rng.choice([2.0, 3.0, 4.0, 4.0, 6.0]), q, taps, nz)


# ---- inputs -----------------------------------------------------------------

def _slab_z0(c):
    return (c["N"] - c["nz"]) // 3


def _rows(c, z0, nz, slack=0):
    """(first, count) of the detector rows slices z0 .. z0 + nz - 1 can read: row = z / U + (Nv - 1) / 2 with U
    within 1 +- (half-diagonal) / R, and the interpolation's second row."""
    N, R, Nv = c["N"], c["r"] * c["N"], c["Nv"]
    rmax = math.sqrt(2.0) * 0.5 * (N - 1)
    v = [(z - 0.5 * (N - 1)) / (1.0 + sg * rmax / R) + 0.5 * (Nv - 1) for z in (z0, z0 + nz - 1) for sg in (-1, 1)]
    a = min(max(0, math.floor(min(v)) - slack), Nv - 1)
    return a, max(1, min(Nv, math.floor(max(v)) + 2 + slack) - a)


def _slab_rows(c):
    return _rows(c, _slab_z0(c), c["nz"], slack=1)


def _balls(N, seed):
    rng = random.Random(seed)
    out = []
    while len(out) < BALLS:
        c = [rng.uniform(-1, 1) for _ in range(3)]
        if sum(x * x for x in c) <= 1.0:
            out.append([x * 0.35 * N for x in c] + [rng.uniform(0.05, 0.15) * N, rng.uniform(0.1, 1.0)])
    return out


def _projections(c, seed, rows=None):
    """float32 [P][rows][Nu] line integrals of random balls plus noise, on the GPU."""
    N, Nu, P, R = c["N"], c["Nu"], c["P"], c["r"] * c["N"]
    v0, nv = rows or (0, c["Nv"])
    gen = torch.Generator(device="cuda").manual_seed(seed)
    proj = torch.zeros((P, nv, Nu), device="cuda")
    a = (torch.arange(Nu, device="cuda") - 0.5 * (Nu - 1)).view(1, 1, Nu)
    b = (torch.arange(v0, v0 + nv, device="cuda") - 0.5 * (c["Nv"] - 1)).view(1, nv, 1)
    d2 = R * R + a * a + b * b
    balls = _balls(N, seed)
    step = max(1, (1 << 25) // (nv * Nu))
    for k0 in range(0, P, step):
        k1 = min(P, k0 + step)
        beta = 2.0 * math.pi * torch.arange(k0, k1, device="cuda", dtype=torch.float64) / P
        cb, sb = torch.cos(beta), torch.sin(beta)
        for cx, cy, cz, rad, rho in balls:
            dep = (cx * cb + cy * sb).float().view(-1, 1, 1)
            lat = (cy * cb - cx * sb).float().view(-1, 1, 1) - a
            h = cz - b
            dot = dep * R + lat * a + h * b
            t = rad * rad - (dep * dep + lat * lat + h * h - dot * dot / d2)
            proj[k0:k1] += (2.0 * rho) * torch.sqrt(torch.clamp_min(t, 0.0))
    top = float(proj.max())
    for k0 in range(0, P, step):
        n = proj[k0:k0 + step]
        n += (NOISE * max(top, 1.0)) * torch.randn(n.shape, device="cuda", generator=gen)
    return proj


def _ramp_spectrum(L):
    """rfft of the discrete Ram-Lak kernel wrapped onto a circle of length L."""
    n = np.arange(L)
    n = np.minimum(n, L - n)
    h = np.zeros(L)
    h[0] = 0.25
    odd = n % 2 == 1
    h[odd] = -1.0 / (math.pi ** 2 * n[odd].astype(np.float64) ** 2)
    return torch.fft.rfft(torch.from_numpy(h).cuda())


def _filter64(c, proj, rows=None):
    """The FDK filter in 64 bits: float64 [P][rows][Nu]."""
    Nu, R = c["Nu"], c["r"] * c["N"]
    v0, nv = rows or (0, c["Nv"])
    L = 1
    while L < 2 * Nu:
        L *= 2
    H = _ramp_spectrum(L)
    a = (torch.arange(Nu, device="cuda", dtype=torch.float64) - 0.5 * (Nu - 1)).view(1, 1, Nu)
    b = (torch.arange(v0, v0 + nv, device="cuda", dtype=torch.float64) - 0.5 * (c["Nv"] - 1)).view(1, nv, 1)
    w = R / torch.sqrt(R * R + a * a + b * b)
    out = torch.empty(proj.shape, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 26) // (nv * L))
    for k in range(0, proj.shape[0], step):
        out[k:k + step] = torch.fft.irfft(torch.fft.rfft(proj[k:k + step].double() * w, n=L) * H, n=L)[..., :Nu]
    return out


def _filtered(c, seed):
    return _filter64(c, _projections(c, seed)).to(_DTYPE[c["q"]])


def _net_weights(seed):
    """Weights of the size the trained nets have after their first steps."""
    rng = np.random.default_rng(seed)
    return np.concatenate([rng.standard_normal(80) * 0.4, rng.standard_normal(1280) * 0.15,
                           rng.standard_normal(80) * 0.08]).astype(np.float32)


def _train_slices(c, seed):
    """(zs, reference slices, reconstructed slices): the balls' densities, and the same off by a few per cent."""
    N = c["N"]
    rng = random.Random(seed + 1)
    zs = sorted(rng.sample(range(N // 10, N - N // 10), c["nz"]))
    x = torch.arange(N, device="cuda") - 0.5 * (N - 1)
    ref = torch.zeros((len(zs), N, N), device="cuda")
    for cx, cy, cz, rad, rho in _balls(N, seed):
        for i, z in enumerate(zs):
            d = (x.view(1, N) - cx) ** 2 + (x.view(N, 1) - cy) ** 2 + (z - 0.5 * (N - 1) - cz) ** 2
            ref[i] += rho * (d <= rad * rad)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return zs, ref, ref + 0.03 * torch.randn(ref.shape, device="cuda", generator=gen)


def _plan(c, **kw):
    return fd.Plan(c["r"] * c["N"], c["N"], c["Nu"], c["Nv"], c["P"], c["s"], c["D"], qtype=c["q"], taps=c["taps"],
                   **kw)


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = {"case": c, "plan": _plan(c, workspace=kind in ("scan", "host"))}
    plan = st["plan"]
    if kind in ("scan", "plain"):
        st["proj"] = _projections(c, seed)
    elif kind == "host":
        st["proj"] = _projections(c, seed).cpu().pin_memory()
        st["vol"] = torch.empty(plan.vol_shape, pin_memory=True)
    elif kind == "slab":
        st["rows"] = _slab_rows(c)
        st["proj"] = _projections(c, seed, st["rows"])
        st["work"] = torch.empty(max(1, plan.slab_workspace_elems(st["rows"][1])), device="cuda")
    else:
        st["Q"] = _filtered(c, seed)
        if kind == "net":
            plan.set_net(_net_weights(seed))
        if kind == "train":
            st["w"] = torch.from_numpy(_net_weights(seed)).cuda()
            st["zs"], st["ref"], st["vol"] = _train_slices(c, seed)
            st["bands"] = _bands(c, st["zs"])
            st["dS"] = torch.empty(plan.decomposed_shape, device="cuda")
            st["dW"] = torch.empty(NET_SIZE, device="cuda")
            st["err"] = torch.empty(1, device="cuda")
    return st


def _bands(c, zs):
    """Detector rows the slices read, merged into disjoint bands."""
    out = []
    for v0, n in sorted(_rows(c, z, 1) for z in zs):
        if out and v0 <= out[-1][1]:
            out[-1][1] = max(out[-1][1], v0 + n)
        else:
            out.append([v0, v0 + n])
    return out


# ---- one pass ---------------------------------------------------------------

def run(st):
    c, plan = st["case"], st["plan"]
    kind = c["kind"]
    if kind in ("scan", "plain"):
        Q = plan.filter(st["proj"])
        vol = plan.backproject(Q) if kind == "scan" else plan.backproject_plain(Q)
        return {"Q": Q, "vol": vol}
    if kind in ("decompose", "net"):
        return {"S": plan.decompose(st["Q"])}
    if kind == "host":
        return {"vol": fd.reconstruct(plan, st["proj"], st["vol"])}
    if kind == "slab":
        v0, _ = st["rows"]
        Q = plan.filter_rows(st["proj"], v0)
        return {"Q": Q, "vol": plan.backproject_slab(Q, v0, st["work"], _slab_z0(c), c["nz"])}
    for t in (st["dS"], st["dW"], st["err"]):
        t.zero_()
    for i, z in enumerate(st["zs"]):
        plan.net_adjoint(st["vol"][i], st["ref"][i], z, st["dS"], st["err"])
    for lo, hi in st["bands"]:
        plan.net_backward(st["Q"], st["w"], st["dS"], lo, hi, st["dW"])
    return {"dS": st["dS"], "dW": st["dW"], "err": st["err"]}


# ---- what a pass cannot do without -------------------------------------------

UPDATE_FLOP = 14    # one voxel update: row coordinate, three lerps, weighted accumulate


def _filter_flop(c, rows):
    L = 1
    while L < 2 * c["Nu"]:
        L *= 2
    return c["P"] * rows * (5.0 * L * math.log2(L) + 4 * L)   # two real rows share two complex transforms


def work(case):
    c, kind = case, case["kind"]
    N, Nu, Nv, P, D = c["N"], c["Nu"], c["Nv"], c["P"], c["D"]
    es = 4 if c["q"] == "f32" else 2
    H = 2 if c["taps"] == "sinc" else 1
    b = _bounds(c)
    cols = float(b["T"].sum())
    lerp_taps = 3.0 + 4.0 * H               # per shifted sample
    dec = cols * P * Nv * lerp_taps if D > 1 else 0.0
    S_bytes = 4.0 * len(b["T"]) * (P // D) * Nv * ((int(b["T"].max()) + 3) & ~3)
    samples = float(P) * Nv * Nu
    if kind == "scan":
        return {"bytes": samples * (4 + es) + 4.0 * N ** 3, "flops": _filter_flop(c, Nv) + dec +
                UPDATE_FLOP * float(N) ** 3 * (P // D)}
    if kind == "host":
        return {"bytes": samples * 4 + 4.0 * N ** 3, "flops": _filter_flop(c, Nv) + dec +
                UPDATE_FLOP * float(N) ** 3 * (P // D)}
    if kind == "plain":
        return {"bytes": samples * (4 + es) + 4.0 * N ** 3,
                "flops": _filter_flop(c, Nv) + UPDATE_FLOP * float(N) ** 3 * P}
    if kind == "slab":
        rows = _slab_rows(c)[1]
        return {"bytes": float(P) * rows * Nu * (4 + es) + 4.0 * N * N * c["nz"],
                "flops": _filter_flop(c, rows) + dec * rows / Nv + UPDATE_FLOP * float(N) * N * c["nz"] * (P // D)}
    if kind == "decompose":
        return {"bytes": samples * es + S_bytes, "flops": dec}
    if kind == "net":
        return {"bytes": samples * es + S_bytes, "flops": dec + cols * P * Nv * 2.0 * (80 + 1280 + 80.0 / D)}
    rows = min(Nv, c["nz"] * 6)
    return {"bytes": samples * es * rows / Nv + S_bytes + 8.0 * c["nz"] * N * N,
            "flops": c["nz"] * float(N) * N * (P // D) * 20 + cols * P * rows * 6.0 * (80 + 1280)}


# ---- the same in 64 bits -----------------------------------------------------

def _squares(c, s):
    """First and last voxel of every square along one axis."""
    m, N = 1 << s, c["N"]
    first = [(i * N + m - 1) // m for i in range(m + 1)]
    return [(first[i], first[i + 1] - 1) for i in range(m)]


def _bounds(c):
    """Shift centre, crop column, offset and width of every square's shifted rows (the library's rules)."""
    N, P, R = c["N"], c["P"], c["r"] * c["N"]
    cb = np.array([math.cos(2.0 * math.pi * k / P) for k in range(P)])
    sb = np.array([math.sin(2.0 * math.pi * k / P) for k in range(P)])
    uc = 0.5 * (c["Nu"] - 1)
    ax = _squares(c, c["s"])

    def col(x, y):
        return R * (y * cb - x * sb) / (R + x * cb + y * sb) + uc

    phi, w0, T = [], [], []
    for y0, y1 in ax:
        for x0, x1 in ax:
            xs, ys = [v - 0.5 * (N - 1) for v in (x0, x1)], [v - 0.5 * (N - 1) for v in (y0, y1)]
            u = np.stack([col(x, y) for y in ys for x in xs])
            p = col(0.5 * (xs[0] + xs[1]), 0.5 * (ys[0] + ys[1]))
            w = math.floor((u.min(0) - p).min()) - 1
            phi.append(p)
            w0.append(w)
            T.append(math.floor((u.max(0) - p).max()) + 3 - w)
    return {"phi": np.stack(phi), "w0": np.array(w0), "T": np.array(T)}


def _shifted(Q, c, b, q, k):
    """Square q's shifted rows of the views k: float64 [len(k)][rows][T]."""
    Nu, T = c["Nu"], int(b["T"][q])
    pos = b["phi"][q][k] + float(b["w0"][q])
    base = np.floor(pos)
    f = torch.from_numpy(pos - base).cuda().view(-1, 1, 1)
    cols = torch.from_numpy(base.astype(np.int64)).cuda().view(-1, 1) + torch.arange(T, device="cuda").view(1, -1)
    kk = torch.from_numpy(np.asarray(k)).cuda().view(-1, 1, 1)
    rr = torch.arange(Q.shape[1], device="cuda").view(1, -1, 1)

    def at(cc):
        ok = ((cc >= 0) & (cc < Nu)).view(len(k), 1, T)
        return Q[kk, rr, cc.clamp(0, Nu - 1).view(len(k), 1, T)].double() * ok

    a = at(cols)
    return a + f * (at(cols + 1) - a)


def _taps(c):
    D = c["D"]
    if c["taps"] == "triangle":
        return np.array([(D - i) / float(D * D) for i in range(D)])
    i = np.arange(2 * D)
    g = np.sinc(i / D) * 0.5 * (1.0 + np.cos(math.pi * i / (2 * D)))
    return g / (g[0] + 2.0 * g[1:].sum())


def _decimate(x, c):
    """Circular low-pass along the views, every D-th kept: [P][..] -> [P/D][..]."""
    D, P, h = c["D"], c["P"], _taps(c)
    out = torch.zeros((P // D,) + tuple(x.shape[1:]), dtype=torch.float64, device=x.device)
    j = torch.arange(P // D, device=x.device) * D
    for i in range(-len(h) + 1, len(h)):
        out += h[abs(i)] * x[(j + i) % P]
    return out


def _net64(x, w, D):
    """Residual net along the views of x [P][n]: float64 [P/D][n] (w: 1440 weights, float64 torch)."""
    W1, W2, W3 = w[:80].view(16, 5), w[80:1360].view(16, 16, 5), w[1360:].view(16, 5)
    P = x.shape[0]
    a1 = torch.relu(sum(W1[:, m].view(16, 1, 1) * torch.roll(x, 2 - m, 0) for m in range(5)))
    a2 = torch.relu(sum((W2[:, :, m] @ torch.roll(a1, 2 - m, 1).reshape(16, -1)).view(a1.shape) for m in range(5)))
    j = torch.arange(P // D, device=x.device) * D
    return sum((W3[:, m].view(16, 1, 1) * a2[:, (j + m - 2) % P]).sum(0) for m in range(5))


def _gather(S, c, cols, views, xs, ys, zs, v0, col0):
    """(pi / n) sum over the views of U^-2 times the bilinear sample of S [n][rows][cols] at column
    a(x, y) + (Nu - 1) / 2 - col0[view] and row z / U + (Nv - 1) / 2 - v0: float64 [zs][ys][xs]."""
    N, R = c["N"], c["r"] * c["N"]
    n, rows = S.shape[0], S.shape[1]
    beta = [2.0 * math.pi * int(k) / c["P"] for k in views]
    cb = torch.tensor([math.cos(t) for t in beta], dtype=torch.float64, device="cuda").view(-1, 1, 1)
    sb = torch.tensor([math.sin(t) for t in beta], dtype=torch.float64, device="cuda").view(-1, 1, 1)
    h = 0.5 * (N - 1)
    x = torch.arange(xs[0], xs[1] + 1, device="cuda", dtype=torch.float64).view(1, 1, -1) - h
    y = torch.arange(ys[0], ys[1] + 1, device="cuda", dtype=torch.float64).view(1, -1, 1) - h
    z = torch.arange(zs[0], zs[1] + 1, device="cuda", dtype=torch.float64).view(1, -1, 1) - h
    den = R + x * cb + y * sb
    invU = (R / den).view(n, 1, -1)
    u = (R * (y * cb - x * sb) / den).view(n, 1, -1) + 0.5 * (c["Nu"] - 1) - torch.as_tensor(
        col0, dtype=torch.float64, device="cuda").view(n, 1, 1)
    nz, nxy = z.shape[1], u.shape[2]
    grid = torch.empty((n, nz, nxy, 2), dtype=torch.float64, device="cuda")
    grid[..., 0] = u * (2.0 / max(1, cols - 1)) - 1.0
    grid[..., 1] = (z * invU + (0.5 * (c["Nv"] - 1) - v0)) * (2.0 / max(1, rows - 1)) - 1.0
    smp = torch.nn.functional.grid_sample(S.unsqueeze(1), grid, mode="bilinear", padding_mode="zeros",
                                          align_corners=True)
    return ((smp.squeeze(1) * (invU * invU)).sum(0) * (math.pi / n)).view(nz, y.shape[1], x.shape[2])


_BUDGET = 1 << 27    # grid points per gather


def _fdk64(Q, c, v0, z0, nz):
    """Plain FDK (also what FDK-OD with D = 1 computes)."""
    N, P = c["N"], c["P"]
    vol = torch.zeros((nz, N, N), dtype=torch.float64, device="cuda")
    nv = max(1, min(P, _BUDGET // (nz * N * N)))
    zstep = max(1, min(nz, _BUDGET // (N * N)))
    for k0 in range(0, P, nv):
        k = np.arange(k0, min(P, k0 + nv))
        S = Q[k0:k0 + len(k)].double()
        for za in range(0, nz, zstep):
            zb = min(nz, za + zstep)
            vol[za:zb] += _gather(S, c, c["Nu"], k, (0, N - 1), (0, N - 1), (z0 + za, z0 + zb - 1), v0,
                                  np.zeros(len(k))) * (len(k) / P)
    return vol


def _fdkod64(Q, c, v0, z0, nz):
    if c["D"] == 1:
        return _fdk64(Q, c, v0, z0, nz)
    N, P, D = c["N"], c["P"], c["D"]
    b, ax, views = _bounds(c), _squares(c, c["s"]), np.arange(0, P, D)
    vol = torch.empty((nz, N, N), dtype=torch.float64, device="cuda")
    for q in range(len(b["T"])):
        ys, xs = ax[q // len(ax)], ax[q % len(ax)]
        S = _decimate(_shifted(Q, c, b, q, np.arange(P)), c)
        col0 = b["phi"][q][views] + float(b["w0"][q])
        step = max(1, _BUDGET // (len(views) * (ys[1] - ys[0] + 1) * (xs[1] - xs[0] + 1)))
        for za in range(0, nz, step):
            zb = min(nz, za + step)
            vol[za:zb, ys[0]:ys[1] + 1, xs[0]:xs[1] + 1] = _gather(S, c, S.shape[2], views, xs, ys,
                                                                   (z0 + za, z0 + zb - 1), v0, col0)
    return vol


def _decompose64(Q, c, w=None):
    b = _bounds(c)
    stride = (int(b["T"].max()) + 3) & ~3
    Pd, rows = c["P"] // c["D"], Q.shape[1]
    out = torch.zeros((len(b["T"]), Pd, rows, stride), dtype=torch.float64, device="cuda")
    for q, T in enumerate(b["T"]):
        x = _shifted(Q, c, b, q, np.arange(c["P"]))
        out[q, ..., :T] = _decimate(x, c)
        if w is not None:
            step = max(1, (1 << 22) // (c["P"] * int(T)))
            for v in range(0, rows, step):
                xv = x[:, v:v + step]
                out[q, :, v:v + step, :T] += _net64(xv.reshape(c["P"], -1), w, c["D"]).view(Pd, -1, int(T))
    return out


def _train64(c, seed):
    """Gradient of (1/2) sum e^2 over the slices with respect to the decomposed data, of its inner product with the
    net's output with respect to the weights, and sum e^2."""
    Q = _filtered(c, seed)
    w = torch.from_numpy(_net_weights(seed)).cuda().double().requires_grad_(True)
    zs, ref, vol = _train_slices(c, seed)
    e = vol.double() - ref.double()
    b, ax, P, D = _bounds(c), _squares(c, c["s"]), c["P"], c["D"]
    stride, views = (int(b["T"].max()) + 3) & ~3, np.arange(0, P, D)
    dS = torch.zeros((len(b["T"]), len(views), c["Nv"], stride), dtype=torch.float64, device="cuda")
    bands = _bands(c, zs)
    for q, T in enumerate(b["T"]):
        ys, xs = ax[q // len(ax)], ax[q % len(ax)]
        S = torch.zeros((len(views), c["Nv"], int(T)), dtype=torch.float64, device="cuda", requires_grad=True)
        col0 = b["phi"][q][views] + float(b["w0"][q])
        f = sum((e[i, ys[0]:ys[1] + 1, xs[0]:xs[1] + 1] * _gather(S, c, int(T), views, xs, ys, (z, z), 0, col0)[0]).sum()
                for i, z in enumerate(zs))
        dS[q, ..., :T] = torch.autograd.grad(f, S)[0]
        x = _shifted(Q, c, b, q, np.arange(P))
        for lo, hi in bands:
            y = _net64(x[:, lo:hi].reshape(P, -1), w, D)
            (y * dS[q, :, lo:hi, :T].reshape(len(views), -1)).sum().backward()
    return {"dS": dS, "dW": w.grad, "err": (e * e).sum().view(1)}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("scan", "plain"):
        Q = _filter64(c, _projections(c, seed))
        vol = _fdkod64(Q, c, 0, 0, c["N"]) if kind == "scan" else _fdk64(Q, c, 0, 0, c["N"])
        return {"Q": Q, "vol": vol}
    if kind == "host":
        return {"vol": _fdkod64(_filter64(c, _projections(c, seed)), c, 0, 0, c["N"]).cpu()}
    if kind == "slab":
        rows = _slab_rows(c)
        Q = _filter64(c, _projections(c, seed, rows), rows)
        return {"Q": Q, "vol": _fdkod64(Q, c, rows[0], _slab_z0(c), c["nz"])}
    if kind == "decompose":
        return {"S": _decompose64(_filtered(c, seed), c)}
    if kind == "net":
        w = torch.from_numpy(_net_weights(seed)).bfloat16().double().cuda()   # the library stores them as BF16
        return {"S": _decompose64(_filtered(c, seed), c, w)}
    return _train64(c, seed)
