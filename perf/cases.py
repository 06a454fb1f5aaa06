"""The calls whose speed is measured: whole passes through the public entry points, as a user's program makes them.

A pass of a tissue is one ``Grid.step(dt, steps)`` between two looks at the state; the state lives in buffers that the
program owns (``bind_state``), so it is looked at without a copy.  Every program tunes its grid once (``autotune``).
Initial states are tissue in activity: every node is put on the model's own action potential at the phase that waves
from a few seeded sources give it.  Lengths are in nodes, everything else in the model's units."""
import functools
import math

import numpy as np
import torch

from paper_1605_06015_gb300 import bbx

DEV = "cuda"


# ---------------------------------------------------------------------------
# the models, written out in 64 bits
# ---------------------------------------------------------------------------

FHN = dict(eps=0.3, beta=0.71, gamma=0.5)
BARKLEY = dict(a=0.75, b=0.02, eps=0.02)
BR = dict(gNa=4.0, gNaC=0.003, ENa=50.0, gs=0.09)

MODELS = {  # id, variables, parameters, h, dt, D_par, D_perp, speed of the waves (nodes a time unit), their period
    "fhn": (bbx.BBX_FHN, 2, [0.3, 0.71, 0.5], 0.5, 0.01, 1.0, 1.0, 2.0, 24.0),
    "barkley": (bbx.BBX_BARKLEY, 2, [0.75, 0.02, 0.02], 0.3, 0.005, 1.0, 0.25, 14.0, 6.0),
    "br": (bbx.BBX_BR, 8, [4.0, 0.003, 50.0, 0.09], 0.2, 0.02, 0.1, 0.025, 2.0, 500.0),
    "br_mrl": (bbx.BBX_BR_MRL, 11, [4.0, 0.003, 50.0, 0.09], 0.2, 0.02, 0.1, 0.025, 2.0, 500.0),
}


def br_rates(V, exp):
    """alpha and beta of x1, m, h, j, d, f (Beeler and Reuter 1977), 1/ms."""
    xm = V + 47.0
    em = exp(-0.1 * xm)
    a_m = (10.0 if abs(xm) < 1e-9 else -xm / (em - 1.0)) if isinstance(V, float) else torch.where(
        xm.abs() < 1e-9, torch.full_like(V, 10.0), -xm / torch.where(xm.abs() < 1e-9, torch.full_like(V, 2.0), em - 1.0))
    al = [0.0005 * exp(0.083 * (V + 50.0)) / (exp(0.057 * (V + 50.0)) + 1.0), a_m, 0.126 * exp(-0.25 * (V + 77.0)),
          0.055 * exp(-0.25 * (V + 78.0)) / (exp(-0.2 * (V + 78.0)) + 1.0),
          0.095 * exp(-0.01 * (V - 5.0)) / (exp(-0.072 * (V - 5.0)) + 1.0),
          0.012 * exp(-0.008 * (V + 28.0)) / (exp(0.15 * (V + 28.0)) + 1.0)]
    be = [0.0013 * exp(-0.06 * (V + 20.0)) / (exp(-0.04 * (V + 20.0)) + 1.0), 40.0 * exp(-0.056 * (V + 72.0)),
          1.7 / (exp(-0.082 * (V + 22.5)) + 1.0), 0.3 / (exp(-0.1 * (V + 32.0)) + 1.0),
          0.07 * exp(-0.017 * (V + 44.0)) / (exp(0.05 * (V + 44.0)) + 1.0),
          0.0065 * exp(-0.02 * (V + 30.0)) / (exp(-0.2 * (V + 30.0)) + 1.0)]
    return al, be


def br_currents(V, Ca, x1, m3, h, j, d, f, exp, log):
    """(total ionic current, slow inward current)"""
    i_na = (BR["gNa"] * m3 * h * j + BR["gNaC"]) * (V - BR["ENa"])
    i_s = BR["gs"] * d * f * (V + 82.3 + 13.0287 * log(Ca))
    i_x1 = x1 * 0.8 * (exp(0.04 * (V + 77.0)) - 1.0) * exp(-0.04 * (V + 35.0))
    w = V + 23.0
    e = exp(-0.04 * w)
    lin = (5.0 if abs(w) < 1e-9 else 0.2 * w / (1.0 - e)) if isinstance(V, float) else torch.where(
        w.abs() < 1e-9, torch.full_like(V, 5.0), 0.2 * w / torch.where(w.abs() < 1e-9, torch.full_like(V, 2.0), 1.0 - e))
    i_k1 = 0.35 * (4.0 * (exp(0.04 * (V + 85.0)) - 1.0) / (exp(0.08 * (V + 53.0)) + exp(0.04 * (V + 53.0))) + lin)
    return i_na + i_s + i_x1 + i_k1, i_s


@functools.lru_cache(maxsize=None)
def action_potential(model):
    """(table [variables][times] float64, its time step): one cell from its excitation to its return to rest."""
    rows = []
    if model == "fhn":
        u, v, dt, n, keep = 1.8, -0.62, 0.01, 2400, 5
        for k in range(n):
            if k % keep == 0:
                rows.append((u, v))
            u, v = u + dt * (u - u ** 3 / 3 - v) / FHN["eps"], v + dt * FHN["eps"] * (u + FHN["beta"] - FHN["gamma"] * v)
    elif model == "barkley":
        u, v, dt, n, keep = 0.3, 0.0, 0.002, 3000, 5
        for k in range(n):
            if k % keep == 0:
                rows.append((u, v))
            u, v = (u + dt * u * (1 - u) * (u - (v + BARKLEY["b"]) / BARKLEY["a"]) / BARKLEY["eps"], v + dt * (u - v))
    else:
        V, Ca, dt, n, keep = -50.0, 1.8e-7, 0.05, 10000, 4
        g = [0.0055, 0.011, 0.988, 0.975, 0.003, 0.99999]
        for k in range(n):
            if k % keep == 0:
                rows.append([V, Ca] + g)
            al, be = br_rates(V, math.exp)
            i_ion, i_s = br_currents(V, Ca, g[0], g[1] ** 3, *g[2:], math.exp, math.log)
            V, Ca = V - dt * i_ion, Ca + dt * (-1e-7 * i_s + 0.07 * (1e-7 - Ca))
            g = [a / (a + b) + (y - a / (a + b)) * math.exp(-dt * (a + b)) for y, a, b in zip(g, al, be)]
        if model == "br_mrl":
            rows = [[r[0], r[1], r[2], r[4], r[5], r[6], r[7]] +
                    [math.comb(3, k) * r[3] ** k * (1 - r[3]) ** (3 - k) for k in range(4)] for r in rows]
    return np.array(rows).T.copy(), dt * keep


def waves(model, nz, ny, nx, gen):
    """State [variables][nz][ny][nx] float32 on the GPU: waves from three seeded sources."""
    _, S, _, _, _, _, _, speed, period = MODELS[model]
    table, dt = action_potential(model)
    tab = torch.tensor(table, dtype=torch.float32, device=DEV)
    ax = [torch.arange(n, dtype=torch.float32, device=DEV) for n in (nz, ny, nx)]
    at = torch.rand((3, 3), generator=gen).tolist()
    r2 = None
    for cz, cy, cx in at:
        d2 = ((ax[0] - cz * nz) ** 2)[:, None, None] + ((ax[1] - cy * ny) ** 2)[:, None] + (ax[2] - cx * nx) ** 2
        r2 = d2 if r2 is None else torch.minimum(r2, d2)
    t0 = (0.2 + 0.5 * float(torch.rand((), generator=gen))) * max(nx, ny, nz) / speed
    phase = t0 - r2.sqrt_() / speed
    if model.startswith("br"):  # one front: rest ahead of it
        k = (phase / dt).clamp_(-1.0, tab.shape[1] - 1.001)
        k = torch.where(k < 0, torch.full_like(k, tab.shape[1] - 1.001), k)
    else:  # wave trains
        k = torch.remainder(phase, period).div_(dt).clamp_(0.0, tab.shape[1] - 1.001)
    i = k.to(torch.int64)
    w = k - i
    out = torch.empty((S, nz, ny, nx), dtype=torch.float32, device=DEV)
    for v in range(S):
        a = tab[v][i]
        out[v] = a + w * (tab[v][i + 1] - a)
    return out


# ---------------------------------------------------------------------------
# geometry
# ---------------------------------------------------------------------------

def geometry(case, gen):
    """(mask uint8 [nz][ny][nx] or None, fibres float32 [nz][ny][nx][3] or None), on the GPU."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    z, y, x = (torch.arange(n, dtype=torch.float32, device=DEV) for n in (nz, ny, nx))
    z, y = z[:, None, None], y[:, None]
    if case["tissue"] == "shell":  # a ventricle-like thick ellipsoidal shell in a cube, helical fibres through its wall
        s = nx / 512.0
        ao = [200.0 * s, 200.0 * s, 240.0 * s]
        ai = [a - 40.0 * s for a in ao]
        c = (nx - 1) / 2.0
        X, Y, Z = x - c, y - c, z - c
        inside = lambda a: (X / a[0]) ** 2 + (Y / a[1]) ** 2 + (Z / a[2]) ** 2  # noqa: E731
        m = (inside(ao) <= 1.0) & (inside(ai) > 1.0)
        idx = m.nonzero()
        pz, py, px = (idx[:, k].to(torch.float32) - c for k in range(3))
        lo, hi = torch.zeros_like(px), torch.ones_like(px)
        for _ in range(20):  # depth in the wall: the member of the family of ellipsoids through the node
            d = 0.5 * (lo + hi)
            r = sum((p / (a + d * (b - a))) ** 2 for p, a, b in zip((px, py, pz), ai, ao))
            hi, lo = torch.where(r <= 1.0, d, hi), torch.where(r <= 1.0, lo, d)
        d = 0.5 * (lo + hi)
        n = torch.stack([p / (a + d * (b - a)) ** 2 for p, a, b in zip((px, py, pz), ai, ao)], 1)
        n /= n.norm(dim=1, keepdim=True)
        circ = torch.stack([-n[:, 1], n[:, 0], torch.zeros_like(px)], 1)
        circ = torch.where(circ.norm(dim=1, keepdim=True) > 1e-6, circ, torch.tensor([1.0, 0.0, 0.0], device=DEV))
        circ /= circ.norm(dim=1, keepdim=True)
        alpha = torch.deg2rad(-60.0 + 120.0 * d)[:, None]
        fib = torch.zeros((nz, ny, nx, 3), dtype=torch.float32, device=DEV)
        fib[m] = torch.cos(alpha) * circ + torch.sin(alpha) * torch.linalg.cross(n, circ)
        return m.to(torch.uint8), fib
    mask = fib = None
    ph = (6.28 * torch.rand(6, generator=gen)).tolist()
    if case["tissue"] == "block":  # a block of tissue with a wavy surface and a cavity
        w = 0.12 * (torch.sin(x * (9.0 / nx) + ph[0]) + torch.sin(y * (8.0 / ny) + ph[1]) + torch.sin(z * (7.0 / nz) + ph[2]))
        r = (((x / nx - 0.5) / 0.5) ** 4 + ((y / ny - 0.5) / 0.5) ** 4 + ((z / max(nz, 2) - 0.5) / 0.55) ** 4) + w
        cav = ((x - 0.6 * nx) / (0.15 * nx)) ** 2 + ((y - 0.4 * ny) / (0.15 * ny)) ** 2 + ((z - 0.5 * nz) / (0.3 * nz + 1)) ** 2
        mask = ((r < 0.8) & (cav > 1.0)).to(torch.uint8)
    if case["fibres"] == "rotational":  # in the x-y plane, turning 120 degrees through z
        th = torch.deg2rad(120.0 * z / max(nz - 1, 1)) + ph[3]
        fib = torch.stack(torch.broadcast_tensors(torch.cos(th), torch.sin(th), torch.zeros((), device=DEV)), -1)
        fib = fib.expand(nz, ny, nx, 3).contiguous()
    elif case["fibres"] == "smooth":  # turning in every direction
        th = 0.6 * torch.sin(0.09 * x + ph[3]) + 0.4 * torch.cos(0.07 * y + ph[4]) + 0.03 * z
        el = 0.5 * torch.cos(0.05 * z + 0.04 * x + ph[5]) + 0.0 * y
        fib = torch.stack([torch.cos(th) * torch.cos(el), torch.sin(th) * torch.cos(el), torch.sin(el)], -1)
    return mask, fib


def host(t):
    return None if t is None else t.cpu().numpy()


def seeded(seed):
    return torch.Generator().manual_seed(1605 + int(seed))


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def tissue(model, nx, ny, nz, steps, tissue="full", fibres="none", scheme="unsplit", tab=False, gates="fp32",
           resident=False, **more):
    return dict(kind="tissue", model=model, nx=nx, ny=ny, nz=nz, steps=steps, tissue=tissue, fibres=fibres, scheme=scheme,
                tab=tab, gates=gates, resident=resident, **more)


def listed():
    return [
        # one small 2D experiment: launches and latency
        tissue("fhn", 200, 200, 1, 20, name="sheet_200"),
        # the same for a parameter scan on the desk: many steps between two looks, sheet kept on the chip
        tissue("fhn", 200, 200, 1, 200, resident=True, name="sheet_200_resident"),
        # spiral turbulence on a very large sheet
        tissue("fhn", 8192, 8192, 1, 4, name="sheet_8192"),
        # the usual 3D slab: scroll waves under rotational anisotropy
        tissue("barkley", 256, 256, 64, 10, fibres="rotational", name="slab_barkley"),
        # the same physics at the size of a whole wall
        tissue("barkley", 512, 512, 256, 2, fibres="rotational", name="slab_barkley_large"),
        # an irregular piece of tissue from an image: odd sides, voids, fibres turning everywhere
        tissue("barkley", 211, 163, 97, 10, tissue="block", fibres="smooth", name="block_masked"),
        # the anatomical run: ventricle-like shell, ionic cell model
        tissue("br", 512, 512, 512, 2, tissue="shell", fibres="helical", name="shell_br"),
        # the ionic cell model on the slab
        tissue("br", 256, 256, 64, 10, fibres="rotational", name="slab_br"),
        # the shell at half the resolution, tabulated rates and 16-bit gates: the fastest setting for long runs
        tissue("br", 256, 256, 256, 10, tissue="shell", fibres="helical", tab=True, gates="unorm16", name="shell_br_tab16"),
        # a parameter sweep: many tissues of uneven sizes together
        dict(kind="batch", sheets=192, blocks=64, steps=16, name="batch_256"),
        # looking at a run: one colour frame and the filaments' tips
        dict(kind="frame", nx=256, ny=256, nz=64, name="frame_and_tips"),
        # learning the reaction from sampled pairs: minibatch steps
        dict(kind="train", pairs=1 << 20, batch=4096, steps=20, name="train"),
    ]


def draw(rng):
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    pick = rng.random()
    if pick < 0.2:
        nx, ny = log(64, 8192), log(64, 8192)
        small = nx * ny <= 90000 and min(nx, ny) >= 64
        return tissue(rng.choice(["fhn", "fhn", "barkley"]), nx, ny, 1, 4 if nx * ny > 4000000 else 20,
                      fibres=rng.choice(["none", "none", "rotational"]) if not small else "none",
                      resident=small and rng.random() < 0.5)
    if pick < 0.65:
        nx, ny, nz = log(48, 512), log(48, 512), log(9, 256)
        model = rng.choice(["barkley", "barkley", "br", "br", "br_mrl", "fhn"])
        big = nx * ny * nz > 8000000
        return tissue(model, nx, ny, nz, 2 if big else 10, fibres=rng.choice(["none", "rotational", "rotational", "smooth"]),
                      tissue=rng.choice(["full", "full", "block"]), tab=model == "br" and rng.random() < 0.4,
                      scheme="lie" if model in ("fhn", "barkley") and rng.random() < 0.25 else "unsplit",
                      gates="unorm16" if model == "br" and rng.random() < 0.25 else "fp32")
    if pick < 0.8:
        n = log(96, 448)
        return tissue("br", n, n, n, 2 if n > 256 else 10, tissue="shell", fibres="helical", tab=rng.random() < 0.5,
                      gates=rng.choice(["fp32", "fp32", "unorm16"]))
    if pick < 0.9:
        return dict(kind="batch", sheets=log(8, 192), blocks=log(4, 64), steps=16)
    if pick < 0.95:
        return dict(kind="frame", nx=log(64, 512), ny=log(64, 512), nz=log(8, 128))
    return dict(kind="train", pairs=log(1 << 16, 1 << 22), batch=log(256, 16384), steps=rng.randint(4, 24))


# ---------------------------------------------------------------------------
# preparation
# ---------------------------------------------------------------------------

def tissue_inputs(case, seed):
    gen = seeded(seed)
    mask, fib = geometry(case, gen)
    return mask, fib, waves(case["model"], case["nz"], case["ny"], case["nx"], gen)


def prepare_tissue(case, seed):
    mask, fib, st = tissue_inputs(case, seed)
    model, S, params, h, dt, d_par, d_perp, _, _ = MODELS[case["model"]]
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    G = bbx.Grid(nx, ny, nz, h, host(mask))
    G.set_fibres(host(fib), d_par, d_perp)
    G.set_ionic_model(model, params)
    G.set_timestep(dt)
    if case["tab"]:
        G.set_tabulation(True)
    if case["scheme"] == "lie":
        G.set_scheme(bbx.BBX_SCHEME_LIE)
    px = G.get_info()["px"]
    g16 = case["gates"] == "unorm16"
    bufs = [torch.zeros((S, nz, ny, px), dtype=torch.float32, device=DEV) for _ in range(2)]
    G.bind_state(*bufs)
    if g16:
        G.set_gate_storage(bbx.BBX_GATES_UNORM16)
    G.autotune(dt)
    views = []
    for b in bufs:
        if g16:  # V and Ca, then the six gates as 16-bit codes
            n = nz * ny * px
            flat = b.view(-1)
            gates = flat[2 * n:5 * n].view(torch.int16).view(6, nz, ny, px)[..., :nx]
            code = (st[2:].clamp(0, 1) * 65535.0).round_().to(torch.int32)
            gates.copy_(torch.where(code > 32767, code - 65536, code))
            first = flat[:2 * n].view(2, nz, ny, px)[..., :nx]
            first.copy_(st[:2])
            views.append((first, gates))
        else:
            b[..., :nx].copy_(st)
            views.append((b[..., :nx],))
    if case["resident"]:
        G.set_resident(True)
    torch.cuda.synchronize()
    return dict(kind="tissue", G=G, bufs=bufs, views=views, dt=dt, steps=case["steps"], done=0)


def batch_members(case, seed):
    """(model, nx, ny, nz, D, parameters) of every tissue of the sweep: its sizes belong to the case."""
    r, sizes = np.random.default_rng(1605 + int(seed)), np.random.default_rng(1000 * case["sheets"] + case["blocks"])
    out = []
    for i in range(case["sheets"] + case["blocks"]):
        k = r.uniform(0.8, 1.2, 4)
        if i < case["sheets"]:
            nx, ny = (int(v) for v in sizes.integers(64, 513, 2))
            out.append(("fhn", nx, ny, 1, k[0], [0.3 * k[1], 0.71 * k[2], 0.5 * k[3]]))
        else:
            nx, ny, nz = (int(v) for v in sizes.integers(64, 129, 3))
            out.append(("barkley", nx, ny, nz, k[0], [0.75 * k[1], 0.02 * k[2], 0.02 * k[3]]))
    return out


def batch_layout(members):
    at, n = [], 0
    for _, nx, ny, nz, _, _ in members:
        px = (nx + 31) // 32 * 32
        at.append((n, px))
        n += 2 * nz * ny * px
    return at, n


def prepare_batch(case, seed):
    gen = seeded(seed)
    members = batch_members(case, seed)
    at, n = batch_layout(members)
    flats = [torch.zeros(n, dtype=torch.float32, device=DEV) for _ in range(2)]
    grids = []
    for (model, nx, ny, nz, D, params), (o, px) in zip(members, at):
        mid, S, _, h, dt, _, _, _, _ = MODELS[model]
        G = bbx.Grid(nx, ny, nz, h)
        G.set_fibres(None, D, D)
        G.set_ionic_model(mid, params)
        G.set_timestep(dt)
        G.bind_state(*(f[o:o + 2 * nz * ny * px] for f in flats))
        grids.append(G)
    B = bbx.Batch(grids)
    B.autotune()
    for f in flats:
        f.zero_()
    for (model, nx, ny, nz, _, _), (o, px) in zip(members, at):
        st = waves(model, nz, ny, nx, gen)
        for f in flats:
            f[o:o + 2 * nz * ny * px].view(2, nz, ny, px)[..., :nx].copy_(st)
    torch.cuda.synchronize()
    return dict(kind="batch", B=B, flats=flats, steps=case["steps"], done=0)


def prepare_frame(case, seed):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    gen = seeded(seed)
    st = waves("barkley", nz, ny, nx, gen)
    # broken fronts: the second variable's waves come from other sources, so the isolines cross
    st[1] = waves("barkley", nz, ny, nx, gen)[1]
    mid, S, params, h, dt, _, _, _, _ = MODELS["barkley"]
    G = bbx.Grid(nx, ny, nz, h)
    G.set_ionic_model(mid, params)
    px = G.get_info()["px"]
    bufs = [torch.zeros((S, nz, ny, px), dtype=torch.float32, device=DEV) for _ in range(2)]
    G.bind_state(*bufs)
    for b in bufs:
        b[..., :nx].copy_(st)
    out = torch.zeros(3 * nx * ny * nz, dtype=torch.uint8, device=DEV)
    xyz = torch.zeros((16384, 3), dtype=torch.float32, device=DEV)  # room for every tip; unused rows stay 0
    along = torch.tensor([1.0, 1e4, 1e9], dtype=torch.float64, device=DEV)
    torch.cuda.synchronize()
    return dict(kind="frame", G=G, bufs=bufs, out=out, xyz=xyz, along=along)


def train_inputs(case, seed):
    """(states, increments) [pairs][8]: cells along the action potential, each with a little of its own."""
    gen = torch.Generator(device=DEV).manual_seed(1605 + int(seed))
    table, dt = action_potential("br")
    tab = torch.tensor(table, dtype=torch.float32, device=DEV)
    n = case["pairs"]
    k = torch.rand(n, generator=gen, device=DEV) * (tab.shape[1] - 2)
    i = k.to(torch.int64)
    w = (k - i)[:, None]
    a, b = tab.T[i], tab.T[i + 1]
    x = a + w * (b - a)
    t = (b - a) * (0.02 / dt) * (1.0 + 0.05 * torch.randn((n, 8), generator=gen, device=DEV))
    return x.contiguous(), t.contiguous()


def train_norm(x, t):
    xd, td = x.double(), t.double()
    sd = lambda v: v.std(0, correction=0).clamp_min(1e-12)  # noqa: E731
    parts = [xd.mean(0), sd(xd), td.mean(0), sd(td), xd.amin(0), xd.amax(0)]
    return torch.cat(parts).to(torch.float32).cpu().numpy()


def train_params(seed):
    r = np.random.default_rng(int(seed))
    s8, s64 = 8 ** -0.5, 0.125
    parts = [r.uniform(-s8, s8, 512), np.zeros(64), r.uniform(-s64, s64, 4096), np.zeros(64), r.uniform(-s64, s64, 512), np.zeros(8)]
    return np.concatenate(parts).astype(np.float32)


def prepare_train(case, seed):
    x, t = train_inputs(case, seed)
    m = bbx.bbx_mlp_create(1)
    bbx.bbx_mlp_set_params(m, train_params(seed))
    bbx.bbx_mlp_set_normalization(m, train_norm(x, t))
    return dict(kind="train", m=Network(m), x=x, t=t, case=dict(case))


class Network:
    """Owner of a network handle."""

    def __init__(self, m):
        self.m = m

    def __del__(self):
        bbx.bbx_mlp_destroy(self.m)


def prepare(case, seed):
    return {"tissue": prepare_tissue, "batch": prepare_batch, "frame": prepare_frame, "train": prepare_train}[case["kind"]](case, seed)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    if s["kind"] == "tissue":
        s["G"].step(s["dt"], s["steps"])
        s["done"] += s["steps"]
        v = s["views"][s["done"] & 1]
        if len(v) == 1:
            return v[0]
        gates = v[1].to(torch.float32)  # the codes as the numbers they stand for
        return [v[0], torch.where(gates < 0, gates + 65536.0, gates) * (1.0 / 65535.0)]
    if s["kind"] == "batch":
        s["B"].step(s["steps"])
        s["done"] += s["steps"]
        return s["flats"][s["done"] & 1]
    if s["kind"] == "frame":
        s["G"].ppm_frame([0, 1, -1], [0.0, 0.0, 0.0], [1.0, 0.8, 1.0], s["out"])
        n = s["G"].phase_singularities(0, 0.5, 1, 0.35, s["xyz"], s["xyz"].shape[0])
        return [s["out"], n, s["xyz"][torch.argsort(s["xyz"].double() @ s["along"])]]  # the filaments along z
    c = s["case"]
    bbx.bbx_mlp_train(s["m"].m, s["x"], s["t"], c["pairs"], c["batch"], c["steps"], 1e-3, seed=7)
    return bbx.bbx_mlp_get_params(s["m"].m)


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------

REACTION = {"fhn": 12, "barkley": 11, "br": 330, "br_mrl": 130}  # operations of a node's reaction


def work(case):
    """Bytes: a step reads the state of the step before (and the tissue's fibres and mask) once and writes the new state once."""
    if case["kind"] == "tissue":
        n = case["nx"] * case["ny"] * case["nz"]
        masked = case["tissue"] != "full"
        share = {"full": 1.0, "shell": 0.14, "block": 0.62}[case["tissue"]]
        S = MODELS[case["model"]][1]
        state = 4.0 * S if case["gates"] == "fp32" else 20.0
        aniso = case["fibres"] != "none"
        flops = (60 if aniso else 12) + (75 if case["tab"] else REACTION[case["model"]])
        return {"bytes": case["steps"] * n * share * (2 * state + 12 * aniso + masked), "flops": case["steps"] * n * share * flops}
    if case["kind"] == "batch":
        n = case["sheets"] * 288.0 ** 2 + case["blocks"] * 96.0 ** 3
        return {"bytes": case["steps"] * n * 16, "flops": case["steps"] * n * 24}
    if case["kind"] == "frame":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": n * 11.0, "flops": n * 20.0}
    return {"bytes": case["steps"] * case["batch"] * 64.0, "flops": case["steps"] * case["batch"] * 3 * 2 * 5120.0}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

class Diffusion:
    """(L u) of the 19-point operator in 64 bits: faces D_kk/h^2 plus the tensor's divergence, edges D_jk/(2 h^2); a void
    or missing neighbour takes no part, and in the divergence its tensor is the node's own."""

    def __init__(self, mask, fib, h, d_par, d_perp, shape):
        nz, ny, nx = shape
        one = torch.ones(shape, dtype=torch.bool, device=DEV)
        self.shape, self.psi = shape, one if mask is None else mask != 0
        self.psi_p = torch.nn.functional.pad(self.psi, (1, 1, 1, 1, 1, 1))
        self.h2, self.fib, self.d = h * h, None, (d_par, d_perp)
        if fib is not None:
            f = fib.movedim(-1, 0).double()
            r = f.square().sum(0).sqrt()
            f /= torch.where(r > 0, r, torch.ones_like(r))
            self.fib = f
            fp = torch.nn.functional.pad(f, (1, 1, 1, 1, 1, 1))
            self.sums = torch.zeros_like(f)
            for j, off in enumerate([(1, 0, 0), (0, 1, 0), (0, 0, 1)]):
                for sgn in (1, -1):
                    o = [sgn * v for v in off]
                    q = torch.where(self.at(self.psi_p, *o), torch.stack([self.at(fp[k], *o) for k in range(3)]), f)
                    for k in range(3):
                        self.sums[k] += sgn * q[j] * q[k]

    def at(self, a, dx, dy, dz):
        nz, ny, nx = self.shape
        return a[1 + dz:1 + dz + nz, 1 + dy:1 + dy + ny, 1 + dx:1 + dx + nx]

    def __call__(self, u):
        up = torch.nn.functional.pad(u, (1, 1, 1, 1, 1, 1))
        diff = lambda *o: torch.where(self.at(self.psi_p, *o), self.at(up, *o) - u, 0.0)  # noqa: E731
        axes = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
        neg = lambda o: tuple(-v for v in o)  # noqa: E731
        d_par, d_perp = self.d
        if self.fib is None:
            return sum(diff(*o) + diff(*neg(o)) for o in axes) * (d_par / self.h2)
        f, dd = self.fib, d_par - d_perp
        L = torch.zeros_like(u)
        for k, o in enumerate(axes):
            L += (d_perp + dd * f[k] * f[k]) * (diff(*o) + diff(*neg(o)))
            both = self.at(self.psi_p, *o) & self.at(self.psi_p, *neg(o))
            L += torch.where(both, 0.25 * dd * self.sums[k] * (self.at(up, *o) - self.at(up, *neg(o))), 0.0)
        for j in range(3):
            for k in range(j):
                p = tuple(a + b for a, b in zip(axes[j], axes[k]))
                q = tuple(a - b for a, b in zip(axes[j], axes[k]))
                L += 0.5 * dd * f[j] * f[k] * (diff(*p) + diff(*neg(p)) - diff(*q) - diff(*neg(q)))
        return L / self.h2


def react(model, params, y, source, dt):
    """One kinetics step from y [variables][nodes] with the source on V."""
    if model == "fhn":
        eps, beta, gamma = params
        u, v = y
        return torch.stack([u + dt * ((u - u ** 3 / 3 - v) / eps + source), v + dt * eps * (u + beta - gamma * v)])
    if model == "barkley":
        a, b, eps = params
        u, v = y
        return torch.stack([u + dt * (u * (1 - u) * (u - (v + b) / a) / eps + source), v + dt * (u - v)])
    V, Ca = y[0], y[1]
    al, be = br_rates(V, torch.exp)
    A = [torch.exp(-dt * (p + q)) for p, q in zip(al, be)]
    B = [p / (p + q) * (1 - a) for p, q, a in zip(al, be, A)]
    if model == "br":
        i_ion, i_s = br_currents(V, Ca, y[2], y[3] ** 3, y[4], y[5], y[6], y[7], torch.exp, torch.log)
        gates = [a * g + b for a, g, b in zip(A, y[2:], B)]
    else:  # x1, h, j, d, f by themselves; three independent activation subunits: P0..P3
        i_ion, i_s = br_currents(V, Ca, y[2], y[10], y[3], y[4], y[5], y[6], torch.exp, torch.log)
        order = [0, 2, 3, 4, 5]
        gates = [A[q] * y[2 + k] + B[q] for k, q in enumerate(order)]
        stay, go = A[1] + B[1], B[1]  # open -> open, closed -> open
        new = [torch.zeros_like(V) for _ in range(4)]
        for j in range(4):  # j of the three are open before
            dist = [torch.ones_like(V)]
            for s in range(3):
                p = stay if s < j else go
                dist = [(dist[k] * (1 - p) if k < len(dist) else 0) + (dist[k - 1] * p if k else 0) for k in range(len(dist) + 1)]
            for k in range(4):
                new[k] += dist[k] * y[7 + j]
        gates += new
    return torch.stack([V + dt * (source - i_ion), Ca + dt * (-1e-7 * i_s + 0.07 * (1e-7 - Ca))] + gates)


def advance(model, params, st, op, dt, steps, lie):
    """`steps` steps of the state [variables][nz][ny][nx] in 64 bits; void nodes stay as they are."""
    tis = op.psi.reshape(-1).nonzero()[:, 0]
    chunk = 1 << 22
    for _ in range(steps):
        L = op(st[0]).reshape(-1)
        flat = st.view(st.shape[0], -1)
        for c in range(0, tis.numel(), chunk):
            t = tis[c:c + chunk]
            y, src = flat[:, t], L[t]
            if lie:
                y[0] += dt * src
                src = torch.zeros_like(src)
            flat[:, t] = react(model, params, y, src, dt)
    return st


def exact_train(case, seed):
    x, t = train_inputs(case, seed)
    norm = torch.tensor(train_norm(x, t), dtype=torch.float64, device=DEV).view(6, 8)
    P = torch.tensor(train_params(seed), dtype=torch.float64, device=DEV)
    cut = [512, 64, 4096, 64, 512, 8]
    M, V = torch.zeros_like(P), torch.zeros_like(P)
    n, batch = case["pairs"], case["batch"]

    def mix(z):
        z = z + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))

    for step in range(1, case["steps"] + 1):
        with np.errstate(over="ignore"):
            i = np.arange(batch, dtype=np.uint64) + np.uint64(step * 0x100000001B3)
            rows = (mix(np.uint64(7) ^ i) % np.uint64(n)).astype(np.int64)
        r = torch.from_numpy(rows).to(DEV)
        xs, ts = (x[r].double() - norm[0]) / norm[1], (t[r].double() - norm[2]) / norm[3]
        W1, b1, W2, b2, W3, b3 = P.split(cut)
        W1, W2, W3 = W1.view(64, 8), W2.view(64, 64), W3.view(8, 64)
        z1 = xs @ W1.T + b1
        h1 = z1.clamp_min(0)
        z2 = h1 @ W2.T + b2
        h2 = z2.clamp_min(0)
        dy = 2.0 / (batch * 8) * (h2 @ W3.T + b3 - ts)
        d2 = (dy @ W3) * (z2 > 0)
        d1 = (d2 @ W2) * (z1 > 0)
        g = torch.cat([(d1.T @ xs).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), (dy.T @ h2).reshape(-1), dy.sum(0)])
        M, V = 0.9 * M + 0.1 * g, 0.999 * V + 0.001 * g * g
        P = P - 1e-3 * (M / (1 - 0.9 ** step)) / ((V / (1 - 0.999 ** step)).sqrt() + 1e-8)
    return P


def exact(case, seed):
    if case["kind"] == "tissue":
        mask, fib, st = tissue_inputs(case, seed)
        _, _, params, h, dt, d_par, d_perp, _, _ = MODELS[case["model"]]
        op = Diffusion(mask, fib, h, d_par, d_perp if fib is not None else d_par, (case["nz"], case["ny"], case["nx"]))
        out = advance(case["model"], params, st.double(), op, dt, case["steps"], case["scheme"] == "lie")
        return out if case["gates"] == "fp32" else [out[:2], out[2:]]
    if case["kind"] == "batch":
        gen = seeded(seed)
        members = batch_members(case, seed)
        at, n = batch_layout(members)
        flat = torch.zeros(n, dtype=torch.float64, device=DEV)
        for (model, nx, ny, nz, D, params), (o, px) in zip(members, at):
            _, _, _, h, dt, _, _, _, _ = MODELS[model]
            st = waves(model, nz, ny, nx, gen).double()
            op = Diffusion(None, None, h, D, D, (nz, ny, nx))
            advance(model, params, st, op, dt, case["steps"], False)
            flat[o:o + 2 * nz * ny * px].view(2, nz, ny, px)[..., :nx].copy_(st)
        return flat
    if case["kind"] == "train":
        return exact_train(case, seed)
    return None  # a frame is bytes, and the tips of its cells are counted
