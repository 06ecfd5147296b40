"""The work that a user of this framework has it do, as measurable cases.

A case names a scene (the simulation grid), an image or network call and its
sizes. `prepare` builds what a program has before the call: the grid handle
(fields drawn from the seed), output buffers, a trained depth network. `run`
is one call through the public entry points. The scenes have the shapes of the
framework's own workloads: the uniform wind + shell, the paper's ring, the
cone shock and the clumps-and-cones grid, at sizes that upload quickly.
"""
import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1010_5534_gb300 as air

K_B_KEV = 8.617333262e-8  # Boltzmann constant, keV / K
LOG_T = (4.0, 9.0)        # range of the emission table
N_TBINS = 64


# ------------------------------------------------------------------ cases
def _air(name, scene, view, n0, levels, **kw):
    return dict(dict(name=name, call="air", scene=scene, view=view, n0=n0, levels=levels, xi=0.5,
                     xi_norm=0, refine_on=0, interior=False, mem="device"), **kw)


def listed():
    return [
        # the smallest whole call: a preview image of a small uniform grid
        # (FP64 fields); launches and the latency of each sweep count
        _air("air_wind_16", "wind", "+z", 16, 3, n=64),
        # the paper's own problem (Section 3, Table 1): optically thin ring on
        # an 8^3-brick grid, a small image of many short sweeps
        _air("air_ring_32", "ring", "+x", 32, 4, n=32, brick=8, grid_levels=4),
        # the headline image: face-on cone shock, 106 M cells, 4096^2 equivalent
        _air("air_cone_256", "cone", "+z", 256, 4, n=128, brick=16, grid_levels=3, bands=1),
        # an inclined four-band image read back to page-locked host arrays that
        # the program keeps, with every traced pixel, refined on intensity and
        # column density with the literal norm; an odd base size
        _air("air_cone_inclined_host", "cone", "r11", 101, 4, n=64, brick=16, grid_levels=3, bands=4,
             refine_on=2, xi_norm=1, interior=True, mem="host"),
        # fixed image along x (the axis along which cells are contiguous), odd size
        dict(name="fixed_cone_axis", call="fixed", scene="cone", view="-x", res=2047, n=64, brick=16,
             grid_levels=3, bands=1),
        # fixed image of a uniform grid, inclined, every cell emitting
        dict(name="fixed_wind_inclined", call="fixed", scene="wind", view="r5", res=1000, n=128),
        # fixed five-band spectral image of a hot uniform grid with unequal sides
        dict(name="fixed_hot_bands", call="fixed", scene="hot", view="r8", res=701, n=96, bands=5),
        # several views of one grid in one launch, sixteen bands each (a light curve)
        dict(name="batch_cone_16band", call="batch", scene="cone", view="r3", views=8, n0=128, levels=3,
             xi=0.5, n=64, brick=16, grid_levels=3, bands=16),
        # many bands, large bricks, deep grid refinement around clumps
        _air("air_clumps_32band", "clumps", "r21", 256, 3, n=256, brick=32, grid_levels=4, bands=32),
        # inclined image through the learned depth proposal
        dict(name="learned_cone", call="learned", scene="cone", view="r17", n0=256, levels=4, xi=0.5,
             n=64, brick=16, grid_levels=3, bands=1),
        # training of the depth network: minibatch Adam with a ragged last batch
        dict(name="mlp_train", call="train", samples=200003, batch=8192, epochs=2),
        # the finished image as a finest-level raster, interpolated across levels
        dict(name="raster_cone", call="raster", scene="cone", view="+y", n0=128, levels=4, xi=0.5, n=64,
             brick=16, grid_levels=3, bands=2, mode="bilinear"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid_of(rng, scene):
    if scene == "wind":
        return dict(scene=scene, n=_log(rng, 48, 160))
    if scene == "hot":
        return dict(scene=scene, n=_log(rng, 48, 128), bands=_log(rng, 1, 12))
    if scene == "ring":
        return dict(scene=scene, n=32, brick=8, grid_levels=rng.choice([3, 4]))
    if scene == "cone":
        brick = rng.choice([8, 16])
        return dict(scene=scene, n=rng.choice([48, 64, 80]), brick=brick,
                    grid_levels=rng.choice([2, 3]), bands=_log(rng, 1, 16))
    return dict(scene=scene, n=rng.choice([128, 192]), brick=32, grid_levels=rng.choice([2, 3]),
                bands=_log(rng, 8, 32))


def draw(rng):
    """One more case of the listed ranges."""
    call = rng.choice(["air", "air", "air", "fixed", "fixed", "batch", "learned", "train", "raster"])
    if call == "train":
        return dict(call="train", samples=_log(rng, 20000, 400000), batch=_log(rng, 1000, 16384),
                    epochs=rng.choice([1, 2]))
    scene = rng.choice(["cone", "clumps"] if call in ("batch", "learned") else
                       ["wind", "hot", "ring", "cone", "cone", "clumps"])
    c = dict(_grid_of(rng, scene), call=call)
    sign = rng.choice("+-")
    c["view"] = rng.choice([sign + rng.choice("xyz"), "r%d" % rng.randrange(1000)])
    if call == "fixed":
        c["res"] = _log(rng, 64, 1500)
        return c
    c["levels"] = rng.choice([2, 3, 4])
    c["n0"] = _log(rng, 12, 2048 / 2 ** c["levels"] if call != "batch" else 768 / 2 ** c["levels"])
    c["xi"] = round(rng.uniform(0.2, 0.8), 3)
    if call == "air":
        c.update(xi_norm=rng.choice([0, 0, 1]), refine_on=rng.choice([0, 0, 1, 2]) if scene != "ring" else 0,
                 interior=rng.random() < 0.3,
                 mem=rng.choice(["device", "device", "host"]) if c.get("bands", 1) <= 8 else "device")
    elif call == "batch":
        c["views"] = rng.randrange(2, 9)
    elif call == "raster":
        c["mode"] = rng.choice(["nearest", "bilinear"])
    return c


# ------------------------------------------------------------------ scenes
def _gen(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(1000003 * int(seed) + 12345)


def _emission(bands, e_lo, e_hi=10.0, kappa0=0.3):
    """Band emissivity table (thermal bremsstrahlung shape) and opacity of
    log-spaced bands."""
    edges = e_lo * (e_hi / e_lo) ** (np.arange(bands + 1) / bands)
    T = 10.0 ** (LOG_T[0] + (LOG_T[1] - LOG_T[0]) * np.arange(N_TBINS) / (N_TBINS - 1))
    kT = K_B_KEV * T
    tab = np.sqrt(T / 1e7) * (np.exp(-edges[:-1, None] / kT) - np.exp(-edges[1:, None] / kT))
    kappa = kappa0 * np.sqrt(edges[:-1] * edges[1:]) ** (-8.0 / 3.0)
    return dict(emis_mode=1, lambda_table=tab.astype(np.float32), logT_lo=LOG_T[0], logT_hi=LOG_T[1],
                kappa=kappa)


def _bricks(n, brick, levels, half_width, refine):
    """Leaf bricks of a block-AMR box [-half_width, half_width]^3: a brick is
    split while refine(centres, edge, level) says so."""
    nb0 = n // brick
    hf = 2.0 * half_width / (n << levels)
    z, y, x = np.meshgrid(*[np.arange(nb0)] * 3, indexing="ij")
    cur = np.stack([x.ravel(), y.ravel(), z.ravel()], axis=1).astype(np.int64) * (brick << levels)
    lev_of, org = [], []
    kids = np.array([[i & 1, (i >> 1) & 1, i >> 2] for i in range(8)], dtype=np.int64)
    for lev in range(levels + 1):
        S = brick << (levels - lev)
        split = refine(-half_width + (cur + S / 2.0) * hf, S * hf) if lev < levels else np.zeros(len(cur), bool)
        keep = cur[~split]
        lev_of.append(np.full(len(keep), lev, np.int32))
        org.append(keep)
        cur = (cur[split][None] + kids[:, None] * (S // 2)).reshape(-1, 3)
        if len(cur):
            cur = cur[np.lexsort((cur[:, 0], cur[:, 1], cur[:, 2]))]
    return np.concatenate(lev_of), np.concatenate(org).astype(np.int32)


def _cone_distance(x, y, z, apex=(-0.5, 0.0, 0.0), sign=1.0, xp=torch):
    a = sign * (x - apex[0])
    r = xp.sqrt((y - apex[1]) ** 2 + (z - apex[2]) ** 2)
    ct, st = math.cos(math.radians(30.0)), math.sin(math.radians(30.0))
    on = a * ct + r * st >= 0.0
    return xp.where(on, r * ct - a * st, xp.sqrt(a * a + r * r)), on


def _cone_near(c, edge, apex=(-0.5, 0.0, 0.0), sign=1.0):
    d, _ = _cone_distance(c[:, 0], c[:, 1], c[:, 2], apex, sign, np)
    return np.abs(d) <= math.sqrt(3.0) * edge / 2 + 0.02


@functools.lru_cache(maxsize=8)
def _cone_bricks(n, brick, levels):
    return _bricks(n, brick, levels, 1.0, _cone_near)


@functools.lru_cache(maxsize=4)
def _ring_bricks(n, brick, levels):
    def refine(c, edge):
        r, ax = np.hypot(c[:, 1], c[:, 2]), np.abs(c[:, 0])
        inside = (ax <= 0.5) & (r >= 3.5) & (r <= 4.0)
        out = np.hypot(np.maximum(ax - 0.5, 0), np.maximum(np.maximum(3.5 - r, r - 4.0), 0))
        d = np.where(inside, np.minimum(np.minimum(0.5 - ax, r - 3.5), 4.0 - r), out)
        return d <= math.sqrt(3.0) * 0.5 * edge
    return _bricks(n, brick, levels, 5.0, refine)


def _amr_fields(lev, org, n, brick, levels, half_width, fill):
    """rho and T of every leaf brick, `fill(x, y, z, brick range)` at its cell
    centres, made on the GPU a slice of bricks at a time."""
    hf = 2.0 * half_width / (n << levels)
    nb = len(lev)
    rho = np.empty((nb, brick, brick, brick), np.float32)
    temp = np.empty_like(rho)
    o = torch.from_numpy(org).cuda().double()
    step = torch.from_numpy(1 << (levels - lev.astype(np.int64))).cuda().double()
    off = torch.arange(brick, device="cuda", dtype=torch.float64) + 0.5
    per = max(1, (1 << 25) // brick ** 3)
    for a in range(0, nb, per):
        b = min(nb, a + per)
        c = [(-half_width + (o[a:b, k:k + 1] + off * step[a:b, None]) * hf).float() for k in range(3)]
        r, t = fill(c[0][:, None, None, :], c[1][:, None, :, None], c[2][:, :, None, None], a, b)
        rho[a:b], temp[a:b] = r.cpu().numpy(), t.cpu().numpy()
    return rho, temp


def _desc(case, seed):
    """The grid description that air.Grid takes."""
    kind, n = case["scene"], case["n"]
    g = _gen(seed)
    if kind == "wind":   # r^-2 wind with a shell, 5% noise on the shell, j = rho^2, FP64 fields
        c = -1.0 + (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * (2.0 / n)
        r = torch.sqrt(c[:, None, None] ** 2 + c[None, :, None] ** 2 + c[None, None, :] ** 2)
        z = torch.randn((n, n, n), generator=g, device="cuda", dtype=torch.float64)
        shell = torch.exp(-((r - 0.5) ** 2) / (2 * 0.05 ** 2)) * torch.exp(0.05 * z - 0.5 * 0.05 ** 2)
        rho = r.clamp(min=0.05) ** -2 * (1.0 + 9.0 * shell)
        return SimpleNamespace(kind="uniform", n=(n, n, n), lo=(-1.0,) * 3, hi=(1.0,) * 3,
                               rho=rho.cpu().numpy(), temp=None, emis_mode=0, kappa=np.array([3.0 / 87.0]))
    if kind == "hot":    # lognormal density, hot gas everywhere, unequal sides
        nx, ny, nz = n, n + n // 6, n - n // 6
        rho = torch.exp(0.5 * torch.randn((nz, ny, nx), generator=g, device="cuda", dtype=torch.float64))
        temp = 10.0 ** (6.0 + 2.5 * torch.rand((nz, ny, nx), generator=g, device="cuda", dtype=torch.float64))
        return SimpleNamespace(kind="uniform", n=(nx, ny, nz), lo=(-1.0,) * 3, hi=(1.0,) * 3,
                               rho=rho.cpu().numpy(), temp=temp.cpu().numpy(),
                               **_emission(case["bands"], 0.5, kappa0=0.5))
    brick, levels = case["brick"], case["grid_levels"]
    if kind == "ring":   # the paper's ring (lengths 1e17 cm), its density modulated in azimuth
        lev, org = _ring_bricks(n, brick, levels)
        m = int(torch.randint(1, 6, (1,), generator=g, device="cuda"))
        ph = float(torch.rand((1,), generator=g, device="cuda")) * 6.2831853

        def fill(x, y, z, a, b):
            r = torch.sqrt(y * y + z * z)
            inside = (x.abs() < 0.5) & (r >= 3.5) & (r <= 4.0)
            rin = 25.0 / r.clamp(min=0.1) ** 2 * (1.0 + 0.2 * torch.cos(m * torch.atan2(z, y) + ph))
            one = torch.ones_like(x + y + z)
            return torch.where(inside, rin * one, 10.0 * one), torch.where(inside, 1e8 * one, 1e4 * one)

        rho, temp = _amr_fields(lev, org, n, brick, levels, 5.0, fill)
        em = dict(_emission(1, 1.0), kappa=np.zeros(1))
        half = 5.0
    else:                # winds, shocked cone shells, per-cell lognormal clumping
        half = 1.0
        clumps = kind == "clumps"
        if clumps:       # dense clumps that the grid is refined around; the cones at the base
            h = _gen(seed, "cpu")
            k = 60
            cr = torch.exp(torch.empty(k).uniform_(math.log(0.008), math.log(0.03), generator=h)).numpy()
            cc = torch.empty((k, 3)).uniform_(-0.8, 0.8, generator=h).numpy()
            cf = torch.exp(torch.empty(k).uniform_(math.log(10.0), math.log(1000.0), generator=h)).numpy()

            def refine(c, edge):
                q = np.clip(cc[None], c[:, None] - edge / 2, c[:, None] + edge / 2)
                return (((q - cc[None]) ** 2).sum(-1) <= cr ** 2).astype(bool)[:, edge > cr].any(1)

            lev, org = _bricks(n, brick, levels, half, refine)
            cones = (((-0.5, 0.0, 0.0), 1.0), ((0.5, 0.1, 0.0), -1.0))
            stars = ((-0.8, 0.0, 0.0), (0.8, 0.1, 0.0))
            hf = 2.0 / (n << levels)
            blo = -1.0 + org * hf
            bhi = blo + (brick << (levels - lev))[:, None] * hf
        else:
            lev, org = _cone_bricks(n, brick, levels)
            cones, stars = (((-0.5, 0.0, 0.0), 1.0),), ((-0.8, 0.0, 0.0),)

        def fill(x, y, z, a, b):
            rho = sum(torch.sqrt((x - s[0]) ** 2 + (y - s[1]) ** 2 + (z - s[2]) ** 2).clamp(min=0.05) ** -2
                      for s in stars)
            temp = torch.full_like(rho, 1e4)
            for apex, sign in cones:
                d, on = _cone_distance(x, y, z, apex, sign)
                shell = (d.abs() <= 0.02) & on
                rho = torch.where(shell, 4.0 * rho, torch.where((d < -0.02) & on, 0.25 * rho, rho))
                temp = torch.where(shell, torch.full_like(temp, 10.0 ** 7.5), temp)
            if clumps:
                for q in range(len(cr)):
                    p = np.clip(cc[q], blo[a:b], bhi[a:b])
                    hit = np.nonzero(((p - cc[q]) ** 2).sum(1) <= cr[q] ** 2)[0]
                    if len(hit):
                        t = torch.from_numpy(hit).cuda()
                        inn = ((x[t] - cc[q, 0]) ** 2 + (y[t] - cc[q, 1]) ** 2 + (z[t] - cc[q, 2]) ** 2) <= cr[q] ** 2
                        rho[t] = torch.where(inn, rho[t] * float(cf[q]), rho[t])
                        temp[t] = torch.where(inn, torch.full_like(temp[t], 1e5), temp[t])
            w = torch.randn(rho.shape, generator=g, device="cuda")
            return rho * torch.exp(0.3 * w - 0.045), temp

        rho, temp = _amr_fields(lev, org, n, brick, levels, half, fill)
        em = _emission(case["bands"], 1.0 if case["bands"] == 1 else 0.5)
    return SimpleNamespace(kind="amr", n=(n,) * 3, lo=(-half,) * 3, hi=(half,) * 3, rho=rho, temp=temp,
                           brick=brick, max_level=levels, brick_level=lev, brick_origin=org, **em)


def _view(case, k=0):
    """"+z" and the like: face-on; "r<number>": an inclined direction. View k
    of a batch; those after a face-on one are inclined."""
    v, half = case["view"], 5.0 if case["scene"] == "ring" else 1.0
    v = "r0" if k and v[0] != "r" else v
    if v[0] == "r":
        d = np.random.RandomState(int(v[1:]) + 7919 * k).standard_normal(3)
        d /= np.linalg.norm(d)
        return SimpleNamespace(dir=tuple(d), up=(0.0, 1.0, 0.0), center=(0.0,) * 3, half_extent=half * math.sqrt(3.0))
    d = [0.0] * 3
    d["xyz".index(v[1])] = -1.0 if v[0] == "-" else 1.0
    up = (0.0, 0.0, 1.0) if v[1] == "x" else ((1.0, 0.0, 0.0) if v[1] == "y" else (0.0, 1.0, 0.0))
    return SimpleNamespace(dir=tuple(d), up=up, center=(0.0,) * 3, half_extent=half)


# ------------------------------------------------------------------ prepare and run
FIELDS = ("level", "i", "j", "coldens", "intensity", "p", "band_flux")
BATCH_FIELDS = ("level", "i", "j", "coldens", "intensity", "band_flux")
COUNTS = ("n_out", "n_leaves", "n_rays", "n_steps", "n_sweeps")


def _network(seed):
    g = _gen(seed, "cpu")
    parts = []
    for a, b in ((16, 64), (64, 64), (64, 5)):
        parts += [(torch.randn((a, b), generator=g) * math.sqrt(2.0 / a)).reshape(-1), torch.zeros(b)]
    return torch.cat(parts).numpy()


def _train_data(case, seed):
    g = _gen(seed)
    x = torch.randn((case["samples"], 16), generator=g, device="cuda").to(torch.bfloat16)
    f = x.float()
    y = (f[:, 0] > 0).int() + (f[:, 1] > 0.5).int() + 2 * (f[:, 2] > 1.0).int()
    return x, y.clamp(max=4).int()


def prepare(case, seed):
    if case["call"] == "train":
        x, y = _train_data(case, seed)
        th = _network(seed)
        return dict(case=case, net=air.MLP(th), theta=th, x=x.view(torch.int16), y=y)
    grid = air.Grid(_desc(case, seed))
    s = dict(case=case, grid=grid, view=_view(case))
    if case["call"] == "batch":
        s["views"] = [_view(case, k) for k in range(case["views"])]
    elif case["call"] == "learned":
        # a network trained on two other views of the grid
        xy = [grid.learn_samples(_view(dict(case, view="r%d" % (100 + k))), case["n0"], case["levels"], case["xi"])
              for k in range(2)]
        s["net"] = air.MLP(_network(seed))
        s["net"].train(torch.cat([p[0] for p in xy]), torch.cat([p[1] for p in xy]), batch=2048, epochs=2)
    elif case["call"] == "raster":
        grid.render_adaptive(s["view"], case["n0"], case["levels"], case["xi"], fields=("band_flux",))
    if case["call"] in ("air", "learned", "batch"):
        # the arrays that the program keeps its images in, view after view,
        # with room for any image of these sizes (page-locked for "host")
        s["out"] = [_zeroed(grid.alloc_image(_capacity(case), case.get("mem", "device"),
                                             BATCH_FIELDS if case["call"] == "batch" else FIELDS))
                    for _ in range(case.get("views", 1))]
    return s


def _capacity(case):
    top = (case["n0"] << case["levels"]) ** 2
    return sum((case["n0"] << l) ** 2 for l in range(case["levels"] + 1)) if case.get("interior") else top


def _zeroed(out):
    for v in out.values():
        v.zero_()
    return out


def _keep(out, image):
    for k, v in out.items():
        v[..., :image[k].shape[-1]].copy_(image[k])
    return dict(out, **{k: image[k] for k in COUNTS})


def run(s):
    c = s["case"]
    if c["call"] == "train":
        s["net"].params(set=s["theta"])
        hist = s["net"].train(s["x"], s["y"], batch=c["batch"], epochs=c["epochs"])
        return dict(params=s["net"].params(), loss=hist, logits=s["net"].forward(s["x"]))
    g = s["grid"]
    if c["call"] == "raster":
        return g.raster("I", band=c.get("bands", 1) - 1, mode=c["mode"])
    if c["call"] == "fixed":
        r = g.render_fixed(s["view"], c["res"], fields=("coldens", "intensity", "p", "band_flux"))
        return {k: r[k] for k in ("coldens", "intensity", "p", "band_flux", "n_steps")}
    if c["call"] == "batch":
        r = g.render_batch(s["views"], c["n0"], c["levels"], c["xi"], fields=BATCH_FIELDS)
        r = [_keep(o, v) for o, v in zip(s["out"], r)]
        return [{k: v[k] for k in BATCH_FIELDS + ("n_steps",)} for v in r]
    if c["call"] == "learned":
        r, _ = g.render_learned(s["view"], c["n0"], c["levels"], c["xi"], s["net"], fields=FIELDS)
        return _keep(s["out"][0], r)
    r = g.render_adaptive(s["view"], c["n0"], c["levels"], c["xi"], xi_norm=c["xi_norm"],
                          refine_on=c["refine_on"], include_interior=c["interior"], mem=c["mem"],
                          fields=FIELDS, out=s["out"][0])
    return dict(s["out"][0], **{k: r[k] for k in COUNTS})


# ------------------------------------------------------------------ work
def _cells(case):
    if case["scene"] == "wind":
        return case["n"] ** 3
    if case["scene"] == "hot":
        return case["n"] * (case["n"] + case["n"] // 6) * (case["n"] - case["n"] // 6)
    if case["scene"] == "clumps":  # 60 clumps, some eight bricks of each level around each
        return case["n"] ** 3 + 60 * 8 * case["grid_levels"] * case["brick"] ** 3
    f = _ring_bricks if case["scene"] == "ring" else _cone_bricks
    return len(f(case["n"], case["brick"], case["grid_levels"])[0]) * case["brick"] ** 3


def work(case):
    """Bytes: the cell fields once (4-byte density, 4-byte temperature), each
    output once. Operations: per cell that a ray crosses two for the column
    density and, per band, a table look-up, an exponential and a sum (about
    12). Crossed cells and traced rays of adaptive images are estimates: the
    image decides them."""
    if case["call"] == "train":
        mac = 16 * 64 + 64 * 64 + 64 * 5
        n = case["samples"] * case["epochs"]
        m = float(case["samples"])  # two more for the logits afterwards
        return dict(bytes=36.0 * n + 52.0 * m, flops=6.0 * mac * n + 2.0 * mac * m)
    nb = case.get("bands", 1)
    if case["call"] == "raster":
        px = float((case["n0"] << case["levels"]) ** 2)
        return dict(bytes=4.0 * px + 0.6 * 8.0 * px, flops=(8.0 if case["mode"] == "bilinear" else 0.0) * px)
    inclined = case["view"][0] == "r"
    nf = case["n"] << case.get("grid_levels", 0)
    # cells of a ray through the box: every cell of a uniform grid, fewer where
    # a refined grid is coarse
    per_ray = {"wind": 1.0 * nf, "hot": 1.0 * nf, "ring": 0.24 * nf, "cone": 0.4 * nf,
               "clumps": 1.3 * case["n"]}[case["scene"]]
    if inclined and case["call"] == "fixed":
        per_ray *= 0.45  # the frame is larger than the box
    field = 4.0 if case["scene"] == "wind" else 8.0
    if case["call"] == "fixed":
        rays, per_px = float(case["res"]) ** 2, 8.0 + 4.0 * nb
    else:
        full = float((case["n0"] << case["levels"]) ** 2)
        part = 0.1 if case["scene"] == "ring" else (0.25 if inclined else 0.46)
        rays, per_px = part * full * case.get("views", 1), 20.0 + 4.0 * nb
    steps = rays * per_ray
    return dict(bytes=min(field * _cells(case), field * steps) + per_px * rays, flops=steps * (2.0 + 12.0 * nb))


# ------------------------------------------------------------------ 64-bit values
class _Exact:
    """The march in FP64: the ray is cut at every plane of the finest grid, a
    piece belongs to the cell that holds its midpoint."""

    def __init__(self, d):
        f64 = dict(device="cuda", dtype=torch.float64)
        self.lo, self.n = d.lo, d.n
        rho = torch.from_numpy(np.ascontiguousarray(d.rho)).cuda()
        self.rho = rho.float().reshape(-1)
        self.amr = d.kind == "amr"
        self.Lm = d.max_level if self.amr else 0
        self.nf = [x << self.Lm for x in d.n]
        self.h = [(d.hi[a] - d.lo[a]) / self.nf[a] for a in range(3)]
        self.kappa = torch.tensor(d.kappa, **f64)
        self.tab = None
        if d.emis_mode:
            self.tab = torch.tensor(d.lambda_table, **f64)
            t = torch.from_numpy(np.ascontiguousarray(d.temp)).cuda().double().reshape(-1)
            nt = self.tab.shape[1]
            self.x = ((torch.log10(t) - d.logT_lo) / (d.logT_hi - d.logT_lo) * (nt - 1)).clamp(0, nt - 1)
        if self.amr:
            self.B = d.brick
            m = torch.empty([x // d.brick for x in reversed(self.nf)], dtype=torch.int32, device="cuda")
            for b, (l, o) in enumerate(zip(d.brick_level, d.brick_origin // d.brick)):
                w = 1 << (self.Lm - int(l))
                m[o[2]:o[2] + w, o[1]:o[1] + w, o[0]:o[0] + w] = b
            self.map, self.lev = m, torch.from_numpy(d.brick_level).cuda()

    def cell(self, c):
        if not self.amr:
            return (c[2] * self.n[1] + c[1]) * self.n[0] + c[0]
        B = self.B
        b = self.map[c[2] // B, c[1] // B, c[0] // B].long()
        s = self.Lm - self.lev[b]
        q = [(x >> s) & (B - 1) for x in c]
        return ((b * B + q[2]) * B + q[1]) * B + q[0]

    def trace(self, view, uc, vc):
        """Column density [R] and intensities [bands, R] of the pixels (uc, vc)."""
        d = np.array(view.dir) / math.sqrt(sum(x * x for x in view.dir))
        u = np.cross(view.up, d)
        u /= np.linalg.norm(u)
        v = np.cross(d, u)
        N, I = [], []
        per = max(1, (1 << 25) // sum(self.nf))
        for a in range(0, len(uc), per):
            O = [(view.center[k] + uc[a:a + per] * u[k] + vc[a:a + per] * v[k] - self.lo[k]) / self.h[k] for k in range(3)]
            D = [d[k] / self.h[k] for k in range(3)]
            t0 = torch.full_like(O[0], -1e300)
            t1 = -t0
            cuts = []
            for k in range(3):
                if D[k] == 0.0:
                    miss = (O[k] < 0) | (O[k] >= self.nf[k])
                    t1 = torch.where(miss, t0 - 1.0, t1)
                    continue
                t = (torch.arange(self.nf[k] + 1, device="cuda", dtype=torch.float64) - O[k][:, None]) / D[k]
                t0 = torch.maximum(t0, torch.minimum(t[:, 0], t[:, -1]))
                t1 = torch.minimum(t1, torch.maximum(t[:, 0], t[:, -1]))
                cuts.append(t)
            hit = t1 > t0
            t1 = torch.where(hit, t1, t0)
            t = torch.cat(cuts, 1).clamp(t0[:, None], t1[:, None]).sort(1).values
            ds, mid = t[:, 1:] - t[:, :-1], 0.5 * (t[:, 1:] + t[:, :-1])
            k = self.cell([(O[q][:, None] + mid * D[q]).floor().long().clamp(0, self.nf[q] - 1) for q in range(3)])
            rho = self.rho[k].double()
            rds = rho * ds
            N.append(rds.sum(1))
            before = rds.cumsum(1) - rds
            out = []
            for b in range(len(self.kappa)):
                kap, e = float(self.kappa[b]), rho * rds
                if self.tab is not None:
                    x = self.x[k]
                    i = x.floor().long().clamp(max=self.tab.shape[1] - 2)
                    e = e * torch.lerp(self.tab[b][i], self.tab[b][i + 1], x - i)
                if kap:
                    tau = kap * rds
                    e = e * torch.where(tau > 1e-12, -torch.expm1(-tau) / tau.clamp(min=1e-12), torch.ones_like(tau)) \
                        * torch.exp(-kap * before)
                out.append(e.sum(1))
            I.append(torch.stack(out))
        return torch.cat(N), torch.cat(I, 1)

    def image(self, view, res):
        pix = 2.0 * view.half_extent / res
        c = -view.half_extent + (torch.arange(res, device="cuda", dtype=torch.float64) + 0.5) * pix
        return self.trace(view, c.repeat(res), c.repeat_interleave(res))


def _exact_air(E, case):
    """Steps i-vi on dense FP64 images of every level."""
    n0, Lm, H = case["n0"], case["levels"], _view(case).half_extent
    N, I = [], []
    for L in range(Lm + 1):
        a, b = E.image(_view(case), n0 << L)
        N.append(a.cpu().numpy().reshape(n0 << L, n0 << L))
        I.append(b.cpu().numpy().reshape(-1, n0 << L, n0 << L))
    P = [x.sum(0) for x in I]
    idx = [np.full((n0 << L, n0 << L), -1, np.int64) for L in range(Lm + 1)]
    idx[0] = np.arange(n0 * n0).reshape(n0, n0)
    nodes = [np.stack([np.zeros(n0 * n0, np.int64), np.tile(np.arange(n0), n0), np.repeat(np.arange(n0), n0)])]
    n, leaf = n0 * n0, np.ones(n0 * n0, bool)
    up = lambda x: x.repeat(2, 0).repeat(2, 1)  # noqa: E731
    while True:
        flags, V = [], None
        for L in range(Lm):
            V = P[0] if L == 0 else np.where(idx[L] >= 0, P[L], up(V))
            q = np.pad(V, 1, mode="edge")
            s = lambda dj, di: q[1 + dj:q.shape[0] - 1 + dj, 1 + di:q.shape[1] - 1 + di]  # noqa: E731
            c = s(0, 0)
            num = (s(0, 1) - 2 * c + s(0, -1)) ** 2 + (s(1, 0) - 2 * c + s(-1, 0)) ** 2 + \
                2 * ((s(1, 1) - s(-1, 1) - s(1, -1) + s(-1, -1)) / 4) ** 2
            den = (abs(s(0, 1) - c) + abs(c - s(0, -1))) ** 2 + (abs(s(1, 0) - c) + abs(c - s(-1, 0))) ** 2
            if case["xi_norm"]:
                den = 2 * den
            xi = np.where(num == 0, 0.0, np.where(den == 0, 1.0, np.sqrt(num / np.where(den == 0, 1.0, den))))
            flags.append((idx[L] >= 0) & leaf[idx[L].clip(0)] & (xi >= case["xi"]))
        for L in range(Lm - 1, 0, -1):
            w = np.pad(flags[L], 1)
            near = np.zeros_like(flags[L])
            for dj in range(3):
                for di in range(3):
                    near |= w[dj:dj + near.shape[0], di:di + near.shape[1]]
            force = near & (idx[L] < 0)
            force = force.reshape(n0 << (L - 1), 2, n0 << (L - 1), 2).any((1, 3))
            flags[L - 1] |= force & (idx[L - 1] >= 0) & leaf[idx[L - 1].clip(0)]
        split = np.sort(np.concatenate([idx[L][flags[L]] for L in range(Lm)])) if Lm else []
        if not len(split):
            break
        par = np.concatenate(nodes, 1)[:, split]
        kid = np.stack([np.repeat(par[0] + 1, 4), np.repeat(2 * par[1], 4) + np.tile([0, 1, 0, 1], len(split)),
                        np.repeat(2 * par[2], 4) + np.tile([0, 0, 1, 1], len(split))])
        for L in range(1, Lm + 1):
            m = np.nonzero(kid[0] == L)[0]
            idx[L][kid[2][m], kid[1][m]] = n + m
        leaf[split] = False
        leaf = np.concatenate([leaf, np.ones(kid.shape[1], bool)])
        nodes.append(kid)
        n += kid.shape[1]
    t = np.concatenate(nodes, 1)
    if not case["interior"]:
        t = t[:, leaf]
    pick = lambda a: np.select([t[0] == L for L in range(Lm + 1)],  # noqa: E731
                               [a[L][t[2] % (n0 << L), t[1] % (n0 << L)] for L in range(Lm + 1)])
    inten = np.stack([pick([x[b] for x in I]) for b in range(I[0].shape[0])])
    isleaf = leaf if case["interior"] else np.ones(t.shape[1], bool)
    flux = (inten * ((2.0 * H / n0) ** 2 * 0.25 ** t[0].astype(float) * isleaf)).sum(1)
    out = dict.fromkeys(FIELDS + COUNTS)
    room = lambda x: np.pad(x, [(0, 0)] * (x.ndim - 1) + [(0, _capacity(case) - x.shape[-1])])  # noqa: E731
    out.update(coldens=room(pick(N)), intensity=room(inten), p=room(inten.sum(0)), band_flux=flux)
    return out


def _exact_train(case, seed):
    """FP64 minibatch Adam of the same network, batches in the same order."""
    x, y = _train_data(case, seed)
    x, y, n, bs = x.double(), y.long(), case["samples"], case["batch"]
    th = torch.from_numpy(_network(seed)).cuda().double()
    W, o = [], 0
    for shape in ((16, 64), (64,), (64, 64), (64,), (64, 5), (5,)):
        k = int(np.prod(shape))
        W.append(th[o:o + k].reshape(shape).clone().requires_grad_())
        o += k
    opt = torch.optim.Adam(W, lr=1e-3, eps=1e-8)
    nb = -(-n // bs)
    stride, c = 1, int(nb * 0.618) | 1
    while c < 2 * nb + 3:
        if math.gcd(c, nb) == 1:
            stride = c % nb or 1
            break
        c += 2
    hist = []
    for e in range(case["epochs"]):
        tot = 0.0
        for q in range(nb):
            s = slice(((q * stride + e * 7) % nb) * bs, min(((q * stride + e * 7) % nb) * bs + bs, n))
            z = torch.relu(torch.relu(x[s] @ W[0] + W[1]) @ W[2] + W[3]) @ W[4] + W[5]
            loss = torch.nn.functional.cross_entropy(z, y[s])
            opt.zero_grad()
            loss.backward()
            opt.step()
            tot += float(loss.detach()) * len(y[s])
        hist.append(tot / n)
    with torch.no_grad():
        logits = torch.relu(torch.relu(x @ W[0] + W[1]) @ W[2] + W[3]) @ W[4] + W[5]
    return dict(params=torch.cat([w.detach().reshape(-1) for w in W]), loss=np.array(hist), logits=logits)


def exact(case, seed):
    """Fixed images, small adaptive images of scenes refined on intensity, and
    training. Large adaptive images hold millions of decisions, some of them
    within FP32 rounding of the threshold, and their pixels at every level
    take long in FP64; a raster or a learned image is of such a one."""
    if case["call"] == "train":
        return _exact_train(case, seed)
    nf = case["n"] << case.get("grid_levels", 0)
    nb = case.get("bands", 1)
    if case["call"] == "fixed":
        if case["res"] ** 2 * nf * (1 if case["view"][0] != "r" else 3) * (nb + 2) > 2.5e10 or nf > 1024:
            return None
        view = _view(case)
        N, I = _Exact(_desc(case, seed)).image(view, case["res"])
        return dict(coldens=N, intensity=I, p=I.sum(0), n_steps=None,
                    band_flux=I.sum(1) * (2.0 * view.half_extent / case["res"]) ** 2)
    if case["call"] == "air" and case["scene"] in ("wind", "ring") and case["refine_on"] == 0 and \
            (case["n0"] << case["levels"]) <= 512 and case["view"][0] != "r":
        return _exact_air(_Exact(_desc(case, seed)), case)
    return None
