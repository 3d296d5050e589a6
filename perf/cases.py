"""What a user of the library has it do, as measurable cases: tracer launches
on regular grids, octrees and uneven batches, the equilibrium step, dust
iterations, maps, and the learned seed's network (whole and layer by layer).

``listed()`` holds the named cases, ``draw(rng)`` gives one more of the same
ranges, ``prepare`` makes the inputs and the handles a program keeps,
``run`` is one pass through the public entry points and ``work`` the bytes
and operations such a pass cannot do without.  ``exact`` gives, where there
is a closed form, the outputs in 64-bit arithmetic without the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1812_06632_gb300 import inputs as I

H, K, C = 6.62607015e-27, 1.380649e-16, 2.99792458e10
OPS_PER_STEP = 54           # FP32 operations of one photon-cell step without scattering
LAYERS = [(16, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128),
          (192, 64), (64, 64), (96, 32), (32, 32), (48, 16), (16, 16), (16, 16)]


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one small launch, where the host path and the launch count: uniform
        # 32^3 cube, one frequency, 1e5 background packages
        dict(name="trace_uniform32_1nu", kind="trace", nx=32, ny=32, nz=32, nf=1, n_bg=100_000, sigma=0.0,
             tau=1.0, g=0.0, ali=False),
        # the benchmark's pass: every frequency of a 128^3 cloud in one
        # prepared launch, then absorbed power and temperatures
        dict(name="pass_lognormal128_64nu", kind="pass", nx=128, ny=128, nz=128, nf=64, n_bg=1_000_000, sigma=1.5,
             tau=5.0, g=0.5),
        # hierarchical grid (32^3 root, three refinements), background and
        # point sources, optically thick core
        dict(name="trace_octree32r3_64nu", kind="octree", root=32, refine=3, nf=64, n_bg=100_000, n_ps=100_000,
             tau=100.0),
        # many clouds of different size and optical depth in one launch
        dict(name="trace_batch12_16nu", kind="batch", clouds=12, lo=32, hi=96, nf=16, n_pk=50_000),
        # one equilibrium step of a program that runs its own iteration:
        # counters -> absorbed power -> temperatures -> dust weights
        dict(name="equilibrium128_64nu", kind="equilibrium", nx=128, ny=128, nz=128, nf=64, sigma=1.5),
        # the learned seed's data path: several hot-core clouds to a few dust
        # iterations at once, uniform dust emission
        dict(name="iterate_batch3_64cube", kind="iterate_batch", clouds=3, side=64, nf=64, n_pk=50_000, iters=4,
             ali=False),
        # one hierarchical cloud with emission-weighted dust packages
        dict(name="iterate_octree_weighted", kind="iterate_octree", root=16, refine=3, nf=32, n_pk=100_000, iters=4,
             mode="weighted"),
        # surface-brightness map of a 128^3 cloud
        dict(name="map1024_lognormal128", kind="map", n=128, npx=1024, npy=1024, refine=0),
        # the network's prediction for a batch of clouds
        dict(name="unet_forward_b4_64", kind="unet", batch=4, side=64, n_in=4, train=False),
        # one training step's gradients
        dict(name="unet_train_b4_64", kind="unet", batch=4, side=64, n_in=4, train=True),
        # one layer through the single-operation entry points: forward, input
        # and weight gradient
        dict(name="conv_b4_32cube_32to32", kind="conv", N=4, D=32, H=32, W=32, cin=32, cout=32),
        # the same of a volume with odd sides
        dict(name="conv_b2_ragged_48to32", kind="conv", N=2, D=13, H=10, W=27, cin=48, cout=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["trace", "pass", "octree", "batch", "equilibrium", "iterate_batch", "iterate_octree", "map",
                       "unet", "unet", "conv", "conv"])
    if kind in ("trace", "pass"):
        c = dict(kind=kind, nx=rng.randint(9, 128), ny=rng.randint(9, 128), nz=rng.randint(9, 128), nf=_log(rng, 1, 64),
                 n_bg=_log(rng, 1_000, 1_000_000), sigma=round(rng.uniform(0.0, 2.0), 3),
                 tau=round(10 ** rng.uniform(-1, 2), 3), g=round(rng.uniform(0.0, 0.7), 3))
        if kind == "trace":
            c["n_bg"] = min(c["n_bg"], 200_000)
            c["ali"] = rng.random() < 0.25
        return c
    if kind == "octree":
        return dict(kind=kind, root=rng.randint(6, 32), refine=rng.randint(1, 3), nf=_log(rng, 1, 64),
                    n_bg=_log(rng, 1_000, 100_000), n_ps=_log(rng, 1_000, 100_000), tau=round(10 ** rng.uniform(0, 2), 3))
    if kind == "batch":
        lo = rng.randint(10, 48)
        return dict(kind=kind, clouds=rng.randint(2, 12), lo=lo, hi=rng.randint(lo, 96), nf=_log(rng, 1, 16),
                    n_pk=_log(rng, 1_000, 50_000))
    if kind == "equilibrium":
        return dict(kind=kind, nx=rng.randint(16, 128), ny=rng.randint(16, 128), nz=rng.randint(16, 128),
                    nf=rng.randint(8, 64), sigma=round(rng.uniform(0.5, 2.0), 3))
    if kind == "iterate_batch":
        return dict(kind=kind, clouds=rng.randint(1, 3), side=8 * rng.randint(2, 8), nf=rng.randint(8, 64),
                    n_pk=_log(rng, 2_000, 50_000), iters=rng.randint(1, 4), ali=rng.random() < 0.4)
    if kind == "iterate_octree":
        return dict(kind=kind, root=rng.randint(6, 16), refine=rng.randint(1, 3), nf=rng.randint(8, 32),
                    n_pk=_log(rng, 2_000, 100_000), iters=rng.randint(1, 4),
                    mode=rng.choice(["plain", "weighted", "ali", "mean", "difference"]))
    if kind == "map":
        return dict(kind=kind, n=rng.choice([16, 32]) if rng.random() < 0.3 else rng.randint(17, 128),
                    npx=_log(rng, 64, 1024), npy=_log(rng, 64, 1024), refine=0)
    if kind == "unet":
        return dict(kind=kind, batch=rng.randint(1, 4), side=8 * rng.randint(2, 8), n_in=rng.randint(2, 4),
                    train=rng.random() < 0.5)
    while True:
        c = dict(kind=kind, N=rng.randint(1, 4), D=_log(rng, 3, 64), H=_log(rng, 3, 64), W=_log(rng, 3, 64),
                 cin=16 * rng.choice([1, 2, 3, 4, 6, 8]), cout=16 * rng.choice([1, 2, 3, 4, 6, 8]))
        if c["N"] * c["D"] * c["H"] * c["W"] * max(c["cin"], c["cout"]) <= 4 * 64 ** 3 * 48:
            return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _lognormal(nx, ny, nz, sigma, gen):
    """(nz, ny, nx) lognormal density of mean about 1, P(k) ~ k^-3.5, with the
    sides cut from a periodic cube (FP64 device tensor)."""
    n = max(nx, ny, nz)
    f = torch.fft.rfftn(torch.randn((n, n, n), generator=gen, device="cuda", dtype=torch.float64))
    k1 = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64)
    kz = torch.fft.rfftfreq(n, device="cuda", dtype=torch.float64)
    k2 = (k1 * k1)[:, None, None] + (k1 * k1)[None, :, None] + (kz * kz)[None, None, :]
    k2[0, 0, 0] = 1.0
    amp = k2 ** (-3.5 / 4.0)
    amp[0, 0, 0] = 0.0
    g = torch.fft.irfftn(f * amp, s=(n, n, n))
    g = (g - g.mean()) / g.std()
    return torch.exp(sigma * g - 0.5 * sigma * sigma)[:nz, :ny, :nx].contiguous()


def _dust(nf, kext_1um, g=0.5):
    nu = I.frequency_grid(nf) if nf > 1 else np.array([I.NU_1UM])
    return I.power_law_dust(nu, kext_1um, g=g)


def _context(seed, dust):
    from paper_1812_06632_gb300 import soc
    ctx = soc.Context(0, seed=seed + 1)
    ctx.dust_upload(dust.nu, dust.kabs, dust.ksca, dust.g)
    return ctx


def _regular_cloud(case, seed):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rho = _lognormal(nx, ny, nz, case["sigma"], _gen(seed)).float().cpu().numpy()
    n = max(nx, ny, nz)
    ell = I.PC_CM / n
    return I.regular(rho, ell=ell), case.get("tau", 5.0) / ((n / 2) * ell)


def _octree_cloud(root, refine, tau, seed, side_pc=0.5):
    """The hierarchy is that of one field per size (so outputs keep their
    shape), the densities in it are the seed's."""
    fine = _lognormal(root << refine, root << refine, root << refine, 1.5, _gen(root)).cpu().numpy()
    ell = side_pc * I.PC_CM / root
    cl = I.octree_from_fine(fine, root, refine, 6.0, ell=ell)
    noise = np.random.default_rng(seed).standard_normal(cl.n_cells)
    cl.rho = (cl.rho * np.exp(0.2 * noise)).astype(np.float32)
    c = (root << refine) // 2
    rays = max(fine[c, c, c:].sum(), fine[c, c:, c].sum(), fine[c:, c, c].sum())
    return cl, tau / (rays * ell / (1 << refine))


def _sources(rng, side, n, nu, L):
    pos = rng.uniform(0.3, 0.7, size=(n, 3)) * side
    return pos, np.stack([I.stellar_luminosity(nu, 1e4, L / n) for _ in range(n)])


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    dev = dict(device="cuda")
    if kind in ("trace", "pass"):
        cl, kext = _regular_cloud(case, seed)
        dust = _dust(case["nf"], kext, case["g"])
        ctx = _context(seed, dust)
        cid = ctx.grid_upload(cl)
        ctx.sources_upload(cid, I.diluted_blackbodies(dust.nu))
        nf, n = case["nf"], cl.n_cells
        items = ctx.items([dict(cloud=cid, freq=f, source=0, n_packages=case["n_bg"], tally_offset=f * n)
                           for f in range(nf)])
        s = dict(case=case, ctx=ctx, cid=cid, cells=n, items=items,
                 tally=torch.zeros((nf, n), dtype=torch.int64, **dev),
                 stats=torch.zeros((nf, 4), dtype=torch.int64, **dev))
        if case.get("ali"):
            s["self"] = torch.zeros_like(s["tally"])
        if kind == "pass":
            s["batch"] = ctx.batch_create(items)
            s["e"] = torch.from_numpy(ctx.package_energy(cid, 0, case["n_bg"])).cuda()
            s["A"] = torch.zeros(n, dtype=torch.float64, **dev)
            s["T"] = torch.full((n,), 10.0, **dev)
            s["dT"] = torch.zeros(1, dtype=torch.float64, **dev)
        return s
    if kind == "octree":
        cl, kext = _octree_cloud(case["root"], case["refine"], case["tau"], seed)
        dust = _dust(case["nf"], kext)
        ctx = _context(seed, dust)
        cid = ctx.grid_upload(cl)
        pos, L = _sources(rng, case["root"], 3, dust.nu, 1e37)
        ctx.sources_upload(cid, I.diluted_blackbodies(dust.nu), pos, L)
        specs, off = [], 0
        for f in range(case["nf"]):
            for src, npk in ((0, case["n_bg"]), (1, case["n_ps"])):
                specs.append(dict(cloud=cid, freq=f, source=src, n_packages=npk, tally_offset=off))
                off += cl.n_cells
        return dict(case=case, ctx=ctx, items=ctx.items(specs), tally=torch.zeros(off, dtype=torch.int64, **dev),
                    stats=torch.zeros((len(specs), 4), dtype=torch.int64, **dev))
    if kind == "batch":
        dust = _dust(case["nf"], 1.0)
        ctx = _context(seed, dust)
        gen, specs, off = _gen(seed), [], 0
        for k in range(case["clouds"]):
            n = case["lo"] + (case["hi"] - case["lo"]) * (7 * k % case["clouds"]) // max(case["clouds"] - 1, 1)
            ell = I.PC_CM / n
            scale = math.exp(rng.uniform(math.log(0.5), math.log(100.0))) / ((n / 2) * ell)
            rho = (_lognormal(n, n, n, float(rng.uniform(1.0, 2.0)), gen) * scale).float().cpu().numpy()
            cid = ctx.grid_upload(I.regular(rho, ell=ell))
            pos, L = _sources(rng, n, int(rng.integers(1, 4)), dust.nu, 1e36)
            ctx.sources_upload(cid, I.diluted_blackbodies(dust.nu), pos, L)
            npk = max(1, int(round(case["n_pk"] * (n / 32) ** 1.66)))
            for f in range(case["nf"]):
                for src in (0, 1):
                    specs.append(dict(cloud=cid, freq=f, source=src, n_packages=npk, tally_offset=off))
                    off += n ** 3
        return dict(case=case, ctx=ctx, items=ctx.items(specs), tally=torch.zeros(off, dtype=torch.int64, **dev),
                    stats=torch.zeros((len(specs), 4), dtype=torch.int64, **dev))
    if kind == "equilibrium":
        cl, kext = _regular_cloud(case, seed)
        dust = _dust(case["nf"], kext)
        ctx = _context(seed, dust)
        cid = ctx.grid_upload(cl)
        bg = I.diluted_blackbodies(dust.nu)
        ctx.sources_upload(cid, bg)
        nf, n = case["nf"], cl.n_cells
        # counters as 1e6 background packages per frequency leave them, with a
        # hot region around an inner source
        gen = _gen(seed + 1)
        rho = torch.from_numpy(cl.rho).cuda().double()
        ax = [torch.arange(m, device="cuda") - m * float(rng.uniform(0.35, 0.65))
              for m in (case["nz"], case["ny"], case["nx"])]
        r2 = (ax[0] ** 2)[:, None, None] + (ax[1] ** 2)[None, :, None] + (ax[2] ** 2)[None, None, :]
        hits = 1e6 * 0.9 * max(case["nx"], case["ny"], case["nz"]) / n * (1 + 1e4 / (1 + r2)).reshape(-1)
        tally = torch.empty((nf, n), dtype=torch.int64, **dev)
        for f in range(nf):
            noise = 0.5 + torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
            tally[f] = (hits * noise * -torch.expm1(-rho * (dust.kabs[f] * cl.ell)) * 2.0 ** 31).long()
        return dict(case=case, ctx=ctx, cid=cid, cloud=cl, dust=dust, tally=tally,
                    e=torch.from_numpy(ctx.package_energy(cid, 0, 1_000_000)).cuda(),
                    A=torch.zeros(n, dtype=torch.float64, **dev), T=torch.full((n,), 10.0, **dev),
                    T0=torch.full((n,), 10.0, **dev), dT=torch.zeros(1, dtype=torch.float64, **dev),
                    w=torch.zeros((nf, n), dtype=torch.int64, **dev), eu=torch.zeros(nf, dtype=torch.float64, **dev))
    if kind == "iterate_batch":
        side = case["side"]
        ell = 0.15 * I.PC_CM / side
        dust = _dust(case["nf"], 1.0 / ((side / 2) * ell))
        ctx = _context(seed, dust)
        gen, ids, T = _gen(seed), [], []
        for _ in range(case["clouds"]):
            tau = math.exp(rng.uniform(math.log(1000.0), math.log(5000.0)))
            rho = (_lognormal(side, side, side, float(rng.uniform(1.0, 2.0)), gen) * tau).float().cpu().numpy()
            cid = ctx.grid_upload(I.regular(rho, ell=ell))
            pos, L = _sources(rng, side, int(rng.integers(1, 3)), dust.nu, 2e38)
            ctx.sources_upload(cid, I.diluted_blackbodies(dust.nu), pos, L)
            ids.append(cid)
            T.append(torch.empty(side ** 3, **dev))
        return dict(case=case, ctx=ctx, ids=ids, T=T)
    if kind == "iterate_octree":
        cl, kext = _octree_cloud(case["root"], case["refine"], 200.0, seed, side_pc=0.1)
        dust = _dust(case["nf"], kext)
        ctx = _context(seed, dust)
        cid = ctx.grid_upload(cl)
        pos, L = _sources(rng, case["root"], 1, dust.nu, 3e36)
        ctx.sources_upload(cid, I.diluted_blackbodies(dust.nu), pos, L)
        leaf = torch.from_numpy(cl.leaves().astype(np.int64)).cuda()
        return dict(case=case, ctx=ctx, cid=cid, T=torch.zeros(cl.n_cells, **dev), leaf=leaf, n_leaf=leaf.numel())
    if kind == "map":
        gen, n = _gen(seed), case["n"]
        rho = _lognormal(n, n, n, 1.5, gen).float().cpu().numpy()
        ell = I.PC_CM / n
        dust = _dust(16, 5.0 / ((n / 2) * ell))
        ctx = _context(seed, dust)
        cl = I.regular(rho, ell=ell)
        cid = ctx.grid_upload(cl)
        T = (15.0 * torch.exp(0.4 * torch.randn(n ** 3, generator=gen, device="cuda"))).clamp(5.0, 300.0)
        d = rng.normal(size=3)
        return dict(case=case, ctx=ctx, cid=cid, cloud=cl, dust=dust, T=T, freq=6, dir=d / np.linalg.norm(d),
                    up=np.array([0.1, 0.2, 1.0]), pix=1.2 * n / max(case["npx"], case["npy"]), center=np.full(3, n / 2),
                    out=torch.zeros((case["npy"], case["npx"]), **dev))
    if kind == "unet":
        from paper_1812_06632_gb300 import soc
        from paper_1812_06632_gb300.learned import init_params
        B, S, gen = case["batch"], case["side"], _gen(seed)
        net = soc.UNet(B, S, n_inputs=case["n_in"])
        p = init_params(seed)
        net.set_params(p)
        x = torch.randn((B, S, S, S, case["n_in"]), generator=gen, device="cuda")
        smooth = F.avg_pool3d(x.permute(0, 4, 1, 2, 3), 3, 1, 1).permute(0, 2, 3, 4, 1)
        x = (x + 4.0 * smooth).clamp(-6.0, 6.0).contiguous()
        y = smooth[..., 0] * 2.0 + 0.1 * torch.randn((B, S, S, S), generator=gen, device="cuda")
        return dict(case=case, net=net, params=p, x=x, y=y.contiguous(), pred=torch.zeros((B, S, S, S), **dev),
                    loss=torch.zeros(1, dtype=torch.float64, **dev))
    gen = _gen(seed)
    shape, ci, co = (case["N"], case["D"], case["H"], case["W"]), case["cin"], case["cout"]

    def bf(*s, scale=1.0):
        return (torch.randn(s, generator=gen, device="cuda") * scale).to(torch.bfloat16)
    return dict(case=case, x=bf(*shape, ci).relu(), w=bf(co, 27, ci, scale=math.sqrt(2.0 / (27 * ci))),
                b=0.1 * torch.randn(co, generator=gen, device="cuda"), gy=bf(*shape, co, scale=0.1),
                y=torch.empty((*shape, co), dtype=torch.bfloat16, **dev),
                scratch=torch.empty(co * 27 * ci, dtype=torch.bfloat16, **dev),
                gx=torch.empty((*shape, ci), **dev), gw=torch.zeros((co, 27, ci), **dev), gb=torch.zeros(co, **dev))


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("trace", "octree", "batch"):
        s["tally"].zero_()
        s["stats"].zero_()
        if case.get("ali"):
            s["self"].zero_()
        s["ctx"].simulate(s["items"], s["tally"], s["stats"], self_tally=s.get("self"))
        return {k: s[k] for k in ("tally", "stats", "self") if k in s}
    if kind == "pass":
        ctx = s["ctx"]
        ctx.batch_launch(s["batch"], s["tally"], s["stats"])
        ctx.absorbed_power(s["cid"], s["tally"], s["cells"], s["e"], s["A"])
        ctx.update_temperature(s["cid"], s["A"], s["T"], s["dT"])
        return {k: s[k] for k in ("tally", "stats", "A", "T")}
    if kind == "equilibrium":
        ctx = s["ctx"]
        ctx.absorbed_power(s["cid"], s["tally"], s["tally"].shape[1], s["e"], s["A"])
        s["T"].copy_(s["T0"])
        ctx.update_temperature(s["cid"], s["A"], s["T"], s["dT"])
        ctx.dust_emission(s["cid"], s["T"], s["w"], s["eu"])
        return {k: s[k] for k in ("A", "T", "dT", "w", "eu")}
    if kind == "iterate_batch":
        rows, _ = s["ctx"].iterate_batch(s["ids"], s["T"], n_background=case["n_pk"], n_point=case["n_pk"],
                                         n_per_cell=1, max_iter=case["iters"], dT_tol=1e-6, ali=case["ali"])
        return {"T": s["T"], "history": [r["history"] for r in rows], "steps": [r["steps"] for r in rows]}
    if kind == "iterate_octree":
        n_leaf, mode = s["n_leaf"], case["mode"]
        opt = {"plain": dict(n_per_cell=2), "weighted": dict(n_weighted=8 * n_leaf, weighted_cap=10_000),
               "ali": dict(n_per_cell=2, ali=True),
               "mean": dict(reference_field="mean", n_dust_first=n_leaf, n_dust_last=8 * n_leaf),
               "difference": dict(reference_field="difference", n_weighted=4 * n_leaf)}[mode]
        r = s["ctx"].iterate(s["cid"], s["T"], n_background=case["n_pk"], n_point=case["n_pk"],
                             max_iter=case["iters"], dT_tol=1e-6, **opt)
        return {"T": s["T"][s["leaf"]], "history": r["history"], "steps": r["steps"]}
    if kind == "map":
        s["ctx"].map(s["cid"], s["T"], s["freq"], s["dir"], s["up"], case["npx"], case["npy"], s["pix"], s["center"],
                     s["out"], I_bg=1e-18)
        return s["out"]
    if kind == "unet":
        if not case["train"]:
            s["net"].forward(s["x"], s["pred"])
            return s["pred"]
        s["net"].backward(s["x"], s["y"], s["pred"], s["loss"])
        return {"pred": s["pred"], "loss": s["loss"], "grads": s["net"].get_params(grads=True)}
    from paper_1812_06632_gb300 import soc
    s["gw"].zero_()
    s["gb"].zero_()
    soc.conv3d(s["x"], s["w"], s["b"], relu=True, out=s["y"])
    soc.conv3d_dgrad(s["gy"], s["w"], s["scratch"], s["gx"])
    soc.conv3d_wgrad(s["gy"], s["x"], s["gw"], s["gb"])
    return {k: s[k] for k in ("y", "gx", "gw", "gb")}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]

    def traced(packages, side, cells, counters):
        # a package crosses about as many cells as the grid has on a side
        return dict(bytes=4.0 * cells + 8.0 * counters, flops=OPS_PER_STEP * 0.9 * side * packages)
    if kind in ("trace", "pass"):
        n = case["nx"] * case["ny"] * case["nz"]
        side = 3.0 / (1 / case["nx"] + 1 / case["ny"] + 1 / case["nz"])
        r = traced(case["nf"] * case["n_bg"], side, n, n * case["nf"])
        if kind == "pass":
            r["bytes"] += 8.0 * n * case["nf"] + 24.0 * n
        return r
    if kind == "octree":
        cells = 4 * case["root"] ** 3
        return traced(case["nf"] * (case["n_bg"] + case["n_ps"]), 2.0 * case["root"], cells, 2 * cells * case["nf"])
    if kind == "batch":
        n = 0.5 * (case["lo"] + case["hi"])
        cells = case["clouds"] * n ** 3
        return traced(2 * case["nf"] * case["clouds"] * case["n_pk"] * (n / 32) ** 1.66, n, cells, 2 * cells * case["nf"])
    if kind == "equilibrium":
        n = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=16.0 * n * case["nf"] + 36.0 * n, flops=20.0 * n * case["nf"])
    if kind == "iterate_batch":
        n, nf = case["side"] ** 3, case["nf"]
        t = traced(case["clouds"] * nf * (2 * case["n_pk"] + case["iters"] * n), 0.2 * case["side"], n, 0)
        t["bytes"] += case["clouds"] * (case["iters"] + 1) * 8.0 * n * nf
        return t
    if kind == "iterate_octree":
        n, nf = 4 * case["root"] ** 3, case["nf"]
        t = traced(nf * (2 * case["n_pk"] + case["iters"] * 4 * n), 0.5 * case["root"], n, 0)
        t["bytes"] += (case["iters"] + 1) * 8.0 * n * nf
        return t
    if kind == "map":
        pix = case["npx"] * case["npy"]
        return dict(bytes=4.0 * pix + 8.0 * case["n"] ** 3, flops=40.0 * pix * 0.5 * case["n"])
    if kind == "unet":
        S, B = case["side"], case["batch"]
        lev = [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0]
        fl = sum(2.0 * 27 * ci * co * B * (S >> v) ** 3 for (ci, co), v in zip(LAYERS, lev))
        par = sum(27 * ci * co + co for ci, co in LAYERS)
        v = B * S ** 3
        return dict(bytes=4.0 * (v * (case["n_in"] + (2 if case["train"] else 1)) + par * (2 if case["train"] else 1)),
                    flops=fl * (3 if case["train"] else 1))
    v = case["N"] * case["D"] * case["H"] * case["W"]
    ci, co = case["cin"], case["cout"]
    return dict(bytes=v * (2.0 * ci + 2.0 * co + 2.0 * co + 4.0 * ci) + 27.0 * ci * co * 6,
                flops=3 * 2.0 * 27 * ci * co * v)


# ---------------------------------------------------------------------------
# The same in 64 bits, without the library
# ---------------------------------------------------------------------------
def _planck(nu, T):
    return (2.0 * H * nu ** 3 / C ** 2) / torch.expm1(H * nu / (K * T))


def _equilibrium(s):
    cl, dust = s["cloud"], s["dust"]
    nu = torch.from_numpy(dust.nu).cuda()
    kabs = torch.from_numpy(dust.kabs).cuda()
    w = torch.zeros_like(nu)
    w[:-1] += 0.5 * (nu[1:] - nu[:-1])
    w[1:] += 0.5 * (nu[1:] - nu[:-1])
    rv = torch.from_numpy(cl.rho).cuda().double() * cl.ell ** 3
    A = torch.zeros_like(rv)
    for f in range(nu.numel()):
        A += w[f] * s["e"][f] * s["tally"][f].double()
    A = A / rv
    lo, hi = torch.full_like(A, math.log(2.7)), torch.full_like(A, math.log(3000.0))

    def power(T):
        E = torch.zeros_like(T)
        for f in range(nu.numel()):
            E += 4 * math.pi * w[f] * kabs[f] * _planck(nu[f], T)
        return E
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        low = power(torch.exp(mid)) < A
        lo, hi = torch.where(low, mid, lo), torch.where(low, hi, mid)
    T = torch.exp(0.5 * (lo + hi))
    eu = torch.stack([(4 * math.pi * rv * kabs[f] * _planck(nu[f], T)).max() for f in range(nu.numel())]) / 2.0 ** 31
    return dict(A=A, T=T, dT=(T - 10.0).abs().max().reshape(1), w=None, eu=eu)


def _map(s):
    case, cl, dust, f = s["case"], s["cloud"], s["dust"], s["freq"]
    d = s["dir"] / np.linalg.norm(s["dir"])
    e1 = np.cross(s["up"], d)
    e1 /= np.linalg.norm(e1)
    e2 = np.cross(d, e1)
    npx, npy, pix = case["npx"], case["npy"], s["pix"]
    px = ((torch.arange(npx, device="cuda", dtype=torch.float64) + 0.5) - 0.5 * npx) * pix
    py = ((torch.arange(npy, device="cuda", dtype=torch.float64) + 0.5) - 0.5 * npy) * pix
    n = case["n"]
    o = [(s["center"][a] + px[None, :] * e1[a] + py[:, None] * e2[a]).reshape(-1) for a in range(3)]
    t0, t1 = torch.full_like(o[0], -1e300), torch.full_like(o[0], 1e300)
    ea = torch.zeros_like(o[0], dtype=torch.long)
    for a in range(3):
        ta, tb = (0.0 - o[a]) / d[a], (n - o[a]) / d[a]
        ta, tb = torch.minimum(ta, tb), torch.maximum(ta, tb)
        ea = torch.where(ta > t0, torch.full_like(ea, a), ea)
        t0, t1 = torch.maximum(t0, ta), torch.minimum(t1, tb)
    live = t0 < t1
    idx = []
    for a in range(3):
        i = torch.floor(o[a] + t0 * d[a]).long().clamp(0, n - 1)
        idx.append(torch.where(ea == a, torch.full_like(i, 0 if d[a] > 0 else n - 1), i))
    rho = torch.from_numpy(cl.rho).cuda().double()
    kext = float(dust.kabs[f] + dust.ksca[f])
    S = float(dust.kabs[f]) / kext * _planck(float(dust.nu[f]), s["T"].double())
    I_, trans, t = torch.zeros_like(t0), torch.ones_like(t0), t0.clone()
    for _ in range(3 * n):
        if not bool(live.any()):
            break
        c = idx[0] + n * (idx[1] + n * idx[2])
        te = torch.stack([((idx[a] + (1 if d[a] > 0 else 0)).double() - o[a]) / d[a] for a in range(3)])
        tn, ax = te.min(0)
        dtau = torch.where(live, rho[c] * kext * cl.ell * (tn - t).clamp_min(0.0), torch.zeros_like(t))
        I_ += S[c] * -torch.expm1(-dtau) * trans
        trans *= torch.exp(-dtau)
        t = tn
        for a in range(3):
            step = torch.where(live & (ax == a), torch.full_like(ax, 1 if d[a] > 0 else -1), torch.zeros_like(ax))
            j = idx[a] + step
            live = live & (j >= 0) & (j < n)
            idx[a] = j.clamp(0, n - 1)
    return (I_ + 1e-18 * trans).reshape(npy, npx)


def _conv(x, w, b=None):
    """3x3x3 convolution of (N, C, D, H, W) with [Cout][27][Cin] weights."""
    co, _, ci = w.shape
    return F.conv3d(x, w.reshape(co, 3, 3, 3, ci).permute(0, 4, 1, 2, 3), b, padding=1)


def _unet(s):
    par, k, flat = [], 0, torch.from_numpy(s["params"]).cuda().double().requires_grad_(s["case"]["train"])
    for ci, co in LAYERS:
        nw = co * 27 * ci
        par.append((flat[k:k + nw].reshape(co, 27, ci), flat[k + nw:k + nw + co]))
        k += nw + co
    x = s["x"].double().permute(0, 4, 1, 2, 3)
    x = F.pad(x, (0, 0, 0, 0, 0, 0, 0, 16 - x.shape[1]))

    def two(v, l):
        return _conv(_conv(v, *par[l]).relu(), *par[l + 1]).relu()

    def up(v):
        return F.interpolate(v, scale_factor=2, mode="nearest")
    e0 = two(x, 0)
    e1 = two(F.max_pool3d(e0, 2), 2)
    e2 = two(F.max_pool3d(e1, 2), 4)
    b = two(F.max_pool3d(e2, 2), 6)
    d2 = two(torch.cat([up(b), e2], 1), 8)
    d1 = two(torch.cat([up(d2), e1], 1), 10)
    d0 = two(torch.cat([up(d1), e0], 1), 12)
    pred = _conv(d0, *par[14])[:, 0]
    if not s["case"]["train"]:
        return pred
    loss = (pred - s["y"].double()).square().mean()
    loss.backward()
    return dict(pred=pred.detach(), loss=loss.detach().reshape(1), grads=flat.grad)


def _conv_layer(s):
    x, gy = s["x"].double().permute(0, 4, 1, 2, 3), s["gy"].double().permute(0, 4, 1, 2, 3)
    x = x.requires_grad_(True)
    w, b = s["w"].double().requires_grad_(True), s["b"].double().requires_grad_(True)
    y = _conv(x, w, b)
    y.backward(gy)
    return dict(y=y.detach().relu().permute(0, 2, 3, 4, 1), gx=x.grad.permute(0, 2, 3, 4, 1), gw=w.grad, gb=b.grad)


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("equilibrium", "map", "unet", "conv"):
        return None
    s = prepare(case, seed)
    return {"equilibrium": _equilibrium, "map": _map, "unet": _unet, "conv": _conv_layer}[kind](s)
