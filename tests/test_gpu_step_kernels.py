"""Kernels of the iteration step at the edges of their short paths: counters
and weights outside the conversion-free product of the absorbed power, source
functions outside the FP32 pairs' range in maps, and tracer launches of many
items smaller than a warp."""
import numpy as np
import pytest

from oracle import mapping as M
from paper_1812_06632_gb300 import inputs as I
from parity_helpers import gpu_context, oracle_grid, oracle_item, run_gpu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _need_gpu(libsoc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("nf", [1, 3, 4, 7, 64])
@pytest.mark.parametrize("kind", ["plain", "huge_counts", "odd_weights"])
def test_absorbed_power_is_the_sequential_sum(libsoc, nf, kind):
    rng = np.random.default_rng([nf, len(kind)])
    rho = rng.uniform(0.5, 2.0, (5, 7, 11)).astype(np.float32)
    rho[0, 0, 0] = 0.0
    cl = I.regular(rho, ell=3e16)
    dust = I.power_law_dust(I.frequency_grid(nf) if nf > 1 else np.array([1e13]), 1e-18)
    ctx = libsoc.Context(0, seed=1)
    ctx.dust_upload(dust.nu, dust.kabs, dust.ksca, dust.g)
    cid = ctx.grid_upload(cl)
    n = cl.n_cells
    t = rng.integers(0, 2 ** 45, (nf, n)).astype(np.int64)
    t[:, ::5] = 0
    if kind == "huge_counts":
        t[:, 1::5] = rng.integers(2 ** 51, 2 ** 62, (nf, len(range(1, n, 5))))
        t[:, 2] = 2 ** 52
        t[:, 3] = 2 ** 52 - 1
        t[:, 4] = -17
    e = rng.uniform(0.5, 2.0, nf) * 1e20
    if kind == "odd_weights":
        e[0] = 0.0
        e[nf // 2] = -e[nf // 2]
        e[-1] = 1e-307
    w = np.ones(1) if nf == 1 else np.zeros(nf)
    if nf > 1:
        d = 0.5 * np.diff(dust.nu)
        w[:-1] += d
        w[1:] += d
    A_in = rng.uniform(0.0, 1e-20, n)
    acc = np.zeros(n)
    for f in range(nf):
        acc = acc + (w[f] * e[f]) * t[f].astype(np.float64)
    rv = cl.rho.astype(np.float64) * ((cl.ell * cl.ell) * cl.ell)
    with np.errstate(divide="ignore", invalid="ignore"):
        ref = np.where(rv > 0, A_in + acc / rv, A_in)
    A = torch.zeros(n, dtype=torch.float64, device="cuda")
    ctx.absorbed_power(cid, torch.from_numpy(t).cuda(), n, torch.from_numpy(e).cuda(), A,
                       A_in=torch.from_numpy(A_in).cuda())
    np.testing.assert_array_equal(A.cpu().numpy(), ref)
    ctx.close()


# cold dust far in the Wien tail (the exponential overflows), hot dust in the
# Rayleigh-Jeans range, and temperatures outside the pairs' range; the bound is
# that of the other map tests (FP32 path lengths)
@pytest.mark.parametrize("f,lo,hi", [(15, 3.0, 12.0), (0, 2000.0, 3000.0), (0, 1e5, 1e8), (8, 5.0, 3000.0)])
@pytest.mark.parametrize("regular", [True, False])
def test_map_source_ranges(libsoc, f, lo, hi, regular):
    w = (I.config_c2(n=19, n_freq=16, n_packages=0) if regular
         else I.config_c3(root_n=6, max_refine=2, threshold=3.0, tau_peak_1um=5.0, n_freq=16))
    cl = w.clouds[0]
    T = np.exp(np.random.default_rng(f).uniform(np.log(lo), np.log(hi), cl.n_cells)).astype(np.float32)
    ctx, ids = gpu_context(w)
    out = torch.zeros((17, 23), dtype=torch.float32, device="cuda")
    d, up, c = [0.3, -0.5, 0.8], [0, 1, 0], [cl.nx / 2] * 3
    ctx.map(ids[0], torch.from_numpy(T).cuda(), f, d, up, 23, 17, cl.nx / 18, c, out, I_bg=0.0)
    ref = M.ray_map(oracle_grid(cl), T.astype(np.float64), w.dust.kabs[f] * cl.ell, w.dust.ksca[f] * cl.ell,
                    w.dust.nu[f], d, up, 23, 17, cl.nx / 18, c, I_bg=0.0)
    np.testing.assert_allclose(out.cpu().numpy().astype(np.float64), ref, rtol=1e-4, atol=1e-6 * np.abs(ref).max() + 2e-45)
    ctx.close()


@pytest.mark.parametrize("octree", [False, True])
def test_items_smaller_than_a_warp(libsoc, octree):
    """Lanes of one warp hold packages of several items and change items
    together and apart: counters, statistics and steps of every item."""
    w = (I.config_c3(root_n=6, max_refine=2, sigma=2.0, threshold=3.0, n_freq=8, tau_peak_1um=60.0) if octree
         else I.config_c2(n=12, n_freq=8, n_packages=0, tau_1um=20.0))
    cl = w.clouds[0]
    ctx, ids = gpu_context(w)
    counts = [1, 7, 33, 2, 64, 5, 31, 1, 100, 3]
    specs = [dict(source=0, freq=k % 8, n_packages=m, pid_offset=11 * k, tally_offset=k * cl.n_cells)
             for k, m in enumerate(counts * 3)]
    tally, stats, steps = run_gpu(ctx, specs, len(specs) * cl.n_cells)
    p = 0
    for k, s in enumerate(specs):
        t_o, st_o, s_o = oracle_item(w, 0, s)
        np.testing.assert_array_equal(tally[k * cl.n_cells:(k + 1) * cl.n_cells], t_o)
        assert (stats[k][0], stats[k][3]) == (st_o["escaped"], st_o["emitted"]) and stats[k][2] == s_o.sum()
        np.testing.assert_array_equal(steps[p:p + s["n_packages"]], s_o)
        p += s["n_packages"]
    ctx.close()
