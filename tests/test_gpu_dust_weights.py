"""The uniform dust weights are the FP64 evaluation's, bit for bit: they equal
rint(L / max L 2^31) formed in FP64 from the luminosities of
soc_dust_luminosity (which evaluates every one in FP64), also where the FP32
bounds of soc_dust_emission do not settle the value: ties, temperatures and
densities outside the bounds' ranges, overflowing Planck exponents, zero
opacity, sizes around the kernels' tiles."""
import numpy as np
import pytest

from paper_1812_06632_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _need_gpu(libsoc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _temperatures(kind, n, rng):
    if kind == "uniform":
        return np.full(n, 17.5, np.float32)                    # every leaf ties
    if kind == "cold":
        return rng.uniform(2.7, 6.0, n).astype(np.float32)     # most frequencies overflow expm1
    if kind == "hot":
        return rng.uniform(500.0, 3000.0, n).astype(np.float32)
    if kind == "wide":
        return np.exp(rng.uniform(np.log(2.7), np.log(3000.0), n)).astype(np.float32)
    T = np.exp(rng.uniform(np.log(1e-4), np.log(1e8), n)).astype(np.float32)     # "odd": past the bounds' ranges
    T[rng.integers(0, n, 4)] = 0.0
    return T


@pytest.mark.parametrize("grid", ["regular", "octree", "empty_cells", "one"])
@pytest.mark.parametrize("kind", ["uniform", "cold", "hot", "wide", "odd"])
@pytest.mark.parametrize("nf", [1, 17, 64])
def test_dust_weights_equal_fp64_evaluation(libsoc, grid, kind, nf):
    rng = np.random.default_rng([nf, len(kind), len(grid)])
    if grid == "octree":
        cl = I.config_c3(root_n=8, max_refine=2, sigma=1.5, threshold=3.0).clouds[0]
    elif grid == "one":
        cl = I.regular(np.ones((1, 1, 1), np.float32), ell=1e17)
    else:
        rho = np.exp(rng.normal(0.0, 1.5, (23, 29, 31))).astype(np.float32)
        if grid == "empty_cells":
            rho[rng.random(rho.shape) < 0.3] = 0.0
            rho.ravel()[:3] = (1e-38, 1e-40, 3e37)             # a denormal, and ends of the FP32 range
        if kind == "uniform":
            rho[rho > 0] = 1.0
        cl = I.regular(rho, ell=3e16)
    dust = I.power_law_dust(I.frequency_grid(nf) if nf > 1 else np.array([2e12]), 1e-18)
    if nf == 17:
        dust.kabs[3] = 0.0
    ctx = libsoc.Context(0, seed=1)
    ctx.dust_upload(dust.nu, dust.kabs, dust.ksca, dust.g)
    cid = ctx.grid_upload(cl)
    leaf = cl.leaves()
    T = np.full(cl.n_cells, 10.0, np.float32)
    T[leaf] = _temperatures(kind, leaf.size, rng)
    Td = torch.from_numpy(T).cuda()
    L = torch.empty((nf, leaf.size), dtype=torch.float64, device="cuda")
    ctx.dust_luminosity(cid, Td, L)
    m = L.max(dim=1, keepdim=True).values
    ref = torch.where(m > 0, torch.round(L / torch.where(m > 0, m, torch.ones_like(m)) * 2.0 ** 31), torch.zeros_like(L))
    for lo, n in ((0, nf), (nf // 3, nf - nf // 3)):
        w = torch.full((n, leaf.size), -1, dtype=torch.int64, device="cuda")
        e = torch.empty(n, dtype=torch.float64, device="cuda")
        ctx.dust_emission(cid, Td, w, e, n_per_cell=3, freq_lo=lo, n_freq=n)
        torch.cuda.synchronize()
        assert torch.equal(w, ref[lo:lo + n].to(torch.int64))
        # divided on the host: torch multiplies by the reciprocal of a scalar on the GPU
        np.testing.assert_array_equal(e.cpu().numpy(), m[lo:lo + n, 0].cpu().numpy() / 3.0 / 2.0 ** 31)
    ctx.close()
