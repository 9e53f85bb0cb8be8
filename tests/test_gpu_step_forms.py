"""Forms of the step kernels at the sizes and values where each can go wrong."""
import numpy as np
import pytest

import oracle as O
from helpers import LAT, lbm_mod, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return lbm_mod()


@pytest.mark.parametrize("lat,ext", [("D3Q19", (34, 9, 5)), ("D2Q9", (66, 7, 1))])
@pytest.mark.parametrize("rho0", [1.0, 0.05, 0.01, 0.0029, 0.0028, 0.002, 50.0])
def test_fp64_step_over_the_range_of_psi(lbm, lat, ext, rho0):
    """One FP64 step with densities up to 2 and exponents -rho/rho0 from 0
    past -700, where the table-driven exponential hands over.  A population
    is a sum of about 40 terms of at most rho, each rounded once: 40 u rho
    (u = 1.1e-16) is 1.4e-14 of the largest population, rho/3."""
    nx, ny, nz = ext
    q = 19 if lat == "D3Q19" else 9
    _, w = O.velocities(LAT[lat])
    rng = np.random.default_rng(7)
    f0 = (w[:, None, None, None] * rng.uniform(1e-3, 2.0, size=(1, nz, ny, nx))
          * rng.uniform(0.9, 1.1, size=(q, nz, ny, nx)))
    L = lbm.Lattice(lat, nx, ny, nz, tau=0.8, G=-5.0, rho0=rho0, storage="f64", kernel="fused")
    L.write_f(f0)
    L.step(1)
    assert rel_err(L.read("f"), O.run(LAT[lat], f0, 1, 0.8, -5.0, rho0=rho0)) < 2e-14
    L.close()


@pytest.mark.parametrize("lat,ext,nl", [
    ("D2Q9", (1, 9, 1), 2), ("D2Q9", (8, 1, 1), 3), ("D2Q9", (65, 33, 1), 8),
    ("D2Q9", (200, 131, 1), 4), ("D3Q19", (1, 5, 2), 1), ("D3Q19", (65, 3, 4), 4),
    ("D3Q19", (33, 6, 5), 5), ("D3Q19", (64, 4, 3), 8)])
@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_multi_lattice_step_tiles(lbm, lat, ext, nl, storage):
    """One multi-lattice step at the edges of its tiles (one-cell extents,
    ragged tiles, the lattice counts where the split changes), one lattice
    empty.  A step rounds each population in about 60 terms of at most the
    total density nl rho: 60 u nl, u = 1.1e-16 or 6e-8, relative to the
    largest population (rho/3): 180 u nl, and FP32 also rounds the input."""
    nx, ny, nz = ext
    q = 19 if lat == "D3Q19" else 9
    _, w = O.velocities(LAT[lat])
    rng = np.random.default_rng(nl)
    f0 = (w[None, :, None, None, None] * rng.uniform(0.1, 1.0, size=(nl, 1, nz, ny, nx))
          * rng.uniform(0.9, 1.1, size=(nl, q, nz, ny, nx)))
    if nl > 2:
        f0[1] = 0.0
    if storage == "f32":
        f0 = f0.astype(np.float32).astype(np.float64)
    M = lbm.MultiLattice(lat, nx, ny, nz, nl=nl, tau=0.9, G=-5.0, G_x=1.0, G_b=2.0,
                         storage=storage)
    M.write_f(f0)
    M.step(1)
    got = M.read_f()
    want = O.ml_run(LAT[lat], f0, 1, 0.9, O.ml_coupling(nl, -5.0, 1.0, 2.0))
    want = want[0] if isinstance(want, tuple) else want
    u = 1.1e-16 if storage == "f64" else 6e-8
    assert rel_err(got, want) < 180 * nl * u
    M.close()


@pytest.mark.parametrize("lat,ext", [
    ("D3Q19", (8, 1, 1)), ("D3Q19", (16, 5, 2)), ("D3Q19", (40, 28, 20)), ("D3Q19", (64, 64, 48)),
    ("D3Q19", (136, 33, 31)), ("D3Q19", (200, 152, 100)), ("D3Q19", (8, 8, 1500)),
    ("D2Q9", (8, 1, 1)), ("D2Q9", (64, 64, 1)), ("D2Q9", (200, 131, 1)), ("D2Q9", (1032, 700, 1)),
    ("D2Q9", (8, 5000, 1))])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16", "f16r", "bf16r"])
def test_default_plan_gives_the_bits_of_tile_1(lbm, lat, ext, storage):
    """The plan chosen where the caller names no tile: whatever tile and
    chunk count it takes (L2-resident and larger lattices, chunks of one
    plane, one-cell extents), the populations, budgets and residuals are
    those of tile 1, with an injection site."""
    nx, ny, nz = ext
    out = []
    for tile in (0, 1):
        L = lbm.Lattice(lat, nx, ny, nz, tau=0.9, G=-5.0, storage=storage.rstrip("r"),
                        rho_ref=1.8, kernel="fused", tile=tile,
                        mass_residual=storage.endswith("r"))
        L.seed_bubbles([[nx / 2, ny / 2, nz // 2, min(nx, max(ny, nz)) / 5]], 1.8, 0.15, 2.0,
                       1e-3, 5)
        L.inject([1e-3], [4.5e-3])
        L.step(7)
        out.append((L.plan(), L.read("f"), L.read_budgets()))
        L.close()
    (plan, f, b), (_, f1, b1) = out
    assert plan[0] == lbm.KERNEL_FUSED and plan[5] > 0
    assert (f == f1).all() and (b == b1).all()
