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


ROWS = [("D3Q19", (1, 1, 1)), ("D3Q19", (1, 9, 4)), ("D3Q19", (29, 6, 3)), ("D3Q19", (30, 7, 2)),
        ("D3Q19", (31, 5, 1)), ("D3Q19", (61, 23, 70)), ("D3Q19", (33, 1, 5)), ("D2Q9", (1, 1, 1)),
        ("D2Q9", (125, 9, 1)), ("D2Q9", (126, 8, 1)), ("D2Q9", (127, 1500, 1)), ("D2Q9", (255, 2, 1))]


# enough cells for the x-pair form: tiles (64 x 8, 128 x 4) with one column or
# row over, an odd and an even last pair, rows narrower than a halo box
WIDE = [("D3Q19", (129, 33, 150)), ("D3Q19", (65, 57, 170)), ("D3Q19", (130, 9, 520)),
        ("D3Q19", (127, 40, 120)), ("D3Q19", (201, 150, 21)), ("D3Q19", (1, 800, 760)),
        ("D3Q19", (3, 460, 450)), ("D3Q19", (600001, 1, 1))]


@pytest.mark.parametrize("lat,ext", ROWS + WIDE)
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_one_launch_step_gives_the_bits_of_the_two_pass_step(lbm, lat, ext, storage):
    """Rows that are no multiple of 16 bytes, at the edges of the march's
    tiles (30 x 6 and 126 cells) and chunks and in the x-pair form: the step an automatic choice
    takes there has the populations and budgets of the two-pass kernels, with
    two injection sites in one cell and a neighbouring one."""
    nx, ny, nz = ext
    out = []
    for kernel in ("auto", "two_pass"):
        L = lbm.Lattice(lat, nx, ny, nz, tau=0.9, G=-5.0, storage=storage, rho_ref=1.8,
                        kernel=kernel)
        x, y, z = nx // 2, ny // 2, nz // 2
        L.seed_bubbles([[x, y, z, nx / 5], [x, y, z, 1.0], [(x + 1) % nx, y, z, 1.0]], 1.8, 0.15,
                       2.0, 1e-3, 5)
        L.inject([1e-3, 2e-3, 3e-3], [4.5e-3, 9e-3, 1.0])
        L.step(7)
        out.append((L.plan()[0], L.read("f"), L.read_budgets()))
        L.close()
    (kind, f, b), (kind1, f1, b1) = out
    assert kind == kind1 == lbm.KERNEL_TWO_PASS
    assert (f == f1).all() and (b == b1).all()


@pytest.mark.parametrize("lat,ext", ROWS)
def test_one_launch_step_fp64(lbm, lat, ext):
    """The FP64 form on odd rows: one step, 40 roundings of at most rho per
    population as above (2e-14 of the largest population)."""
    nx, ny, nz = ext
    q = 19 if lat == "D3Q19" else 9
    _, w = O.velocities(LAT[lat])
    rng = np.random.default_rng(nx + ny)
    f0 = (w[:, None, None, None] * rng.uniform(0.1, 2.0, size=(1, nz, ny, nx))
          * rng.uniform(0.9, 1.1, size=(q, nz, ny, nx)))
    L = lbm.Lattice(lat, nx, ny, nz, tau=0.8, G=-5.0, storage="f64")
    L.write_f(f0)
    L.step(1)
    assert rel_err(L.read("f"), O.run(LAT[lat], f0, 1, 0.8, -5.0)) < 2e-14
    L.close()


@pytest.mark.parametrize("lat,ext", ROWS + [("D3Q19", (32, 12, 3)), ("D2Q9", (128, 4, 1))])
def test_static_step_gives_the_bits_of_the_two_pass_step(lbm, lat, ext):
    import torch
    nx, ny, nz = ext
    q = 19 if lat == "D3Q19" else 9
    _, w = O.velocities(LAT[lat])
    rng = np.random.default_rng(nx * ny)
    f0 = (w[:, None, None, None] * rng.uniform(0.1, 2.0, size=(1, nz, ny, nx))
          * rng.uniform(0.9, 1.1, size=(q, nz, ny, nx))).astype(np.float32)
    L = lbm.Lattice(lat, nx, ny, nz, tau=0.8, G=-5.0, storage="f32", kernel="two_pass",
                    rho_ref=0.0)
    L.write_f(f0.astype(np.float64))
    L.step(4)
    a = torch.from_numpy(f0).cuda()
    b = torch.empty_like(a)
    for _ in range(4):
        lbm.step_static_f32(lat, nx, ny, nz, 0.8, -5.0, 1.0, a.data_ptr(), b.data_ptr(),
                            torch.cuda.current_stream().cuda_stream)
        a, b = b, a
    assert (a.cpu().numpy().astype(np.float64) == L.read("f").reshape(f0.shape)).all()
    L.close()
