"""Lattices far narrower than a kernel's tile: rows or columns of a few cells,
one row or one plane.  A form that leaves most of its threads idle there takes
many times as long as on a cube of as many cells."""
import time

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


def _time(step, sync, n=20):
    """seconds per step, the best of five"""
    step(n)
    sync()
    best = 1e9
    for _ in range(5):
        t = time.perf_counter()
        step(n)
        sync()
        best = min(best, (time.perf_counter() - t) / n)
    return best


# both sides of the dispatch: boxes of whole and of split axes with ragged
# ends, one row, one plane, rows just narrower and wider than a warp
BOX = [("D3Q19", (3, 46, 450)), ("D3Q19", (1, 70, 171)), ("D3Q19", (1, 1, 60001)),
       ("D3Q19", (5, 20001, 1)), ("D3Q19", (20001, 5, 1)), ("D3Q19", (9, 3, 4001)),
       ("D3Q19", (31, 8, 2016)), ("D3Q19", (33, 5051, 3)), ("D3Q19", (17, 60, 343)),
       ("D2Q9", (1, 60001, 1)), ("D2Q9", (3, 33333, 1)), ("D2Q9", (33, 30303, 1)),
       ("D2Q9", (9, 111111, 1))]


@pytest.mark.parametrize("lat,ext", BOX)
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16", "f64"])
def test_box_form(lbm, lat, ext, storage):
    """The step of the automatic choice against the two-pass kernels, two
    injection sites in one cell and one beside it: the same bits in FP32
    arithmetic; in FP64 seven steps of 40 roundings of at most rho per
    population (1.4e-14 of the largest a step)."""
    nx, ny, nz = ext
    out = []
    for kernel in ("auto", "two_pass"):
        L = lbm.Lattice(lat, nx, ny, nz, tau=0.9, G=-5.0, storage=storage, rho_ref=1.8,
                        kernel=kernel)
        x, y, z = nx // 2, ny // 2, nz // 2
        L.seed_bubbles([[x, y, z, 3.0], [x, y, z, 1.0], [(x + 1) % nx, y, z, 1.0]], 1.8, 0.15,
                       2.0, 1e-3, 5)
        L.inject([1e-3, 2e-3, 3e-3], [4.5e-3, 9e-3, 1.0])
        L.step(7)
        out.append((L.read("f"), L.read_budgets()))
        L.close()
    (f, b), (f1, b1) = out
    assert (b == b1).all()
    if storage == "f64":
        assert np.abs(f - f1).max() < 7 * 1.4e-14 * np.abs(f1).max()
    else:
        assert (f == f1).all()


@pytest.mark.parametrize("lat,ext", [("D3Q19", (3, 460, 450)), ("D3Q19", (1, 1, 300001)),
                                     ("D3Q19", (9, 3, 22222)), ("D2Q9", (3, 333333, 1))])
@pytest.mark.parametrize("storage", ["f32", "f16", "f64"])
def test_automatic_choice_is_not_slower_than_two_passes(lbm, lat, ext, storage):
    """Half as long again as the two-pass kernels at most (forms that idle
    take 2 to 25 times as long)."""
    t = {}
    for kernel in ("auto", "two_pass"):
        L = lbm.Lattice(lat, *ext, tau=0.9, storage=storage, rho_ref=1.8, kernel=kernel)
        L.seed_bubbles([[1.0, 1.0, 0.0, 1.0]], 1.8, 0.15, 2.0, 1e-3, 5)
        t[kernel] = _time(L.step, L.sync)
        L.close()
    assert t["auto"] < 1.5 * t["two_pass"], t


@pytest.mark.parametrize("ext", [(1, 1, 300000), (3, 816, 816), (8, 500, 500), (5, 400000, 1)])
def test_static_step_on_narrow_lattices(lbm, ext):
    """No more than three times as long as the cube of about as many cells
    (2 to 30 times where most threads idle)."""
    import torch
    stream = torch.cuda.current_stream().cuda_stream

    def per_step(nx, ny, nz):
        a = torch.full((19, nx * ny * nz), 0.1, device="cuda")
        b = a.clone()
        p, q = a.data_ptr(), b.data_ptr()

        def step(n):
            for _ in range(n // 2):
                lbm.step_static_f32("D3Q19", nx, ny, nz, 0.9, -5.0, 1.0, p, q, stream)
                lbm.step_static_f32("D3Q19", nx, ny, nz, 0.9, -5.0, 1.0, q, p, stream)
        return _time(step, torch.cuda.synchronize)
    n = round((ext[0] * ext[1] * ext[2]) ** (1 / 3))
    t, cube = per_step(*ext), per_step(n, n, n)
    assert t < 3 * cube, (t, cube)


@pytest.mark.parametrize("lat,ext,nl", [
    ("D2Q9", (1, 300, 1), 3), ("D2Q9", (5, 211, 1), 8), ("D2Q9", (9, 1200, 1), 2),
    ("D2Q9", (63, 65, 1), 4), ("D2Q9", (64, 40, 1), 1), ("D3Q19", (1, 40, 9), 3),
    ("D3Q19", (3, 21, 30), 8), ("D3Q19", (67, 3, 5), 2), ("D3Q19", (130, 2, 3), 5)])
@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_multi_lattice_tiles_of_whole_rows(lbm, lat, ext, nl, storage):
    """One multi-lattice step where a tile takes whole rows (D2Q9) and on runs
    of cells that cross rows (D3Q19): 180 u nl of the largest population, as
    for the tiles of the step."""
    nx, ny, nz = ext
    q = 19 if lat == "D3Q19" else 9
    _, w = O.velocities(LAT[lat])
    rng = np.random.default_rng(nl)
    f0 = (w[None, :, None, None, None] * rng.uniform(0.1, 1.0, size=(nl, 1, nz, ny, nx))
          * rng.uniform(0.9, 1.1, size=(nl, q, nz, ny, nx)))
    if storage == "f32":
        f0 = f0.astype(np.float32).astype(np.float64)
    M = lbm.MultiLattice(lat, nx, ny, nz, nl=nl, tau=0.9, G=-5.0, G_x=1.0, G_b=2.0,
                         storage=storage)
    M.write_f(f0)
    M.step(1)
    got = M.read_f()
    M.close()
    want = O.ml_run(LAT[lat], f0, 1, 0.9, O.ml_coupling(nl, -5.0, 1.0, 2.0))
    want = want[0] if isinstance(want, tuple) else want
    assert rel_err(got, want) < 180 * nl * (1.1e-16 if storage == "f64" else 6e-8)


@pytest.mark.parametrize("lat,ext,cube", [
    ("D3Q19", (1, 300, 300), (45, 45, 44)), ("D3Q19", (3, 20000, 3), (57, 57, 55)),
    ("D2Q9", (1, 160000, 1), (400, 400, 1)), ("D2Q9", (9, 30000, 1), (520, 520, 1))])
@pytest.mark.parametrize("nl,storage", [(1, "f32"), (3, "f32"), (3, "f64")])
def test_multi_lattice_step_on_narrow_lattices(lbm, lat, ext, cube, nl, storage):
    """No more than three times as long as a square or cube of about as many
    cells (2 to 16 times where most threads idle)."""
    import torch
    t = []
    for e in (ext, cube):
        M = lbm.MultiLattice(lat, *e, nl=nl, tau=0.9, storage=storage)
        M.seed([[1.0, 1.0, 0.0, 1.0]] * (nl - 1), 1.8, 0.15, 0.05, 2.0, 1e-3, 5)
        t.append(_time(M.step, torch.cuda.synchronize))
        M.close()
    assert t[0] < 3 * t[1], t


@pytest.mark.parametrize("ext,storage", [
    ((8, 500, 500), "f32"), ((8, 250000, 1), "f32"), ((24, 289, 289), "f32"),
    ((16, 8, 15625), "f32"), ((24, 83333, 1), "f16"), ((16, 354, 354), "f16"),
    ((24, 289, 289), "f16r")])
def test_default_plan_on_narrow_lattices(lbm, ext, storage):
    """The plan taken where the caller names no tile against tile 1 with its
    own chunk rule: a fifth slower at most (1.3 to 2.2 times where the plan
    counts cells only)."""
    t = {}
    for tile in (0, 1):
        L = lbm.Lattice("D3Q19", *ext, tau=0.9, storage=storage.rstrip("r"), rho_ref=1.8,
                        mass_residual=storage.endswith("r"), kernel="fused", tile=tile)
        L.seed_bubbles([[1.0, 1.0, 0.0, 1.0]], 1.8, 0.15, 2.0, 1e-3, 5)
        t[tile] = _time(L.step, L.sync)
        L.close()
    assert t[0] < 1.2 * t[1], t
