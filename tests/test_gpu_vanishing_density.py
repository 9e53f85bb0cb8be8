"""The multi-lattice step where a lattice's density vanishes.  A gas lattice
is exactly zero some twenty cells from its bubble, and the front that moves
into that region falls by up to 1/36 per step: through every power of two of
the storage, the subnormal ones included, down to zero."""
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


@pytest.mark.parametrize("nx,ny,R,nb,storage,steps,tol", [
    (72, 72, 11.0, 2, "f32", 100, 1e-5), (104, 104, 20.0, 2, "f32", 100, 1e-5),
    (176, 176, 38.0, 2, "f32", 100, 1e-5),
    (480, 24, 8.0, 1, "f64", 250, 1e-12)])   # 2^-1022 is passed at step 189
def test_gas_front_through_the_subnormals(lbm, nx, ny, R, nb, storage, steps, tol):
    """The bubble-size sweep's recipe: finite, and the oracle's populations
    within the bounds of the multi-lattice parity tests."""
    c = [nx / 2 - R - 2.0, nx / 2 + R + 2.0][:nb]
    b = np.array([[x, ny / 2, 0.0, R] for x in c])
    M = lbm.MultiLattice("D2Q9", nx, ny, 1, nl=nb + 1, tau=1.0, G=-5.0, G_x=1.0, G_b=2.0,
                         storage=storage)
    M.seed(b, 2.0, 0.15, 0.05, 2.0, 1e-4, 9)
    f0 = M.read_f()
    M.step(steps)
    got = M.read_f()
    M.close()
    assert np.isfinite(got).all()
    want = O.ml_run(O.D2Q9, f0, steps, 1.0, O.ml_coupling(nb + 1, -5.0, 1.0, 2.0))
    want = want[0] if isinstance(want, tuple) else want
    assert rel_err(got, want) < tol


@pytest.mark.parametrize("lat,ext", [("D2Q9", (40, 9, 1)), ("D3Q19", (40, 3, 4))])
@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_one_step_of_vanishing_lattices(lbm, lat, ext, storage):
    """One step of states in which a lattice's density is any of zero, the
    smallest subnormal, the numbers around the one whose reciprocal is
    infinite, and small normal ones: 180 u nl of the largest population, as
    for the multi-lattice step on ordinary densities."""
    nx, ny, nz = ext
    nl, q = 3, 19 if lat == "D3Q19" else 9
    fi = np.finfo(np.float64 if storage == "f64" else np.float32)
    tiny, sub = float(fi.smallest_normal), float(fi.smallest_subnormal)
    _, w = O.velocities(LAT[lat])
    rng = np.random.default_rng(3)
    f0 = (w[None, :, None, None, None] * rng.uniform(0.1, 1.0, size=(nl, 1, nz, ny, nx))
          * rng.uniform(0.9, 1.1, size=(nl, q, nz, ny, nx)))
    small = [0.0, sub, 40 * sub, tiny / 64, tiny / 4, tiny / 2, tiny, 2 * tiny, 1e9 * tiny, 1e-17,
             1e-9]
    for s in (1, 2):
        pick = np.resize(small + [None] * (2 * s), nz * ny * nx).reshape(nz, ny, nx)
        for v in small:
            f0[s][:, pick == v] = w[:, None] * v
            f0[s, 0][pick == v] = max(v, sub) if v else 0.0
    f0 = f0.astype(fi.dtype).astype(np.float64)
    M = lbm.MultiLattice(lat, nx, ny, nz, nl=nl, tau=0.9, G=-5.0, G_x=1.0, G_b=2.0,
                         storage=storage)
    M.write_f(f0)
    M.step(1)
    got = M.read_f()
    M.close()
    assert np.isfinite(got).all()
    want = O.ml_run(LAT[lat], f0, 1, 0.9, O.ml_coupling(nl, -5.0, 1.0, 2.0))
    want = want[0] if isinstance(want, tuple) else want
    assert rel_err(got, want) < 180 * nl * (1.1e-16 if storage == "f64" else 6e-8)


@pytest.mark.parametrize("lat,ext", [("D2Q9", (40, 9, 1)), ("D3Q19", (40, 3, 4))])
@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_one_step_where_every_lattice_vanishes(lbm, lat, ext, storage):
    """As above with cells in which the total density is subnormal, whose
    reciprocal the common velocity must not take."""
    nx, ny, nz = ext
    nl, q = 2, 19 if lat == "D3Q19" else 9
    fi = np.finfo(np.float64 if storage == "f64" else np.float32)
    tiny = float(fi.smallest_normal)
    _, w = O.velocities(LAT[lat])
    rng = np.random.default_rng(4)
    f0 = (w[None, :, None, None, None] * rng.uniform(0.1, 1.0, size=(nl, 1, nz, ny, nx))
          * rng.uniform(0.9, 1.1, size=(nl, q, nz, ny, nx)))
    scale = np.resize([1.0, 1.0, tiny / 4, 1.0, tiny / 2048, 1.0, tiny], (nz, ny, nx))
    f0 = (f0 * scale).astype(fi.dtype).astype(np.float64)
    M = lbm.MultiLattice(lat, nx, ny, nz, nl=nl, tau=0.9, G=-5.0, G_x=1.0, G_b=2.0,
                         storage=storage)
    M.write_f(f0)
    M.step(1)
    got = M.read_f()
    M.close()
    assert np.isfinite(got).all()
    want = O.ml_run(LAT[lat], f0, 1, 0.9, O.ml_coupling(nl, -5.0, 1.0, 2.0))
    want = want[0] if isinstance(want, tuple) else want
    assert rel_err(got, want) < 180 * nl * (1.1e-16 if storage == "f64" else 6e-8)


@pytest.mark.parametrize("lat,ext", [("D2Q9", (40, 9, 1)), ("D3Q19", (40, 3, 4)),
                                     ("D2Q9", (41, 9, 1)), ("D3Q19", (41, 3, 4))])
def test_fp64_step_where_the_density_vanishes(lbm, lat, ext):
    """The single-component FP64 step (even rows fused, odd ones in one
    launch) with cells of subnormal density: 40 roundings per population."""
    nx, ny, nz = ext
    q = 19 if lat == "D3Q19" else 9
    tiny = float(np.finfo(np.float64).smallest_normal)
    _, w = O.velocities(LAT[lat])
    rng = np.random.default_rng(5)
    f0 = (w[:, None, None, None] * rng.uniform(0.1, 1.0, size=(1, nz, ny, nx))
          * rng.uniform(0.9, 1.1, size=(q, nz, ny, nx)))
    f0 = f0 * np.resize([1.0, 1.0, tiny / 4, 1.0, tiny / 2048, 1.0, tiny], (nz, ny, nx))
    L = lbm.Lattice(lat, nx, ny, nz, tau=0.8, G=-5.0, storage="f64")
    L.write_f(f0)
    L.step(1)
    got = L.read("f")
    L.close()
    assert np.isfinite(got).all()
    assert rel_err(got, O.run(LAT[lat], f0, 1, 0.8, -5.0)) < 2e-14
