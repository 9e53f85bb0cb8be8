"""Total mass over many steps.  A relaxation whose constants do not add up to
1 multiplies the mass of every cell by the same wrong factor in every step,
which one step of any test cannot see."""
import numpy as np
import pytest

import oracle as O
from helpers import LAT, lbm_mod

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return lbm_mod()


def _mass(f):
    return np.asarray(f, dtype=np.longdouble).sum()


@pytest.mark.parametrize("lat,ext", [("D3Q19", (16, 16, 16)), ("D2Q9", (48, 48, 1)),
                                     ("D3Q19", (17, 16, 15)), ("D2Q9", (47, 48, 1))])
@pytest.mark.parametrize("tau", [0.6, 0.7, 0.9, 1.0, 1.1, 1.37])
def test_fp64_mass_follows_the_oracle(lbm, lat, ext, tau):
    """1000 steps of a bubble, the fused step (even rows) and the one-launch
    step (odd rows).  A step stores every population with a rounding of at
    most 2^-54 of it, 2^-55 on average: 1000 times that, as if every rounding
    had one sign."""
    nx, ny, nz = ext
    c = [nx / 2, ny / 2, nz // 2, nx * 0.3]
    f0, _ = O.init(LAT[lat], nx, ny, nz, np.array([c]), 2.0, 0.15, 2.0, 1e-3, 1)
    want = _mass(O.run(LAT[lat], f0, 1000, tau, -5.0))
    if not np.isfinite(want):
        pytest.skip("the method itself is unstable here")
    L = lbm.Lattice(lat, nx, ny, nz, tau=tau, G=-5.0, storage="f64")
    L.write_f(f0)
    L.step(1000)
    got = _mass(L.read("f"))
    L.close()
    assert abs(got - want) / want < 1000 * 2.0 ** -55


@pytest.mark.parametrize("lat,ext", [("D2Q9", (48, 48, 1)), ("D3Q19", (16, 16, 16))])
@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("tau", [0.6, 0.7, 0.8, 0.9, 1.0, 1.1])
def test_multi_lattice_mass_follows_the_oracle(lbm, lat, ext, storage, tau):
    """400 steps of a bubble and its gas, each lattice's mass.  FP64 as above;
    FP32 is off by no more than velocity by velocity, where the weights
    rounded to the storage add up to 1 + 2^-26 (D3Q19) and 1 + 2^-27."""
    nx, ny, nz = ext
    b = np.array([[nx / 2, ny / 2, nz // 2, nx * 0.28]])
    f0 = O.ml_init(LAT[lat], nx, ny, nz, b, 2.0, 0.15, 0.05, 2.0, 1e-3, 3)
    if storage == "f32":
        f0 = f0.astype(np.float32).astype(np.float64)
    fo = O.ml_run(LAT[lat], f0, 400, tau, O.ml_coupling(2, -5.0, 1.0, 0.0))
    fo = fo[0] if isinstance(fo, tuple) else fo
    if not np.isfinite(fo).all():
        pytest.skip("the method itself is unstable here")
    M = lbm.MultiLattice(lat, nx, ny, nz, nl=2, tau=tau, G=-5.0, G_x=1.0, G_b=0.0,
                         storage=storage)
    M.write_f(f0)
    M.step(400)
    fg = M.read_f()
    M.close()
    bound = (400 * 2.0 ** -55 if storage == "f64" else
             400 / tau * (2.0 ** -26 if lat == "D3Q19" else 2.0 ** -27))
    for s in (0, 1):
        want = _mass(fo[s])
        assert abs(_mass(fg[s]) - want) / want < bound, s
