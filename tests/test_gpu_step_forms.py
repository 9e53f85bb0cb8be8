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
