"""The FP64 step's psi as an exponential: the function's own source, compiled
for the host (its operations are IEEE ones), against long double."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1708_01608_gb300", "csrc")

SHIM = r"""
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>
#define __device__
#define __forceinline__ inline
struct double2 { double x, y; };
template <class T> inline T __ldg(const T *p) { return *p; }
inline double __drcp_rn(double v) { return 1.0 / v; }
inline int __double2hiint(double v) { int64_t u; memcpy(&u, &v, 8); return (int)(u >> 32); }
inline int __double2loint(double v) { int64_t u; memcpy(&u, &v, 8); return (int)(u & 0xffffffff); }
inline double __hiloint2double(int h, int l) {
  const uint64_t u = ((uint64_t)(uint32_t)h << 32) | (uint32_t)l;
  double v;
  memcpy(&v, &u, 8);
  return v;
}
using std::exp;
using std::fma;
namespace sclbm {
enum { D2Q9 = 0, D3Q19 = 1 };
template <int LAT> struct Lattice;
template <int N, class F> void static_for(F &&f);
}
"""

MAIN = r"""
#include "shim.h"
#include "collide_f64.cuh"
extern "C" void psi(const double *rho, int n, double rho0, double *out, double *err) {
  for (int k = 0; k < n; ++k) {
    out[k] = sclbm::psi_f64(rho[k], rho0, 1.0 / rho0);
    const long double want = -expm1l(-(long double)rho[k] / rho0);
    err[k] = (double)(((long double)out[k] / rho0 - want) * 0x1p53L);
  }
}
"""


@pytest.fixture(scope="module")
def psi(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("psi")
    for name in ("internal.h", "lattice.cuh"):
        (d / name).write_text('#pragma once\n')
    (d / "shim.h").write_text(SHIM)
    (d / "collide_f64.cuh").write_text(open(os.path.join(CSRC, "collide_f64.cuh")).read())
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC",
                    str(d / "main.cpp"), "-o", str(d / "psi.so")], check=True)
    lib = C.CDLL(str(d / "psi.so"))
    p = np.ctypeslib.ndpointer(np.float64)
    lib.psi.argtypes = [p, C.c_int, C.c_double, p, p]

    def f(rho, rho0):
        rho = np.ascontiguousarray(rho, dtype=np.float64)
        out, err = np.empty_like(rho), np.empty_like(rho)
        lib.psi(rho, rho.size, rho0, out, err)
        return out, err
    return f


@pytest.mark.parametrize("rho0", [1.0, 0.05, 0.7, 3.0, 50.0])
def test_psi_error(psi, rho0):
    """Of rho0, in units of u = 2^-53: the two last roundings, of e^x <= 1 and
    of 1 - e^x <= 1, are half a unit each, and the polynomial's are below a
    tenth; where rho0 is not 1, 1/rho0 and rho/rho0 are rounded, at most
    2 u x e^-x <= 2 u / e."""
    rng = np.random.default_rng(1)
    rho = rho0 * np.concatenate([
        rng.uniform(0, 4, 200000), rng.uniform(0, 0.01, 50000), rng.uniform(0, 60, 50000),
        np.exp2(rng.uniform(-60, 9.4, 50000)), [0.0, 5e-324 / rho0]])
    _, err = psi(rho, rho0)
    assert np.isfinite(err).all()
    assert np.abs(err).max() < 1.1 + (0.0 if rho0 == 1.0 else 2 / np.e)
    if rho0 == 1.0:   # rms over a run's densities: that of 1 - exp() is 0.32
        assert np.sqrt((err[:200000] ** 2).mean()) < 0.325


def test_psi_outside_the_table(psi):
    out, _ = psi([700.0, 1e4, np.inf, np.nan, 0.0], 1.0)
    assert (out[[0, 1, 2, 4]] == [1.0, 1.0, 1.0, 0.0]).all() and np.isnan(out[3])
