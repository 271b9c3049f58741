"""psi inside the interface band on the float32 path (eos_fp64 = 1) is the float64 value
rounded to float32, at every float32 density of the band; and with every density inside
the band, a run equals one with float64 everywhere (eos_fp64 = 2) bit for bit, also near the
densities where P = rho/3."""
import ctypes

import numpy as np
import pytest

import oracle as O
from cases import case, lbm_params, oracle_params, shape
from device_ops import load
from paper_2201_12404_gb300 import inputs as I
from paper_2201_12404_gb300 import lbm

pytestmark = pytest.mark.gpu

# a, T/Tc, densities of the state, densities of the phases (P = rho/3 at 0.329.. for a = 0.5)
EOS = {"paper": (0.003, 0.59, (0.3, 7.0), (0.1, 9.0)), "warm": (0.003, 0.85, (1.2, 6.0), (0.5, 7.5)),
       "root": (0.5, 0.6, (0.25, 0.9), (0.2, 1.0)), "at_root": (0.5, 0.6, None, (0.2, 1.0)),
       "dense": (3.0 / 49.0, 0.7, (0.5, 10.0), (0.05, 10.5))}


@pytest.mark.parametrize("precision", [lbm.LBM_FP32, lbm.LBM_FP16DEV], ids=["fp32", "fp16dev"])
@pytest.mark.parametrize("name", list(EOS))
@pytest.mark.parametrize("D", [2, 3])
def test_band_equals_float64_everywhere(D, name, precision):
    a, T, span, phases = EOS[name]
    dims = dict(nx=512, ny=256) if D == 2 else dict(nx=65, ny=50, nz=40)
    out = []
    for eos in (1, 2):
        c = case(D, **dims, Tr=T, a=a, rho_v=phases[0], rho_l=phases[1], kappa=1e-4, precision=precision, eos_fp64=eos)
        sh = shape(c)
        if span is None:
            root = lbm.lbm_psi_sign_changes(lbm_params(c))[0][0]
            rho = root * (1 + 1e-5 * I.rng(3).uniform(-1, 1, sh))
        else:
            rho = I.rng(3).uniform(*span, sh)
        f = O.init_equilibrium(oracle_params(c), rho, np.zeros((D,) + sh)).astype(np.float32).astype(np.float64)
        assert f.sum(axis=0).min() > phases[0] + 0.011 * (phases[1] - phases[0])
        assert f.sum(axis=0).max() < phases[1] - 0.011 * (phases[1] - phases[0])
        with lbm.Domain(lbm_params(c)) as dom:
            dom.lbm_write_populations(f)
            dom.lbm_step(1)
            out.append(dom.lbm_read_populations())
    assert np.array_equal(out[0], out[1], equal_nan=True)


SOURCE = r"""
#include "lbm_kernels.cuh"
#include "lbm_phys.h"
using namespace lbm;
__device__ unsigned long long differ;
__global__ void every_density(DevDomain d, DevDomain d64, unsigned lo, unsigned hi) {
  const unsigned step = gridDim.x * blockDim.x;
  for (unsigned long long b = (unsigned long long)lo + blockIdx.x * blockDim.x + threadIdx.x; b <= hi; b += step) {
    const float rho = __uint_as_float((unsigned)b);
    if (__float_as_uint(psi_of<float>(d, rho)) != __float_as_uint(psi_of<float>(d64, rho))) atomicAdd(&differ, 1ull);
  }
}
extern "C" long long run(double a, double T, double rho_v, double rho_l) {
  lbm_params p = {};
  p.a = a; p.b = 0.095; p.R = 1.0; p.T_over_Tc = T; p.acentric = 0.344;
  p.rho_vapour = rho_v; p.rho_liquid = rho_l; p.nu_liquid = p.nu_vapour = 0.1;
  DevDomain d = {}, d64 = {};
  p.eos_fp64 = 1;
  fill_phys(d, p, 3);
  p.eos_fp64 = 2;
  fill_phys(d64, p, 3);
  if (d.eos != kEosBandPairs || d64.eos != kEosFloat64) return -1;
  unsigned long long n = 0;
  cudaMemcpyToSymbol(differ, &n, sizeof(n));
  const float lo = std::nextafter(d.pf.band_lo, 1e9f), hi = std::nextafter(d.pf.band_hi, 0.0f);
  unsigned first, last;
  memcpy(&first, &lo, 4);
  memcpy(&last, &hi, 4);
  every_density<<<1216, 256>>>(d, d64, first, last);
  if (cudaMemcpyFromSymbol(&n, differ, sizeof(n)) != cudaSuccess) return -2;
  return (long long)n;
}
"""


@pytest.fixture(scope="module")
def differ(tmp_path_factory):
    lib = load(str(tmp_path_factory.mktemp("band")), SOURCE)
    lib.run.restype = ctypes.c_longlong
    lib.run.argtypes = [ctypes.c_double] * 4
    return lib.run


@pytest.mark.parametrize("phases", [(1e-4, 9.5), (0.2, 1.0), (0.05, 10.5)])
@pytest.mark.parametrize("T", [0.4, 0.59, 0.75, 0.9, 1.2])
@pytest.mark.parametrize("a", [1e-3, 0.003, 3.0 / 49.0, 0.5, 20.0])
def test_every_density_of_the_band(differ, a, T, phases):
    assert differ(a, T, *phases) == 0
