"""The tanh shortcut of real couplings: the figure its margin rests on, over every float, and decisions
whose sums are placed within the margin of zero, against the float32 rule."""
import ctypes as C
import functools
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle
from paper_2604_17109_gb300 import build as pkg_build

from gpu_helpers import pim

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "real_rule.cuh"
__global__ void gap_kernel(unsigned int* gap, unsigned int* odd) {
  float most = 0.0f;
  for (unsigned long long k = blockIdx.x * 256ull + threadIdx.x; k < (1ull << 32); k += gridDim.x * 256ull) {
    const float x = __uint_as_float(static_cast<unsigned int>(k));
    const float a = pim::tanh_approx(x), t = tanhf(x);
    if (isnan(a) != isnan(x) || isnan(t) != isnan(x)) atomicAdd(odd, 1u);
    if (!isnan(x)) most = fmaxf(most, fabsf(a - t));  // exact: neighbours within a factor of two, or tiny
  }
  atomicMax(gap, __float_as_uint(most));
}
__global__ void tanh_kernel(const float* x, float* y, int n) {
  const int k = blockIdx.x * 256 + threadIdx.x;
  if (k < n) y[k] = tanhf(x[k]);
}
extern "C" float gap_bound() { return pim::kTanhGap; }
extern "C" int measure_gap(unsigned int* out) {
  gap_kernel<<<1216, 256>>>(out, out + 1);
  return cudaDeviceSynchronize();
}
extern "C" int tanh_values(const float* x, float* y, int n) {
  tanh_kernel<<<(n + 255) / 256, 256>>>(x, y, n);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def device(tmp_path_factory):
    d = tmp_path_factory.mktemp("tanh")
    (d / "tanh.cu").write_text(SOURCE)
    so = str(d / "tanh.so")
    subprocess.run([pkg_build._nvcc(), "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", pkg_build.CSRC]
                   + pkg_build.ARCH + ["-o", so, os.path.join(str(d), "tanh.cu")], check=True)
    lib = C.CDLL(so)
    lib.gap_bound.restype = C.c_float
    lib.measure_gap.argtypes = [C.c_void_p]
    lib.tanh_values.argtypes = [C.c_void_p, C.c_void_p, C.c_int]
    return lib


def test_gap_over_every_float(device):
    out = torch.zeros(2, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert device.measure_gap(out.data_ptr()) == 0
    gap, odd = out.cpu().numpy().view(np.uint32)
    gap = np.array([gap], np.uint32).view(np.float32)[0]
    print(f"largest |tanh.approx - tanhf|: {gap:.4g}")
    assert odd == 0
    assert 0.0 < gap <= device.gap_bound()


R = 32768  # replicas: eight of them draw a given level


@functools.lru_cache(maxsize=1)
def _keys(n):
    return oracle.noise_draw16(21, 0, np.arange(R)[:, None], 0, np.arange(n)[None, :]) >> 4


@pytest.mark.parametrize("xi,eta", [(0.5, 0.3), (0.0, 0.25), (2.0, 0.8)])
@pytest.mark.parametrize("n", [64, 256, 300])  # the fused kernel in two capacities, the large-N kernel
def test_decisions_within_the_margin(device, n, xi, eta):
    """No couplings: a spin's field is its bias, here the one that puts the sum of one noise level
    within 2e-5 of zero (the approximation is off by up to 8e-6 there, the margin is 4.4e-5 and more).
    One replica in 4096 draws that level; every decision has to be the rule's."""
    P = pim()
    g = np.random.default_rng(n)
    xi, eta = np.float32(xi), np.float32(eta)
    z = P.pim_noise_levels("gauss")
    s = np.where(g.random(n) < 0.5, -1, 1).astype(np.float32)
    rest = np.float64(xi) * s[:, None] + np.float64(eta) * z[None, :]
    key = np.array([g.choice(np.flatnonzero(np.abs(r) < 0.97)) for r in rest])
    tau = np.clip(-rest[np.arange(n), key] + g.uniform(-2e-5, 2e-5, n), -0.999, 0.999)
    h = np.arctanh(tau).astype(np.float32)
    x, y = torch.tensor(h, device="cuda"), torch.zeros(n, device="cuda")
    torch.cuda.synchronize()
    assert device.tanh_values(x.data_ptr(), y.data_ptr(), n) == 0
    tau = y.cpu().numpy()

    hd = P.pim_create(np.zeros((n, n), np.float32), h, 1.0)
    try:
        P.pim_set_schedule(hd, np.ones(1, np.float32), np.array([eta], np.float32), float(xi))
        P.pim_anneal(hd, R, 1, 21, init_spins=np.tile(s.astype(np.int8), (R, 1)))
        got = P.pim_final_state(hd, n)
    finally:
        P.pim_destroy(hd)
    a = (tau + xi * s).astype(np.float32)  # exact products: s is +-1
    delta = a[None, :] + (eta * z)[_keys(n)]
    close = np.abs(delta) < 2.1e-5
    assert close.sum() > 4 * n
    assert delta.dtype == np.float32
    assert np.array_equal(got, np.where(delta >= 0, 1, -1))
