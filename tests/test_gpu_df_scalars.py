"""The scalars on the serial chains of the factorizations, from the kernels' own headers: the double-float
reciprocal of a pivot and Householder reflector, and a warp's FP64 reflector, against FP64 arithmetic."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from gpu_util import dev, require_lib

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "dense_kernels.cuh"
using namespace hbs;
__global__ void k_recip(const cplx* d, cplx* r, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r[i] = from_dfc_bits(dfc_recip(to_dfc_bits(d[i])));
}
// reflector of (x0, x1): v0, beta, tau
__global__ void k_reflect(const cplx* x, cplx* v0, cplx* beta, double* tau, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float sh = 0.f, sl = 0.f, th, tl;
  df_abs2_acc(to_dfc_bits(x[2 * i + 1]), sh, sl);
  df_norm(sh, sl);
  dfc v, b;
  df_householder(to_dfc_bits(x[2 * i]), sh, sl, &v, &b, &th, &tl);
  v0[i] = from_dfc_bits(v);
  beta[i] = from_dfc_bits(b);
  tau[i] = f2d_bits(th) + f2d_bits(tl);
}
__global__ void k_warp_reflect(const cplx* x, cplx* v0, cplx* beta, double* tau, int n) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x & 31;
  if (i >= n) return;
  cplx v, b;
  double t;
  warp_householder(x[2 * i], cabs2(x[2 * i + 1]), lane, &v, &b, &t);
  if (lane == 17) { v0[i] = v; beta[i] = b; tau[i] = t; }
}
extern "C" int warp_reflect(const void* x, void* v0, void* beta, void* tau, int n) {
  k_warp_reflect<<<(n + 3) / 4, 128>>>((const cplx*)x, (cplx*)v0, (cplx*)beta, (double*)tau, n);
  return (int)cudaDeviceSynchronize();
}
extern "C" int recip(const void* d, void* r, int n) {
  k_recip<<<(n + 127) / 128, 128>>>((const cplx*)d, (cplx*)r, n);
  return (int)cudaDeviceSynchronize();
}
extern "C" int reflect(const void* x, void* v0, void* beta, void* tau, int n) {
  k_reflect<<<(n + 127) / 128, 128>>>((const cplx*)x, (cplx*)v0, (cplx*)beta, (double*)tau, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    require_lib()
    from paper_1301_1247_gb300 import build
    d = tmp_path_factory.mktemp("probe")
    (d / "p.cu").write_text(SOURCE)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O3", "-shared", "-Xcompiler", "-fPIC",
                    "-I", build.CSRC, str(d / "p.cu"), "-o", str(d / "p.so")], check=True)
    return ctypes.CDLL(os.fspath(d / "p.so"))


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def _complex(rng, shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def test_reciprocal(probe):
    """|d|^2, its quotient and the product are each within a few roundings of 2^-48: 1e-13 is ample."""
    n = 100000
    d = _complex(np.random.default_rng(0), n) * 10.0 ** np.linspace(-12, 12, n)
    r = dev(np.zeros(n, complex))
    assert probe.recip(_ptr(dev(d)), _ptr(r), n) == 0
    assert np.abs(r.cpu().numpy() * d - 1).max() < 1e-13


@pytest.mark.parametrize("scale,bound", [(1.0, 1e-13), (1e-9, 1e-13), (1e6, 1e-13), (7e-19, 1e-6)])
def test_reflector(probe, scale, bound):
    """H = I - tau v v^H takes x to beta e_1 and beta has the norm of x.  At 7e-19 the squares (5e-37) have
    neighbours 3e-9 apart in FP32: the reflector is that coarse, but the column is not taken for an empty one."""
    n = 20000
    x = _complex(np.random.default_rng(1), (n, 2)) * scale
    v0, beta, tau = dev(np.zeros(n, complex)), dev(np.zeros(n, complex)), dev(np.zeros(n))
    assert probe.reflect(_ptr(dev(x)), _ptr(v0), _ptr(beta), _ptr(tau), n) == 0
    v = np.stack([v0.cpu().numpy(), x[:, 1]], axis=1)
    b, t = beta.cpu().numpy(), tau.cpu().numpy()
    hx = x - v * (t * np.sum(np.conj(v) * x, axis=1))[:, None]
    norm = np.linalg.norm(x, axis=1)
    big = norm > 0.7 * scale
    assert (np.abs(np.abs(b) - norm) / norm)[big].max() < bound
    assert (np.linalg.norm(hx - np.stack([b, 0 * b], axis=1), axis=1) / norm)[big].max() < bound


@pytest.mark.parametrize("scale", [1.0, 1e-140, 3e100])
@pytest.mark.parametrize("head", [1.0, 0.0, 1e-12, 1e12])
def test_warp_reflector_is_fp64(probe, scale, head):
    """A few roundings of 2^-53 in each of |x|, the phase and tau: 4e-15 in all.  `head` is the first entry's size
    beside the other's."""
    n = 20000
    x = _complex(np.random.default_rng(2), (n, 2)) * scale / max(head, 1.0)
    x[:, 0] *= head
    v0, beta, tau = dev(np.zeros(n, complex)), dev(np.zeros(n, complex)), dev(np.zeros(n))
    assert probe.warp_reflect(_ptr(dev(x)), _ptr(v0), _ptr(beta), _ptr(tau), n) == 0
    s = np.abs(x).max(axis=1)[:, None]
    v, b, t = np.stack([v0.cpu().numpy(), x[:, 1]], axis=1) / s, beta.cpu().numpy() / s[:, 0], tau.cpu().numpy() * s[:, 0] ** 2
    y = x / s
    hx = y - v * (t * np.sum(np.conj(v) * y, axis=1))[:, None]
    norm = np.linalg.norm(y, axis=1)
    assert (np.abs(np.abs(b) - norm) / norm).max() < 4e-15
    assert (np.linalg.norm(hx - np.stack([b, 0 * b], axis=1), axis=1) / norm).max() < 4e-15
