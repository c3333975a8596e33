"""The step kernels' own reciprocal, reciprocal square root (FP64) and two-float logarithm against
CUDA's double functions: a small program around the header, compiled here for the purpose."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "step_impl.cuh"
using namespace adress;
__global__ void k_div(const double* x, double* r, double* q, double* r_ref, double* q_ref, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    r[i] = rcp_nr(x[i]);
    q[i] = rsqrt_nr(x[i]);
    r_ref[i] = 1.0 / x[i];
    q_ref[i] = 1.0 / sqrt(x[i]);
  }
}
__global__ void k_log(const float* g, const float4* tab, double* l, double* ref, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    Sum2 s;
    acc_log(s, g[i], tab);
    l[i] = s.value();
    ref[i] = log((double)g[i]);
  }
}
extern "C" int run_div(const double* x, double* r, double* q, double* r_ref, double* q_ref, int n) {
  k_div<<<256, 128>>>(x, r, q, r_ref, q_ref, n);
  return (int)cudaDeviceSynchronize();
}
extern "C" int run_log(const float* g, double* l, double* ref, int n) {
  float4 tab[128], *d = nullptr;
  fill_log_table(tab);
  cudaError_t e = cudaMalloc(&d, sizeof(tab));
  if (e == cudaSuccess) e = cudaMemcpy(d, tab, sizeof(tab), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) k_log<<<256, 128>>>(g, d, l, ref, n);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  cudaFree(d);
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1806_10841_gb300 import build

    d = tmp_path_factory.mktemp("device_math")
    (d / "math.cu").write_text(SOURCE)
    cmd = [build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-shared", "-cudart", "static", "-o",
           str(d / "math.so"), str(d / "math.cu")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return ctypes.CDLL(str(d / "math.so"))


def call(lib, name, x, n_out):
    import torch

    x = torch.from_numpy(x).cuda()
    out = [torch.zeros(x.numel(), dtype=torch.float64, device="cuda") for _ in range(n_out)]
    torch.cuda.synchronize()
    assert getattr(lib, name)(*[ctypes.c_void_p(t.data_ptr()) for t in (x, *out)], ctypes.c_int(x.numel())) == 0
    return [t.cpu().numpy() for t in out]


def ulps(a, b):
    """Places between positive doubles."""
    return np.abs(a.view(np.int64) - b.view(np.int64))


def test_reciprocal_and_reciprocal_square_root(lib):
    """One and two units in the last place (the derivation is beside the functions; the reference
    1 / sqrt is itself rounded twice, one unit more)."""
    rng = np.random.default_rng(1)
    x = np.concatenate([rng.uniform(0.1, 10.0, 1 << 20), np.exp2(rng.uniform(-300.0, 300.0, 1 << 20)),
                        np.nextafter(np.exp2(np.arange(-300.0, 301.0)), 0.0), np.exp2(np.arange(-300.0, 301.0)),
                        np.nextafter(np.exp2(np.arange(-300.0, 301.0)), np.inf)])
    r, q, r_ref, q_ref = call(lib, "run_div", x, 4)
    print("reciprocal", ulps(r, r_ref).max(), "reciprocal square root", ulps(q, q_ref).max(), "units in the last place")
    assert ulps(r, r_ref).max() <= 1
    assert ulps(q, q_ref).max() <= 3
    r, q, _, _ = call(lib, "run_div", np.array([0.0, np.nan]), 4)
    assert not np.isfinite(r).any() and not np.isfinite(q).any()  # the force's check sees them


def test_two_float_logarithm(lib):
    """Within 1e-11 + 8e-12 |e| (g = 2^e m), the bound stated beside the function."""
    rng = np.random.default_rng(2)
    g = np.concatenate([rng.uniform(0.5, 1.0, 1 << 20), rng.uniform(0.001, 0.5, 1 << 20), np.exp2(rng.uniform(-126, 127, 1 << 20)),
                        1.0 + np.arange(512) / 512.0, 0.5 + np.arange(512) / 1024.0]).astype(np.float32)
    l, ref = call(lib, "run_log", g, 2)
    e = np.floor(np.log2(g.astype(np.float64)))
    err = np.abs(l - ref)
    for lo, hi in ((0.5, 1.0), (0.2, 0.5), (0.0, 0.2)):
        m = (g >= lo) & (g < hi)
        print(f"{lo} <= g < {hi}: largest error {err[m].max():.2e}, mean {np.mean((l - ref)[m]):+.2e}")
    assert (err <= 1e-11 + 8e-12 * np.abs(e)).all()
    special = np.array([0.0, -1.0, np.nan, np.inf, 1e-40], dtype=np.float32)
    l, ref = call(lib, "run_log", special, 2)
    assert l[0] == -np.inf and np.isnan(l[1]) and np.isnan(l[2]) and l[3] == np.inf
    assert abs(l[4] - ref[4]) < 1e-4
