"""The filters' own normals on the GPU.  The FP64 filter's (csrc/soft64.cuh) are held to the bounds of
test_soft64.py, whose host build takes other forms of the reciprocal square root, the leading-zero count
and the wide products than the device does; the FP32 filter's packed pairs are bit for bit the random
stream's (smc2_philox_normals in mixed precision), which test_gpu_rng.py holds to the oracle."""
import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_2311_12973_gb300 import build as B

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pf_fast.cuh"
using namespace smc2;
__global__ void normals64_kernel(int n, const uint32_t* w, double* z) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) s64_normal_pair(w[2 * i], w[2 * i + 1], g_soft64, z[2 * i], z[2 * i + 1]);
}
__global__ void exps_kernel(int n, const double* x, uint64_t* m, int* k) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) m[i] = s64_exp_q57(s64_q57(x[i]), g_soft64, k[i]);
}
// counters (c0, c1, c2, c3) of two particles in turn: their four normals each
__global__ void normals32_kernel(int n_pairs, const uint4* ctr, uint64_t seed, float* z) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_pairs) return;
  const uint4 a = philox4x32_10(ctr[2 * i], seed_key(seed)), b = philox4x32_10(ctr[2 * i + 1], seed_key(seed));
  float2 v[4];
  box_muller2(a.x, b.x, a.y, b.y, v[0], v[1]);
  box_muller2(a.z, b.z, a.w, b.w, v[2], v[3]);
  for (int e = 0; e < 4; ++e) {
    z[8 * i + e] = v[e].x;
    z[8 * i + 4 + e] = v[e].y;
  }
}
extern "C" int normals64(int n, const uint32_t* w, double* z) {
  normals64_kernel<<<(n + 127) / 128, 128>>>(n, w, z);
  return (int)cudaDeviceSynchronize();
}
extern "C" int exps(int n, const double* x, uint64_t* m, int* k) {
  exps_kernel<<<(n + 127) / 128, 128>>>(n, x, m, k);
  return (int)cudaDeviceSynchronize();
}
extern "C" int normals32(int n_pairs, const uint4* ctr, uint64_t seed, float* z) {
  normals32_kernel<<<(n_pairs + 127) / 128, 128>>>(n_pairs, ctr, seed, z);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("normals")
    src, so = str(d / "normals.cu"), str(d / "normals.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", "-O3", "-Xcompiler", "-fPIC", "-I", B.INCLUDE, "-I", B.CSRC,
                    "-shared", "-cudart", "static", src, "-o", so], check=True)
    lib = C.CDLL(so)
    vp = C.c_void_p
    lib.normals64.argtypes = [C.c_int, vp, vp]
    lib.exps.argtypes = [C.c_int, vp, vp, vp]
    lib.normals32.argtypes = [C.c_int, vp, C.c_uint64, vp]
    return lib


def _cuda(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("which", ["random", "first_near_one", "small_angle", "octant_edges"])
def test_fp64_normals(lib, which):
    import torch
    rng = np.random.default_rng(1)
    n = 100000
    w = rng.integers(0, 2 ** 32, (n, 2), dtype=np.uint64).astype(np.uint32)
    k = np.arange(n, dtype=np.uint32)
    if which == "first_near_one":
        w[:, 0] = np.uint32(0xFFFFFFFF) - (k << np.uint32(6))
    elif which == "small_angle":
        w[:, 1] = k << np.uint32(9)
    elif which == "octant_edges":
        w[:, 1] = ((k & np.uint32(7)) << np.uint32(29)) + (((k >> np.uint32(3)) - np.uint32(6000)) << np.uint32(9))
    wd, z = _cuda(w.view(np.int32)), torch.empty((n, 2), dtype=torch.float64, device="cuda")
    assert lib.normals64(n, wd.data_ptr(), z.data_ptr()) == 0
    z = z.cpu().numpy()
    L = np.longdouble
    ua = L(2 * (w[:, 0] >> 9).astype(np.int64) + 1) * L(2) ** -24
    ub = L(2 * (w[:, 1] >> 9).astype(np.int64) + 1) * L(2) ** -24
    turn = np.rint(4 * ub)
    a = 2 * np.arctan2(L(0), L(-1)) * (ub - turn / 4)
    turn = turn.astype(np.int64) % 4
    r = np.sqrt(2 * np.log1p((1 - ua) / ua))
    c, s = np.cos(a), np.sin(a)
    for got, ref in ((z[:, 0], r * np.choose(turn, [c, -s, -c, s])), (z[:, 1], r * np.choose(turn, [s, c, -s, -c]))):
        err = np.abs(got - ref) / np.ldexp(L(1), np.frexp(np.abs(ref))[1] - 53)
        assert err.max() < 1.5 and np.sqrt(np.mean(err ** 2)) < 0.35


def test_exponential(lib):
    import torch
    rng = np.random.default_rng(2)
    x = np.concatenate([rng.uniform(-60, 60, 50000), -np.exp(rng.uniform(-40, 3.6, 50000)), [0.0, 2.0 ** -57, -37.0]])
    m, k = torch.empty(len(x), dtype=torch.int64, device="cuda"), torch.empty(len(x), dtype=torch.int32, device="cuda")
    xd = _cuda(x)
    assert lib.exps(len(x), xd.data_ptr(), m.data_ptr(), k.data_ptr()) == 0
    m, k = m.cpu().numpy().view(np.uint64), k.cpu().numpy()
    got = np.ldexp(np.longdouble(m), k - 61)
    assert np.max(np.abs(got / np.exp(np.longdouble(x)) - 1)) < 2.0 ** -56
    assert m[-3] == 2 ** 61 and k[-3] == 0


def test_fp32_normals_are_the_random_streams(lib):
    import torch
    from paper_2311_12973_gb300 import smc2 as S
    n = 1 << 18
    ctr = _cuda(np.random.default_rng(4).integers(0, 2 ** 32, (n, 4), dtype=np.uint64).astype(np.uint32).view(np.int32))
    z = torch.empty((n, 4), dtype=torch.float32, device="cuda")
    assert lib.normals32(n // 2, ctr.data_ptr(), 77, z.data_ptr()) == 0
    want = torch.empty((n, 4), dtype=torch.float64, device="cuda")
    S.philox_normals(77, ctr, S.PREC_MIXED, z=want)
    assert torch.equal(z.double(), want)
