"""GPU test of the inner products' sums within a warp (lane_sums.cuh): eight rows per lane (four in float64),
two basis vectors against u and w.  Integers whose sums float32 cannot hold have to come out exactly, and
random rows within the roundings of two rows per float32 sum.  The header is compiled into a small kernel."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = """
#include "common.cuh"
#include "lane_sums.cuh"
using namespace swm;
template <typename TV, int KR, typename Sum>
__global__ void k_sums(const cplx<TV>* __restrict__ rows, double* __restrict__ out) {
  const int lane = threadIdx.x;
  const cplx<TV>* at = rows + (size_t)blockIdx.x * 4 * 32 * KR;  // v0, v1, x, y
  cplx<TV> r[4][KR];
  for (int a = 0; a < 4; ++a)
    for (int k = 0; k < KR; ++k) r[a][k] = at[(a * KR + k) * 32 + lane];
  Sum d[8];
  lane_dot(r[0], r[2], d);
  lane_dot(r[0], r[3], d + 2);
  lane_dot(r[1], r[2], d + 4);
  lane_dot(r[1], r[3], d + 6);
  const double t = widen(warp_sum8(d, lane));
  if ((lane & 3) == 0) out[blockIdx.x * 8 + (lane >> 2)] = t;
}
extern "C" int run(int f64, int warps, const void* rows, void* out) {
  if (f64)
    k_sums<double, 4, double><<<warps, 32>>>((const c128*)rows, (double*)out);
  else
    k_sums<float, 8, FPair><<<warps, 32>>>((const c64*)rows, (double*)out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2410_03060_gb300 import build as B

    d = tmp_path_factory.mktemp("lane_sums")
    (d / "sums.cu").write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-shared", str(d / "sums.cu"), "-o", str(d / "sums.so")],
                   check=True)
    return ctypes.CDLL(str(d / "sums.so"))


def _sums(lib, rows):
    import torch

    dev = torch.from_numpy(np.ascontiguousarray(rows)).cuda()
    out = torch.zeros(len(rows), 8, dtype=torch.float64, device="cuda")
    assert lib.run(int(rows.dtype == np.complex128), len(rows), ctypes.c_void_p(dev.data_ptr()),
                   ctypes.c_void_p(out.data_ptr())) == 0
    return out.cpu().numpy().reshape(-1, 2, 2, 2)  # vector, u or w, re and im


def _want(rows):
    w = rows.astype(np.complex128).reshape(len(rows), 4, -1)
    s = np.einsum("bvn,bxn->bvx", w[:, :2].conj(), w[:, 2:])
    return np.stack([s.real, s.imag], -1)


@pytest.mark.parametrize("dtype,kr", [(np.complex64, 8), (np.complex128, 4)])
def test_integer_sums_are_exact(lib, dtype, kr):
    rng = np.random.default_rng(3)
    rows = (rng.integers(900, 1024, (40, 4, kr, 32)) + 1j * rng.integers(-1024, 1024, (40, 4, kr, 32))).astype(dtype)
    # products of two rows stay below 2^23, the sums of 128 and 256 rows reach 2^27 and 2^28
    assert np.array_equal(_sums(lib, rows), _want(rows))


@pytest.mark.parametrize("dtype,kr,eps", [(np.complex64, 8, 2.0 ** -24), (np.complex128, 4, 2.0 ** -53)])
def test_random_sums_stay_within_their_roundings(lib, dtype, kr, eps):
    rng = np.random.default_rng(4)
    rows = (rng.standard_normal((40, 4, kr, 32)) + 1j * rng.standard_normal((40, 4, kr, 32))).astype(dtype)
    a = np.abs(rows.astype(np.complex128)).reshape(40, 4, -1)
    size = np.einsum("bvn,bxn->bvx", a[:, :2], a[:, 2:])[..., None]
    # float32: two rows, four roundings (1 % for those of the pairs' remainders); float64: four rows and five
    # levels, and the reference's own sum of 128 rows
    n = 4 * 1.01 if dtype == np.complex64 else 8 + 5 + 128
    assert (np.abs(_sums(lib, rows) - _want(rows)) <= n * eps * size).all()


def test_infinity_and_nan_come_through(lib):
    rows = np.ones((2, 4, 8, 32), dtype=np.complex64)
    rows[0, 0, 3, 17] = np.inf
    rows[1, 2, 5, 30] = np.nan
    got = _sums(lib, rows)
    assert not np.isfinite(got[0, 0]).any() and (got[0, 1, :, 0] == 256).all()
    assert not np.isfinite(got[1, :, 0]).any() and (got[1, :, 1, 0] == 256).all()
