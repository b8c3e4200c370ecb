"""The FP32 return scale min(1, Y / sqrt(J2)) of the packed sweeps against the quotient in 64 bits."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = """
#include "ep_lanes.cuh"
static __global__ void k(const float *J2, const float *Y, float *s, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  s[i] = ep::scale_of(J2[i], Y[i]);
  // a pair's scales are those of its members, in either place
  const int j = i ^ 1;
  if (j < n) {
    const float2 a = ep::vscale(make_float2(J2[i], J2[j]), make_float2(Y[i], Y[j]));
    const float2 b = ep::vscale(make_float2(J2[j], J2[i]), make_float2(Y[j], Y[i]));
    if (__float_as_uint(a.x) != __float_as_uint(s[i]) || __float_as_uint(b.y) != __float_as_uint(s[i])) s[i] = -1.f;
  }
}
extern "C" int scale_of(const float *J2, const float *Y, float *s, int n) {
  k<<<(n + 255) / 256, 256>>>(J2, Y, s, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def scale_of(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_01701_gb300 import build as B
    d = tmp_path_factory.mktemp("scale")
    src, lib = str(d / "scale.cu"), str(d / "libscale.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-shared", "-cudart=shared", "-I", os.path.join(B.CSRC), src,
                    "-o", lib], check=True)
    fn = ctypes.CDLL(lib).scale_of
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]

    def call(J2, Y):
        a = [torch.tensor(np.asarray(x, np.float32)).cuda() for x in (J2, Y)]
        s = torch.empty_like(a[0])
        torch.cuda.synchronize()
        assert fn(a[0].data_ptr(), a[1].data_ptr(), s.data_ptr(), s.numel()) == 0
        return s.cpu().numpy()

    return call


def test_quotient_is_rounded_once(scale_of):
    rng = np.random.default_rng(2)
    n = 1 << 20
    J2 = np.exp(rng.uniform(np.log(1e-25), np.log(1e25), n)).astype(np.float32)
    Y = (np.sqrt(J2.astype(np.float64)) * np.where(rng.random(n) < 0.5, rng.random(n), 1.0 - 1e-3 * rng.random(n)))
    Y = Y.astype(np.float32)
    s = scale_of(J2, Y)
    act = J2 > Y * Y          # the comparison of squares in FP32, as the kernel makes it
    assert act.mean() > 0.9
    ref = Y.astype(np.float64) / np.sqrt(J2.astype(np.float64))
    ulp = np.spacing(np.minimum(ref, 1.0 - 2.0 ** -24).astype(np.float32)).astype(np.float64)
    # one rounding of a quotient known to 2^-40
    assert (np.abs(s - ref)[act] / ulp[act]).max() <= 0.5 + 2.0 ** -14
    assert (s[~act] == 1.0).all() and s.max() <= 1.0


def test_special_values(scale_of):
    inf, nan = np.inf, np.nan
    J2 = [inf, inf, nan, 0.0, 0.0, 1.0, 1.0, 4.0, 3e38]
    Y = [1.0, 0.0, 1.0, 0.0, 1.0, -1.0, nan, 1.0, 3e38]
    want = [0.0, 0.0, 1.0, 1.0, 1.0, 0.0, 0.0, 0.5, 1.0]
    np.testing.assert_array_equal(scale_of(J2, Y), np.asarray(want, np.float32))
