"""Sums of FP32 values over a warp and a CTA (ax_common.cuh).

The error of an FP64 tree over the 32 values v of a warp is at most 5 2^-53 sum |v|
(one rounding on each of 5 levels), that over 8 warps 12 2^-53 sum |v|; the kernels'
sums must be no less exact, and finite wherever an FP64 sum is.
"""
import ctypes
import importlib
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

B = importlib.import_module("paper_1002_3094_gb300.build")

pytestmark = pytest.mark.gpu

SOURCE = """
#include "ax_common.cuh"
// out[w] = the sum of warp w's 32 values, out[nw + b] that of block b's 256
__global__ void sums(const float *v, double *out, int nw) {
  __shared__ double red[8];
  const int i = blockIdx.x * 256 + threadIdx.x;
  const double w = ax::warp_sum_of(v[i]);
  if ((threadIdx.x & 31) == 0) out[i >> 5] = w;
  const double b = ax::block_sum_of(v[i], red);
  if (threadIdx.x == 0) out[nw + blockIdx.x] = b;
}
extern "C" int run_sums(const float *v, double *out, int blocks) {
  sums<<<blocks, 256>>>(v, out, blocks * 8);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("sums")
    src, so = d / "sums.cu", d / "sums.so"
    src.write_text(SOURCE)
    subprocess.run([B.nvcc_path()] + B._flags() + ["-I", B.CSRC, "-I", os.path.join(B.CSRC, "..", "..", "include"),
                                                   "-shared", "-cudart", "static", "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


def test_sums_of_fp32_values(lib):
    rng = np.random.default_rng(1)
    blocks = 64
    v = rng.normal(size=(blocks * 8, 32)) * np.exp2(rng.uniform(-30, 30, (blocks * 8, 32)))
    v[:32] = rng.normal(size=(32, 32))
    v[32:64] = np.abs(rng.normal(size=(32, 32))) * 1e-3
    v[64:96] = rng.normal(size=(32, 32)) * 1e-38           # subnormal low parts
    v[96:128] = 3.0e38 * rng.uniform(0.5, 1.0, (32, 32))   # the sums exceed FP32's range
    v[128:160, ::2], v[128:160, 1::2] = 3.2e38, -3.1e38
    v[160:192, 1:] *= 2.0 ** -40
    v = v.astype(np.float32)
    vd = torch.from_numpy(v).cuda()
    out = torch.zeros(blocks * 9, dtype=torch.float64, device="cuda")
    assert lib.run_sums(ctypes.c_void_p(vd.data_ptr()), ctypes.c_void_p(out.data_ptr()), blocks) == 0
    got = out.cpu().numpy()
    # exact sums: whole multiples of 2^-149 as Python integers
    ints = [[int(np.ldexp(float(x), 100)) * 2 ** 49 if abs(x) >= 2.0 ** -70 else int(np.ldexp(float(x), 149)) for x in r]
            for r in v]
    unit = 2 ** 53

    def check(value, terms, c):
        assert np.isfinite(value)
        m, e = np.frexp(value)
        want, scale = sum(terms), sum(abs(t) for t in terms)
        have = int(m * 2.0 ** 53)  # value = have 2^(e - 53)
        sh = int(e) - 53 + 149
        have = have << sh if sh >= 0 else have >> -sh
        assert abs(have - want) * unit <= c * scale + unit

    for w in range(blocks * 8):
        check(got[w], ints[w], 5)
    for b in range(blocks):
        check(got[blocks * 8 + b], sum(ints[8 * b:8 * b + 8], []), 12)
