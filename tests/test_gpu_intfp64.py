"""The integer-ALU binary64 operations on the GPU, from its own reciprocal and root estimates, against
its FP64 unit: the same bits over random, sparse and extreme significands and all exponents."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from tests.test_intfp64 import CSRC, _operands

pytestmark = pytest.mark.gpu

SRC = """
#include "dg_intfp64.cuh"
__global__ void k(long n, const double *a, const double *b, double *o)
{
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        o[i] = dg::ifp::mul(a[i], b[i]);
        o[n + i] = dg::ifp::div(a[i], b[i]);
        o[2 * n + i] = dg::ifp::root(a[i]);
        o[3 * n + i] = __dmul_rn(a[i], b[i]);
        o[4 * n + i] = __ddiv_rn(a[i], b[i]);
        o[5 * n + i] = __dsqrt_rn(a[i]);
    }
}
extern "C" int run(long n, const double *a, const double *b, double *o, cudaStream_t s)
{
    k<<<1024, 256, 0, s>>>(n, a, b, o);
    return cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1609_00098_gb300 import build as b
    d = tmp_path_factory.mktemp("intfp64_gpu")
    src, so = str(d / "t.cu"), str(d / "t.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([b._nvcc(), *b.ARCH, "-O3", "-std=c++17", "-fmad=false", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC,
                    src, "-o", so], check=True, capture_output=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("ka", ["near", "sparse", "ends", "any", "special"])
@pytest.mark.parametrize("kb", ["near", "sparse", "ends", "any", "special"])
def test_same_bits_on_the_gpu(lib, ka, kb):
    import torch
    a, b = _operands(ka), np.roll(_operands(kb), 7)
    ga, gb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    out = torch.empty(6, len(a), dtype=torch.float64, device="cuda")
    vp = ctypes.c_void_p
    assert lib.run(ctypes.c_long(len(a)), vp(ga.data_ptr()), vp(gb.data_ptr()), vp(out.data_ptr()),
                   vp(torch.cuda.current_stream().cuda_stream)) == 0
    got, ref = out[:3], out[3:]
    same = (got.view(torch.int64) == ref.view(torch.int64)) | (got.isnan() & ref.isnan())
    assert bool(same.all()), same.logical_not().sum(1).tolist()


def test_every_reciprocal_and_root_estimate(lib):
    """Divisors and radicands at both ends of every FP32 value of [1, 4) that the estimates are taken
    of (2^24 of them, in parts), dividends random: each estimate is used."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    vp = ctypes.c_void_p
    n = 1 << 20
    for part in range(16):
        f = torch.arange(part * n, (part + 1) * n, dtype=torch.int64, device="cuda")  # exponent and significand
        for low in (0, (1 << 29) - 1):
            bits = (1023 << 52) + ((f & ((1 << 23) - 1)) << 29) + ((f >> 23) << 52) + low
            x = bits.view(torch.float64)
            r = torch.randint(0, 1 << 52, (n,), dtype=torch.int64, device="cuda", generator=g) + (1023 << 52)
            for a, b in ((r.view(torch.float64), x), (x, r.view(torch.float64))):
                out = torch.empty(6, n, dtype=torch.float64, device="cuda")
                assert lib.run(ctypes.c_long(n), vp(a.data_ptr()), vp(b.data_ptr()), vp(out.data_ptr()),
                               vp(torch.cuda.current_stream().cuda_stream)) == 0
                assert bool((out[:3].view(torch.int64) == out[3:].view(torch.int64)).all())
