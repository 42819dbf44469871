"""The arithmetic primitives of the kernels against correctly rounded results."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2202_01631_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lbdp_kernels.cuh"
#include "lbdp_vec.cuh"
using namespace lbdp;

template <class R>
static __global__ void k_over(const R* a, const R* d, R* q, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        q[i] = inv_norm(a[i]).times(d[i]);
}
// every value of binade ex, both signs: how many differ from the rounded quotient
static __global__ void k_recip(int ex, unsigned long long* bad)
{
    for (unsigned m = blockIdx.x * blockDim.x + threadIdx.x; m < (1u << 23); m += gridDim.x * blockDim.x) {
        const float a = __uint_as_float((unsigned)(ex + 127) << 23 | m);
        const Vec<float, 2> r = recip(Vec<float, 2>{make_float2(a, -a)});
        if (__float_as_uint(r.v.x) != __float_as_uint(__frcp_rn(a)) ||
            __float_as_uint(r.v.y) != __float_as_uint(__frcp_rn(-a)))
            atomicAdd(bad, 1ull);
    }
}
extern "C" int recip32(int ex, unsigned long long* bad)
{
    k_recip<<<1024, 256>>>(ex, bad);
    return (int)cudaDeviceSynchronize();
}
extern "C" int over32(const float* a, const float* d, float* q, int n)
{
    k_over<float><<<1024, 256>>>(a, d, q, n);
    return (int)cudaDeviceSynchronize();
}
extern "C" int over64(const double* a, const double* d, double* q, int n)
{
    k_over<double><<<1024, 256>>>(a, d, q, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    where = tmp_path_factory.mktemp("arithmetic")
    src, so = str(where / "arithmetic.cu"), str(where / "arithmetic.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", src, "-o", so], check=True)
    torch.cuda.init()
    torch.zeros(1, device="cuda")
    return C.CDLL(so)


# |e| <= 2^-20.8 (CUDA's bound of 2 ulp for rsqrtf, and a rounded to FP32 in the
# FP64 form): what the series leaves out, 3/8 e^2 in FP32 and 5/16 e^3 in FP64,
# is below 2^-17 and 2^-10 ulp
@pytest.mark.parametrize("bits,slack", [(32, 2.0 ** -17), (64, 2.0 ** -10)])
def test_quotient_by_a_norm(lib, bits, slack):
    dtype = np.float32 if bits == 32 else np.float64
    wide = np.float64 if bits == 32 else np.longdouble   # 80 or 128 bits
    rng = np.random.default_rng(bits)
    n = 4_000_000 if bits == 32 else 1_000_000
    # squared distances of link points: from a sphere of half a node to one of
    # several hundred; the last half with |d| as large as the norm
    a = (0.25 * 10.0 ** rng.uniform(0.0, 6.0, n)).astype(dtype)
    d = (np.sqrt(a.astype(np.float64)) * rng.uniform(-1.0, 1.0, n)).astype(dtype)
    d[n // 2:] = np.copysign(np.sqrt(a[n // 2:]), d[n // 2:])
    d[:4] = (0.0, -0.0, 0.5, -0.5)
    ga, gd = torch.from_numpy(a).cuda(), torch.from_numpy(d).cuda()
    q = torch.empty_like(ga)
    torch.cuda.synchronize()
    fn = lib.over32 if bits == 32 else lib.over64
    fn.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_int]
    assert fn(ga.data_ptr(), gd.data_ptr(), q.data_ptr(), n) == 0
    got = q.cpu().numpy()
    assert np.array_equal(got[:2], d[:2])
    x = d.astype(wide) / np.sqrt(a.astype(wide))
    # ulp of the binade x lies in (np.spacing of x rounded towards zero)
    r = np.abs(x).astype(dtype)
    r = np.where(r.astype(wide) > np.abs(x), np.nextafter(r, dtype(0)), r)
    err = np.abs(got.astype(wide) - x) / np.spacing(r).astype(wide)
    assert float(err[4:].max()) <= 0.5 + slack


def test_reciprocal_of_a_density_is_the_rounded_quotient(lib):
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    lib.recip32.argtypes = [C.c_int, C.c_void_p]
    for ex in range(-126, 126):
        assert lib.recip32(ex, bad.data_ptr()) == 0
        assert int(bad.item()) == 0, ex
