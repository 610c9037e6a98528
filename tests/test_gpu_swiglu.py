"""silu(g) * u as the SwiGLU epilogues compute it, against the IEEE division it stands for: every one of the 2^32 gates."""
import ctypes
import subprocess

import pytest
import torch

from paper_2602_11133_b200 import build as jot_build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "ptx.cuh"
// counts: gates where one side is a NaN and the other is not; gates whose bits differ; the largest distance in ulps
__global__ void compare(unsigned long long* counts) {
    unsigned long long nan = 0, differ = 0, worst = 0;
    for (unsigned long long i = blockIdx.x * 1024ull + threadIdx.x; i < 1ull << 32; i += gridDim.x * 1024ull) {
        const float g = __uint_as_float((unsigned)i);
        const float got = jot::silu_mul(g, 1.f), want = __fdiv_rn(g, 1.f + __expf(-g));
        if (isnan(got) || isnan(want)) { nan += isnan(got) != isnan(want); continue; }
        const int a = __float_as_int(got), b = __float_as_int(want);           // as points of one ordered scale
        const long long x = a < 0 ? -(long long)(a & 0x7fffffff) : a, y = b < 0 ? -(long long)(b & 0x7fffffff) : b;
        const unsigned long long d = x > y ? x - y : y - x;
        differ += a != b;
        worst = d > worst ? d : worst;
    }
    atomicAdd(counts, nan); atomicAdd(counts + 1, differ); atomicMax(counts + 2, worst);
}
__global__ void products(const float* g, const float* u, float* out, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) out[i] = jot::silu_mul(g[i], u[i]);
}
extern "C" int run_compare(unsigned long long* counts) { compare<<<1184, 1024>>>(counts); return (int)cudaGetLastError(); }
extern "C" int run_products(const float* g, const float* u, float* out, int n) {
    products<<<1, 256>>>(g, u, out, n);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    at = tmp_path_factory.mktemp("swiglu")
    (at / "swiglu.cu").write_text(SOURCE)
    subprocess.run([jot_build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
                    "-shared", "-I", jot_build.CSRC, "-o", str(at / "swiglu.so"), str(at / "swiglu.cu")], check=True)
    made = ctypes.CDLL(str(at / "swiglu.so"))
    made.run_compare.argtypes = [ctypes.c_void_p]
    made.run_products.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    return made


def test_every_gate_against_the_division(lib):
    counts = torch.zeros(3, dtype=torch.int64, device="cuda")
    assert lib.run_compare(counts.data_ptr()) == 0
    torch.cuda.synchronize()
    nan, differ, worst = counts.tolist()
    print(f"{differ} of 2^32 gates with other bits than the division, at most {worst} ulp")
    assert nan == 0
    assert worst <= 1 and differ <= 8                                          # 3 measured


def test_products_against_64_bits(lib):
    """`u` lifts the smallest quotients into view.  Bound: __expf's documented error, 2 + floor(1.173 |g|) ulp, and four roundings."""
    g = torch.cat([torch.linspace(-88.6, 88.6, 4001), torch.tensor([-87.4, -88.0, -88.5, -20.0, 20.0, 1e-30, -1e-30, 3e38])])
    u = torch.full_like(g, 1e30).where(g < 0, torch.tensor(1.5))
    d_g, d_u, out = g.cuda(), u.cuda(), torch.empty(len(g), device="cuda")
    assert lib.run_products(d_g.data_ptr(), d_u.data_ptr(), out.data_ptr(), len(g)) == 0
    torch.cuda.synchronize()
    want = g.double() / (1 + torch.exp(-g.double())) * u.double()
    fits = want.abs() < 3.4e38
    err = ((out.cpu().double() - want).abs() / want.abs())[fits & (want != 0)]
    bound = ((2 + torch.floor(1.173 * g.abs()) + 4) * 2.0 ** -23).double()[fits & (want != 0)]
    assert (err <= bound).all(), (err / bound).max()
    assert torch.isinf(out.cpu()[~fits]).all()
