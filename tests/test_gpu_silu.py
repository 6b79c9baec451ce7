"""The SwiGLU arithmetic of the projection epilogues (csrc/silu.cuh), element by element against the division operator and fp64."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_17404_b200", "csrc")
SOURCE = r"""
#include "silu.cuh"
__global__ void silu_kernel(const float* g, const float* u, float* mine, float* op, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) { mine[i] = trj::silu_times(g[i], u[i]); op[i] = g[i] / (1.f + expf(-g[i])) * u[i]; }
}
__global__ void quotient_kernel(const float* a, const float* d, float* mine, float* op, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) { mine[i] = trj::quotient_by_1_to_2(a[i], d[i]); op[i] = a[i] / d[i]; }
}
extern "C" int run(int what, const float* a, const float* b, float* mine, float* op, int n) {
    if (what == 0) silu_kernel<<<(n + 255) / 256, 256>>>(a, b, mine, op, n);
    else quotient_kernel<<<(n + 255) / 256, 256>>>(a, b, mine, op, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("silu")
    (d / "s.cu").write_text(SOURCE)
    subprocess.run(["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC, str(d / "s.cu"),
                    "-o", str(d / "s.so")], check=True)
    fn = ctypes.CDLL(str(d / "s.so")).run

    def call(what, a, b):
        a, b = torch.from_numpy(a.astype(np.float32)).cuda(), torch.from_numpy(b.astype(np.float32)).cuda()
        mine, op = torch.empty_like(a), torch.empty_like(a)
        torch.cuda.synchronize()
        assert fn(what, *(ctypes.c_void_p(t.data_ptr()) for t in (a, b, mine, op)), a.numel()) == 0
        return mine.cpu().numpy(), op.cpu().numpy()
    return call


def test_quotient_equals_the_operator(run):
    """Random and edge denominators of [1, 2]; numerators of every exponent whose remainder is still a normal number."""
    r = np.random.Generator(np.random.Philox(1))
    n = 1 << 22
    d = np.concatenate([r.uniform(1, 2, n - 4), [1, 2, np.nextafter(np.float32(1), np.float32(2)), np.nextafter(np.float32(2), np.float32(1))]])
    a = np.ldexp(r.uniform(1, 2, n), r.integers(-100, 127, n)) * r.choice([-1.0, 1.0], n)
    mine, op = run(1, a, d)
    np.testing.assert_array_equal(mine, op)
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 3.4028235e38, -3.4028235e38, 1e-40, -1e-45])
    mine, op = run(1, special, np.full(special.size, 1.0))
    np.testing.assert_array_equal(mine, op)


def test_silu_against_fp64(run):
    """|g| up to 104, where silu(g) leaves the denormal numbers.  In units in the last place of the result: exp 2 (its stated
    bound), in numerator and (halved or less) denominator, plus half for the product, the sum and the quotient: 4.5.  Below -87
    exp is denormal itself: an absolute error of up to 2^-149, times |g|."""
    g = np.concatenate([np.linspace(-104, 104, 1 << 21), np.ldexp(np.linspace(1, 2, 1 << 16), -30), -np.ldexp(np.linspace(1, 2, 1 << 16), -30)]).astype(np.float32)
    mine, op = run(0, g, np.ones(g.size))
    x = g.astype(np.float64)
    e = np.exp(-np.abs(x))
    ref = np.where(x < 0, x * e, x) / (1 + e)
    ulp = np.maximum(np.ldexp(1.0, np.frexp(ref)[1] - 24), 2.0 ** -149)
    assert (np.abs(mine - ref) <= 4.5 * ulp + np.where(x < -87, -x * 2.0 ** -149, 0)).all()
    # where the operator's form neither overflows nor loses bits the two are equally good
    plain = x > -85
    assert np.abs((mine - ref) / ulp)[plain].max() <= np.abs((op - ref) / ulp)[plain].max() + 0.5


def test_silu_of_large_and_special_gates(run):
    g = np.array([np.inf, 3e38, 1e6, 0.0, -0.0, -88.0, -1e3, -1e6, -1e30, -3e38, np.nan, -np.inf, np.inf, np.inf])
    u = np.array([2.0, 1.0, -3.0, 5.0, 5.0, 1e30, 1e30, 1e30, 1e30, 1e30, 1.0, 1.0, -1.0, 0.0])
    mine, op = run(0, g, u)
    same = np.ones(g.size, bool)
    same[5] = False                                          # -88 * exp(-88): the operator's form has lost bits there
    np.testing.assert_array_equal(mine[same], op[same])
    assert mine[0] == np.inf and np.abs(mine[6:10]).max() == 0.0
    assert abs(mine[5] / (-88.0 * np.exp(-88.0) * 1e30) - 1) < 1e-6
