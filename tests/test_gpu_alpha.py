"""The packed form of alpha (two pixels per instruction) takes the scalar rule's
value, bit for bit: both from csrc/spec.cuh, in a kernel compiled here."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2410_14462_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "spec.cuh"
using namespace ludvig;
// g: [n][6] mx, my, conic a, b, c, opacity; px: [n][2] first pixel centre's x, y
__global__ void k_compare(const float* g, const float* px, long n, float2 one2, unsigned* bad, unsigned* hits) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float *p = g + 6 * i, x = px[2 * i], y = px[2 * i + 1];
    const F2 dx = f2_add(f2(p[0], p[0]), f2(-x, -(x + 1.f))), dy = f2_add(f2(p[1], p[1]), f2(-y, -y));
    const F2 ax = f2_mul(f2(p[2], p[2]), f2_mul(dx, dx)), cy = f2_mul(f2(p[4], p[4]), f2_mul(dy, dy));
    const float2 got = alpha_at_x2(dx, ax, dy, cy, f2(p[3], p[3]), f2(p[5], p[5]), f2(one2.x, one2.y));
    for (int k = 0; k < 2; ++k) {
        float want = alpha_at(p[0], p[1], p[2], p[3], p[4], p[5], x + (float)k, y);
        if (!(want > 0.f)) want = 0.f;   // as the walks take it: a NaN is skipped
        const float have = k ? got.y : got.x;
        if (__float_as_uint(have) != __float_as_uint(want)) atomicAdd(bad, 1u);
        if (want > 0.f) atomicAdd(hits, 1u);
    }
}
extern "C" int compare(const float* g, const float* px, long n, unsigned* out) {
    k_compare<<<(unsigned)((n + 255) / 256), 256>>>(g, px, n, make_float2(1.f, 1.f), out, out + 1);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def compare(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    d = tmp_path_factory.mktemp("alpha")
    src, lib = d / "alpha.cu", d / "libalpha.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-shared", str(src), "-o", str(lib)], check=True)
    f = ctypes.CDLL(str(lib)).compare
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long, ctypes.c_void_p]

    def run(g, px):
        g, px = torch.from_numpy(g).cuda(), torch.from_numpy(px).cuda()
        out = torch.zeros(2, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert f(g.data_ptr(), px.data_ptr(), g.shape[0], out.data_ptr()) == 0
        return out.tolist()
    return run


def _random(n, seed):
    rng = np.random.default_rng(seed)
    a, c = np.exp(rng.uniform(-8, 1.2, (2, n)))        # conics of 0.3 to 3000 square pixels
    rho = np.clip(rng.normal(0, 0.5, n), -0.999, 0.999)
    px = np.floor(rng.uniform(0, 2000, (n, 2))) + 0.5
    mean = px + rng.normal(size=(n, 2)) / np.sqrt(np.stack([a, c], 1)) * rng.uniform(0, 4, (n, 1))
    g = np.stack([mean[:, 0], mean[:, 1], a, rho * np.sqrt(a * c), c, rng.uniform(0, 1, n)], 1)
    return g.astype(np.float32), px.astype(np.float32)


def test_packed_alpha_is_the_scalar_alpha(compare):
    hits = 0
    for seed in range(4):
        bad, h = compare(*_random(2_000_000, seed))
        assert bad == 0
        hits += h
    assert hits > 4_000_000


@pytest.mark.parametrize("column", range(6))
def test_packed_alpha_of_odd_values(compare, column):
    """A NaN or an infinity in any parameter, opacities outside (0, 1), and zeros."""
    g, px = _random(100_000, 10 + column)
    odd = np.array([np.nan, np.inf, -np.inf, 0.0, -0.5, 1.0, 2.0, 1 / 255, 0.99, 1e-30, 1e30, 1e38], np.float32)
    g[:, column] = odd[np.arange(len(g)) % odd.size]
    assert compare(g, px)[0] == 0
