"""Eq 27 on one cut link as the level step evaluates it, against 64 bits.

Reference for the size of its error: the same equation with the weights 1 / (1 + q) and q / (1 + q)
rounded from 64 bits to FP32 and every operation rounded to FP32.  The step's form may be no further
off in the mean square.  The bound on a single value counts its roundings (u = 2^-24), with S the sum
of the terms' magnitudes: one of the weight, four of sums up to 2 S times a weight up to 1/2, the
product's and two of sums up to 2 S: at most 10 u S."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2601_18443_gb300 import _build_ext as ext

pytestmark = pytest.mark.gpu

PROBE = """
#include "level.cuh"
__global__ void k(const float *v, float *out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = lbmdev::yu_link(v[i], v[n + i], v[2 * n + i], v[3 * n + i], v[4 * n + i]);
}
extern "C" int links(const float *in, float *out, int n)
{
    float *d = nullptr;
    if (cudaMalloc(&d, 6 * (size_t)n * sizeof(float)) != cudaSuccess) return 1;
    cudaMemcpy(d, in, 5 * (size_t)n * sizeof(float), cudaMemcpyHostToDevice);
    k<<<(n + 255) / 256, 256>>>(d, d + 5 * (size_t)n, n);
    const cudaError_t e = cudaMemcpy(out, d + 5 * (size_t)n, n * sizeof(float), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
"""


@pytest.fixture(scope="module")
def links(tmp_path_factory):
    d = tmp_path_factory.mktemp("links")
    src, so = os.path.join(d, "links.cu"), os.path.join(d, "links.so")
    with open(src, "w") as f:
        f.write(PROBE)
    subprocess.run([ext._nvcc(), "-shared", "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I", ext.CSRC, *ext.ARCH, "-o", so,
                    src], check=True, capture_output=True)
    return C.CDLL(so).links


# size of the populations' departures, share of it that differs between neighbours
@pytest.mark.parametrize("amp,spread", [(1e-3, 0.05), (1e-2, 0.05), (0.05, 1.0)])
def test_a_cut_link_is_as_precise_as_with_tabulated_weights(links, amp, spread):
    n = 1 << 20
    rng = np.random.default_rng(27)
    base = amp * rng.uniform(-1, 1, n)
    Q = rng.uniform(0, 1, n)
    Q[:2] = 0.0, 1.0
    q, wa, wb = (a.astype(np.float32) for a in (Q, 1 / (1 + Q), Q / (1 + Q)))
    gin, fo, f = ((base + spread * amp * rng.uniform(-0.5, 0.5, n)).astype(np.float32) for _ in range(3))
    mom = (0.3 * amp * rng.uniform(-0.5, 0.5, n)).astype(np.float32)
    v = np.ascontiguousarray(np.stack([wb, gin, fo, f, mom]))
    out = np.empty(n, dtype=np.float32)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    assert links(ptr(v), ptr(out), n) == 0
    G, Fo, F, M = (a.astype(np.float64) for a in v[1:])
    want = ((1 - Q) * G + Q * Fo + M + Q * F) / (1 + Q)
    table = ((np.float32(1) - q) * gin + q * fo + mom) * wa + wb * f
    rms = lambda x: np.sqrt(np.mean((x.astype(np.float64) - want) ** 2))
    assert rms(out) <= rms(table), (rms(out), rms(table))
    assert (np.abs(out - want) <= 10 * 2.0**-24 * (np.abs(G) + np.abs(Fo) + np.abs(F) + np.abs(M))).all()
