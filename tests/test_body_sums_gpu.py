"""Body sums of the affine fit and of the nonlinear model's mean (k_aff_sums): each
block's partial sum is the FP64 sum of its threads' sums.

A block adds 256 values. Without the moments they have 24 bits, are below 1 and whole
multiples of 2^-45; with them they have 18 bits (their products with the node
offsets, at most 32, are then exact in FP32), and all terms are below 32 and multiples
of 2^-39. Every partial sum is so a multiple of 2^-45 below 2^8, or of 2^-39 below
2^13, and exact in FP64, in any order: the tolerance is zero. A merge of the threads'
sums in pairs of FP32 (48 bits) misses the last bits."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2105_06055_gb300", "csrc")
SRC = """
#include "pd_affine.cuh"
#define RUN(NAME, D, NV)                                                                                             \\
    extern "C" int NAME(const float *u, const uint8_t *chi, int lg1, int lg2, const int *c, int64_t N, int blocks,    \\
                        double *red)                                                                                 \\
    {                                                                                                                \\
        pd::k_aff_sums<float, D, NV><<<blocks, 256>>>(u, chi, lg1, lg2, c[0], c[1], c[2], N, red);                    \\
        return (int)cudaDeviceSynchronize();                                                                         \\
    }
RUN(mean2, 2, 2)
RUN(fit2, 2, 6)
RUN(mean3, 3, 3)
RUN(fit3, 3, 12)
"""


@pytest.fixture(scope="module")
def sums(tmp_path_factory):
    from paper_2105_06055_gb300 import build
    d = tmp_path_factory.mktemp("sums")
    src, so = d / "sums.cu", d / "sums.so"
    src.write_text(SRC)
    subprocess.check_call([build._nvcc()] + build.ARCH + ["-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared",
                          "-Xcompiler", "-fPIC", "-cudart=shared", "-I", CSRC, "-I", build.INCLUDE, "-o", str(so),
                          str(src)])
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("shape", [(32, 64), (16, 16, 32)])
@pytest.mark.parametrize("fit", [False, True])
def test_block_sums_are_fp64(sums, shape, fit):
    D, N = len(shape), int(np.prod(shape))
    g = np.random.Generator(np.random.PCG64(4))
    # half of the values with a leading bit at 2^-1, half with the lowest bits
    bits, low = (18, -39) if fit else (24, -45)
    big = g.integers(1 << (bits - 1), 1 << bits, (D, N)) * 2.0 ** -bits
    small = g.integers(0, 1 << bits, (D, N)) * 2.0 ** low
    u = np.where(g.random((D, N)) < 0.5, big, small).astype(np.float32)
    u *= np.where(g.random((D, N)) < 0.3, -1, 1).astype(np.float32)
    chi = (g.random(N) < 0.9).astype(np.uint8)
    c = [n // 2 for n in shape[::-1]] + [0] * (3 - D)
    nv = D + D * D if fit else D
    blocks = (N + 255) // 256
    ud, cd = torch.tensor(u, device="cuda"), torch.tensor(chi, device="cuda")
    red = torch.zeros(nv * blocks, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    run = getattr(sums, ("fit" if fit else "mean") + str(D))
    assert run(ctypes.c_void_p(ud.data_ptr()), ctypes.c_void_p(cd.data_ptr()), int(np.log2(shape[-1])),
               int(np.log2(shape[-2])), (ctypes.c_int * 3)(*c), ctypes.c_int64(N), blocks,
               ctypes.c_void_p(red.data_ptr())) == 0
    got = red.cpu().numpy().reshape(blocks, nv)
    idx = np.arange(N)
    e = [idx % shape[-1] - c[0], (idx // shape[-1]) % shape[-2] - c[1]]
    if D == 3:
        e.append(idx // (shape[-1] * shape[-2]) - c[2])
    terms = [chi * u[j] for j in range(D)]
    if fit:
        terms += [chi * (e[k].astype(np.float32) * u[j]) for j in range(D) for k in range(D)]
    for v, t in enumerate(terms):
        ref = np.array([math.fsum(r) for r in t.astype(np.float64).reshape(blocks, -1)])
        assert np.array_equal(got[:, v], ref), v
