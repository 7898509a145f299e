"""The block scan that the binning and the densification share, at every number of warps it may be called
with: a small kernel around the library's header, compiled here."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2507_20239_gb300 import build as gbuild

pytestmark = pytest.mark.gpu

SOURCE = """
#include "scan.cuh"
namespace gs { void count_launch() {} }
__global__ void scan(const uint32_t *x, uint32_t *out, uint32_t *total) {
  uint32_t all;
  out[threadIdx.x] = gs::block_exclusive_scan<uint32_t>(x[threadIdx.x], &all);
  if (threadIdx.x == 0) *total = all;
}
extern "C" int run(const uint32_t *x, uint32_t *out, uint32_t *total, int threads) {
  scan<<<1, threads>>>(x, out, total);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("scan")
    src, so = os.path.join(d, "scan.cu"), os.path.join(d, "scan.so")
    open(src, "w").write(SOURCE)
    subprocess.run([gbuild.nvcc(), *gbuild.FLAGS, *gbuild.ARCH, "-shared", "-I", gbuild.INCLUDE, "-I", gbuild.CSRC, src,
                    "-o", so], check=True, capture_output=True)
    return C.CDLL(so)


@pytest.mark.parametrize("threads", [32, 64, 256, 512, 992, 1024])
def test_block_exclusive_scan(probe, threads):
    x = np.random.default_rng(threads).integers(0, 1000, threads).astype(np.int32)
    dx, out, total = torch.as_tensor(x).cuda(), torch.zeros(threads, dtype=torch.int32, device="cuda"), \
        torch.zeros(1, dtype=torch.int32, device="cuda")
    p = lambda t: C.c_void_p(t.data_ptr())   # noqa: E731
    assert probe.run(p(dx), p(out), p(total), threads) == 0
    assert np.array_equal(out.cpu().numpy(), np.cumsum(x) - x) and int(total) == x.sum()
