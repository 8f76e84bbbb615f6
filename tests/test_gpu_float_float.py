"""The accumulators' float-float distances against float64, each as its kernel compiles it."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = """
#include "st_accum_dev.cuh"
__global__ void k_dist(const float* a, const float* b, int n, float* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float *p = a + 3 * i, *q = b + 3 * i;
    const st::acc::ff d = st::acc::dist_ff(p[0], p[1], p[2], q[0], q[1], q[2]);
    float inv;
    const st::acc::ff e = st::acc::dist_inv_ff(p[0], p[1], p[2], q[0], q[1], q[2], &inv);
    out[5 * i] = d.hi;
    out[5 * i + 1] = d.lo;
    out[5 * i + 2] = e.hi;
    out[5 * i + 3] = e.lo;
    out[5 * i + 4] = inv;
}
extern "C" int run(const float* a, const float* b, int n, float* out) {
    k_dist<<<(n + 127) / 128, 128>>>(a, b, n, out);
    return (int)cudaDeviceSynchronize();
}
"""


def test_distances_are_as_accurate_as_each_other(tmp_path):
    """dist_inv_ff (few bins) against dist_ff: both hold the square root's argument to about 2^-46 and correct a root
    that is within an ulp, so each is within 2^-45 of float64 and their mean errors are alike (25 % left for the rounding
    of the root each starts from)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_19652_gb300 import build
    src, lib = os.path.join(tmp_path, "d.cu"), os.path.join(tmp_path, "d.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, *build.COMMON, "-Xcompiler", "-fvisibility=default", "-shared", "-cudart",
                    "shared", src, "-o", lib, "-Xlinker", "-rpath", "-Xlinker", "/usr/local/cuda/lib64"], check=True)
    rng = np.random.default_rng(0)
    n = 1 << 20
    a = (10 * rng.normal(size=(n, 3))).astype(np.float32)
    b = (a + rng.normal(size=(n, 3)) * np.exp(rng.uniform(np.log(0.05), np.log(60), (n, 1)))).astype(np.float32)
    A, B = (torch.as_tensor(x, device="cuda") for x in (a, b))
    out = torch.empty((n, 5), device="cuda")
    L = ctypes.CDLL(lib)
    L.run.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    assert L.run(A.data_ptr(), B.data_ptr(), n, out.data_ptr()) == 0
    o = out.cpu().numpy().astype(np.float64)
    r = np.sqrt(((a.astype(np.float64) - b) ** 2).sum(1))
    e0, e1 = (np.abs((o[:, c] - r) + o[:, c + 1]) / r for c in (0, 2))
    rms = [float(np.sqrt((e ** 2).mean())) for e in (e0, e1)]
    print("max 2^%.2f 2^%.2f, rms 2^%.2f 2^%.2f" % tuple(np.log2([e0.max(), e1.max(), *rms])))
    assert e0.max() <= 2.0 ** -45 and e1.max() <= 2.0 ** -45
    assert rms[1] <= 1.25 * rms[0]
    assert np.abs(o[:, 4] * r - 1).max() <= 2.0 ** -21
