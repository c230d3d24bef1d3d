"""chi's bits do not depend on what the compiler contracts: every kernel shape forms chi of a
particle with chi_of or, two leptons at a time, with step_pair, and a particle's bits must not
depend on which.  The routine is compiled with contraction on and off."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2301_07684_gb300 import build as B

pytestmark = pytest.mark.gpu

PROBE = """#include "sfq_step.cuh"
template <typename T> __global__ void chi_kernel(int n, const T *in, T *general, T *wave) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const T *v = in + 11 * i;
        const T E[3] = {v[4], v[5], v[6]}, Bf[3] = {v[7], v[8], v[9]};
        general[i] = sfq::chi_of<T>(v[0], v[1], v[2], v[3], E, Bf, v[10]);
        wave[i] = sfq::chi_pw<T>(v[0], v[1], v[2], v[5], v[10]);
    }
}
template <typename T> static int run(int n, const void *in, void *general, void *wave) {
    chi_kernel<T><<<64, 128>>>(n, static_cast<const T *>(in), static_cast<T *>(general), static_cast<T *>(wave));
    return (int)cudaDeviceSynchronize();
}
extern "C" int chi_f32(int n, const void *in, void *g, void *w) { return run<float>(n, in, g, w); }
extern "C" int chi_f64(int n, const void *in, void *g, void *w) { return run<double>(n, in, g, w); }
"""


@pytest.fixture(scope="module")
def probes(tmp_path_factory):
    d = tmp_path_factory.mktemp("chi")
    (d / "p.cu").write_text(PROBE)
    libs = []
    for contract in ("true", "false"):
        so = os.path.join(d, f"p_{contract}.so")
        subprocess.run([B.NVCC, *B.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", f"-fmad={contract}", "-shared",
                        "-Xcompiler", "-fPIC", "-cudart", "shared", "-I", B.INCLUDE, "-I", B.CSRC, "-o", so,
                        os.path.join(d, "p.cu")], check=True, capture_output=True)
        libs.append(ctypes.CDLL(so))
    return libs


@pytest.mark.parametrize("name,dtype", [("chi_f32", torch.float32), ("chi_f64", torch.float64)])
def test_chi_is_the_same_with_and_without_contraction(probes, name, dtype):
    g = np.random.default_rng(2)
    n = 200000
    p = np.stack([-10.0 ** g.uniform(0, 4, n), g.normal(0, 10, n), g.normal(0, 10, n)], 1)
    fields = g.normal(0, 100, (n, 6))
    fields[: n // 4, [0, 2, 3, 4]] = 0.0                    # a wave's fields
    gam = np.sqrt(1 + (p * p).sum(1))
    rows = np.concatenate([gam[:, None], p, fields, np.full((n, 1), 1 / 4.1e5)], 1)
    x = torch.as_tensor(rows).to("cuda", dtype).contiguous()
    out = [[torch.empty(n, dtype=dtype, device="cuda") for _ in range(2)] for _ in probes]
    vp = ctypes.c_void_p
    torch.cuda.synchronize()
    for lib, (a, b) in zip(probes, out):
        assert getattr(lib, name)(n, vp(x.data_ptr()), vp(a.data_ptr()), vp(b.data_ptr())) == 0
    bits = torch.int32 if dtype == torch.float32 else torch.int64
    for k in range(2):
        assert float(out[0][k].max()) > 0.0
        assert torch.equal(out[0][k].view(bits), out[1][k].view(bits)), ("general", "wave")[k]
