"""GPU test of the training kernels' SiLU (csrc/silu.cuh) on every FP32 number:
where the branch-free form answers for itself (2^-100 <= |x| <= 87), the
activation, and the reciprocal inside the derivative, are those of the
correctly rounded divisions, bit for bit; everywhere else (zeros, subnormals,
large numbers, infinities, NaN) it hands over.  And infinite pre-activations
in a training step: the loss is the infinity that the divisions give."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SOURCE = r"""
#include "silu.cuh"
#include <cuda_runtime.h>
__global__ void compare(unsigned long long* out)
{
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    unsigned long long differ = 0, range = 0, ones = 0;
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < 1ull << 32; i += stride) {
        const float x = __uint_as_float((uint32_t)i);
        float a, d;
        bool ok = true;
        sde_train::silu_fast(x, a, d, ok);
        range += ok != (fabsf(x) >= 0x1p-100f && fabsf(x) <= 87.0f);
        if (!ok) continue;
        const float q = 1.0f + __expf(-x), s = __fdiv_rn(1.0f, q);
        differ += __float_as_uint(a) != __float_as_uint(__fdiv_rn(x, q));
        differ += __float_as_uint(d) != __float_as_uint(__fmul_rn(s, fmaf(x, 1.0f - s, 1.0f)));
        ones += (__float_as_uint(q) & 0x7fffffu) == 0x7fffffu;
    }
    atomicAdd(out, differ); atomicAdd(out + 1, range); atomicAdd(out + 2, ones);
}
extern "C" int run(unsigned long long* host)
{
    unsigned long long* d = nullptr;
    cudaError_t e = cudaMalloc(&d, 24);
    if (e == cudaSuccess) e = cudaMemset(d, 0, 24);
    if (e == cudaSuccess) { compare<<<1216, 256>>>(d); e = cudaGetLastError(); }
    if (e == cudaSuccess) e = cudaMemcpy(host, d, 24, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
"""


@pytest.fixture(autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_every_number_against_the_divisions(tmp_path):
    from paper_1409_4923_gb300 import build
    src, so = tmp_path / "silu_all.cu", tmp_path / "silu_all.so"
    src.write_text(SOURCE)
    subprocess.check_call([build.nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                                                         "-I", build.CSRC, str(src), "-o", str(so)])
    out = (ctypes.c_ulonglong * 3)()
    assert ctypes.CDLL(os.fspath(so)).run(out) == 0
    assert out[0] == 0 and out[1] == 0
    assert out[2] > 0                       # a divisor of all-ones mantissa is among them


@pytest.mark.parametrize("M", [5, 2433])
def test_infinite_activations_give_an_infinite_loss(M):
    """Weights above zero throughout, first biases infinite: every activation and
    output is +inf, and so is the loss (never NaN)."""
    from paper_1409_4923_gb300 import surrogate as S
    net = S.Surrogate(3)
    try:
        P = omlp.unflatten(net.get_params().astype(np.float64))
        for name in P:
            P[name] = np.abs(P[name]) + (0.01 if name in ("W2", "W3") else 0.0)
        P["W4"][:2] = 0.02
        P["b1"][:] = np.inf
        net.set_params(omlp.flatten(P).astype(np.float32))
        _, loss = net.gradients(torch.full((M, 7), 0.5, device="cuda"), torch.zeros((M, 2), device="cuda"))
        assert loss == np.inf
    finally:
        net.close()
