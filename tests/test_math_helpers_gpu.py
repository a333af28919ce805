"""The Box-Muller helpers of the step over all their arguments (the 2^23 uniforms, in
[2^-24, 1)): log_unit gives logf's bits, sqrt_normal is within one ulp of CUDA's correctly
rounded sqrtf, hence 1.5 ulp of FP64."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SOURCE = r"""
#include <cstdio>
#include "lpm_device.cuh"
using namespace lpm;

// out: 0 uniforms outside [2^-24, 1), 1 largest ulps of sqrt_normal from sqrtf, 2 its largest
// error against FP64 in 1/1000 ulp, 3 uniforms whose log_unit is not logf
__device__ unsigned long long milli_ulp(float got, double want)
{
    const float a = fabsf((float)want);
    const double ulp = (double)__uint_as_float(__float_as_uint(a) + 1u) - (double)a;
    return (unsigned long long)(fabs((double)got - want) / ulp * 1000.0);
}

__global__ void probe_kernel(unsigned long long *out)
{
    const unsigned int i = blockIdx.x * blockDim.x + threadIdx.x;    // 2^23 in all
    const float u = unit_uniform(i << 9);
    if (!(u >= 5.9604645e-08f && u < 1.0f)) atomicAdd(out, 1ull);
    const float l = logf(u), x = -2.0f * l;
    if (__float_as_uint(log_unit(u)) != __float_as_uint(l)) atomicAdd(out + 3, 1ull);
    const float s = sqrt_normal(x), r = sqrtf(x);
    atomicMax(out + 1, (unsigned long long)abs(__float_as_int(s) - __float_as_int(r)));
    atomicMax(out + 2, milli_ulp(s, sqrt((double)x)));
}

extern "C" int probe(unsigned long long *host)
{
    unsigned long long *d;
    if (cudaMalloc(&d, 4 * sizeof *d) != cudaSuccess) return 1;
    cudaMemset(d, 0, 4 * sizeof *d);
    probe_kernel<<<(1 << 23) / 256, 256>>>(d);
    const cudaError_t e = cudaMemcpy(host, d, 4 * sizeof *d, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e != cudaSuccess;
}
"""


def test_log_and_root_of_every_uniform(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0912_3223_gb300 import build
    src, lib = tmp_path / "probe.cu", tmp_path / "probe.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", os.path.join(build.HERE, "csrc"),
                    "-shared", "-o", str(lib), str(src)], check=True, capture_output=True)
    out = (ctypes.c_ulonglong * 4)()
    assert ctypes.CDLL(str(lib)).probe(out) == 0
    print(f"root: {out[2] / 1000} ulp of FP64")
    assert out[0] == 0 and out[3] == 0
    assert out[1] <= 1 and out[2] <= 1500
