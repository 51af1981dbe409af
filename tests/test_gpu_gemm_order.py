"""A product on the caller's stream is done before the next launch there begins, also a launch that may start
early (programmatic stream serialization) and does not wait by itself: it reads the outputs as they are.  The
reader is a small kernel of this test, built with nvcc."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2503_06757_gb300 import build as B
from paper_2503_06757_gb300 import prrtc as P

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

READER = r'''
#include <cuda_runtime.h>
__global__ void read(const float* __restrict__ c, float* __restrict__ out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = c[i];
}
extern "C" int read_after(const float* c, float* out, int n, void* stream) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((n + 255) / 256);
  lc.blockDim = dim3(256);
  lc.stream = (cudaStream_t)stream;
  lc.attrs = at;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, read, c, out, n);
}
'''


@pytest.fixture(scope="module")
def reader(tmp_path_factory):
    B.build()
    d = tmp_path_factory.mktemp("reader")
    src, so = os.path.join(d, "reader.cu"), os.path.join(d, "reader.so")
    with open(src, "w") as f:
        f.write(READER)
    cmd = [B.nvcc()] + B.ARCH + ["-std=c++17", "-shared", "-Xcompiler", "-fPIC", src, "-o", so]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    fn = C.CDLL(so).read_after
    fn.argtypes = [C.c_void_p, C.c_void_p, C.c_int, C.c_void_p]
    return fn


@pytest.mark.parametrize("m,n,k,splits", [(128, 64, 64, 1), (512, 512, 1024, 0), (512, 1024, 4160, 8), (300, 2048, 256, 1),
                                          (512, 512, 1024, 3), (2048, 4096, 512, 0)])
def test_outputs_are_there_for_the_next_launch(reader, m, n, k, splits):
    g = torch.Generator(device="cuda").manual_seed(m + n + k)
    a = torch.randn(m, k, generator=g, device="cuda").to(torch.bfloat16)
    b = torch.randn(n, k, generator=g, device="cuda").to(torch.bfloat16)
    c, out = (torch.zeros(m, n, device="cuda") for _ in range(2))
    stream = torch.cuda.current_stream().cuda_stream
    for turn in range(20):
        c.fill_(-turn)
        out.zero_()
        P.prrtc_gemm_bf16_splitk(a.data_ptr(), b.data_ptr(), m, n, k, 0, False, c.data_ptr(), 0, splits, stream)
        assert reader(c.data_ptr(), out.data_ptr(), m * n, stream) == 0
        torch.cuda.synchronize()
        assert P.prrtc_gemm_error() == 0
        assert torch.equal(out, c), turn
