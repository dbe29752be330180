"""The tensor-core products when waits inside the kernel run out: built here with a limit of one
try per wait that does not park the thread (csrc/kd_tc.cuh), where almost any wait expires.  A call returns, each output is
NaN or right to the bit, and the device works on as before."""

import ctypes
import os
import subprocess

import pytest
import torch

from tests.test_gpu_fold import kd  # noqa: F401  (the module's fixture)
from tests.test_gpu_fold_tc import _case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def impatient(tmp_path_factory):
    from paper_2609_11687_gb300 import build
    so = str(tmp_path_factory.mktemp("impatient") / "lib.so")
    srcs = [os.path.join(build.CSRC, f) for f in ("kd_fold.cu", "kd_fold_tc.cu", "kd_fold16.cu", "kd_fold16_tc.cu")]
    subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-DKD_WAIT_TRIES=1", '-DKD_MBAR_WAIT="mbarrier.test_wait"',
                    "-shared", "-o", so] + srcs, check=True)
    return ctypes.CDLL(so)


def _call(lib, name, dec, x, xp, y):
    p, i = ctypes.c_void_p, ctypes.c_int64
    fn = getattr(lib, name)
    fn.argtypes = [p, p, p, p, i, i, p, p, i, i, p, i, p]
    return fn(dec.codes_u.data_ptr(), dec.codes_v.data_ptr(), dec.centres_u.data_ptr(), dec.centres_v.data_ptr(),
              x.shape[1], dec.codes_u.shape[0], x.data_ptr(), xp.data_ptr(), x.shape[0], x.stride(0), y.data_ptr(),
              y.stride(0), torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("name,batch", [("kd_matmul_2bit", 16), ("kd_matmul_2bit", 33), ("kd_matmul_2bit_f16", 12),
                                        ("kd_matmul_2bit_f16", 100), ("kd_matmul_2bit_f16", 300)])
def test_expired_waits(kd, impatient, name, batch):  # noqa: F811
    dec, x, xp = _case(kd, 4096, 1030, batch)
    if name.endswith("f16"):
        x, xp = x.half(), xp.half()
    good = (kd.matmul_2bit_f16 if name.endswith("f16") else kd.matmul_2bit)(dec, x, xp)
    y = torch.zeros_like(good)
    for _ in range(3):
        y.zero_()
        assert _call(impatient, name, dec, x, xp, y) == 0
        torch.cuda.synchronize()
        assert (torch.isnan(y) | (y == good)).all()
    again = (kd.matmul_2bit_f16 if name.endswith("f16") else kd.matmul_2bit)(dec, x, xp)
    assert torch.equal(again, good)


PROBE = r"""
#include "kd_tc.cuh"
__global__ void probe(long long* out) {
  __shared__ uint64_t bar;
  __shared__ int fail;
  if (threadIdx.x == 0) {
    fail = 0;
    kd::mbar_init(&bar, 1);
  }
  __syncthreads();
  const long long t0 = clock64();
  const bool ok = kd::tc_wait(&bar, 0, &fail);  // nothing arrives
  const long long t1 = clock64();
  const bool again = kd::tc_wait(&bar, 0, &fail);
  const long long t2 = clock64();
  __syncthreads();
  if (threadIdx.x == 0) {
    out[0] = ok || again;
    out[1] = fail;
    out[2] = t1 - t0;
    out[3] = t2 - t1;
  }
}
extern "C" int run(long long* host) {
  long long* d;
  if (cudaMalloc(&d, 32) != cudaSuccess) return 1;
  probe<<<1, 32>>>(d);
  const int bad = cudaMemcpy(host, d, 32, cudaMemcpyDeviceToHost) != cudaSuccess;
  cudaFree(d);
  return bad;
}
"""


def test_the_limit_is_a_second(kd, tmp_path):  # noqa: F811
    """A wait that nothing ends gives up after 0.2 to 3 s of SM cycles at 2 GHz, with the flag
    set; the next one at once."""
    from paper_2609_11687_gb300 import build
    (tmp_path / "probe.cu").write_text(PROBE)
    so = str(tmp_path / "probe.so")
    subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-shared", "-o", so, str(tmp_path / "probe.cu")], check=True)
    out = (ctypes.c_longlong * 4)()
    assert ctypes.CDLL(so).run(out) == 0
    assert out[0] == 0 and out[1] == 1
    assert 4e8 <= out[2] <= 6e9 and out[3] <= 1e6, list(out)
