"""Packing while another stream's kernel holds every SM but one for longer than the
packer's limit on waits: the call is delayed, not given up."""
import ctypes
import subprocess
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HOLD = r"""
#include <cuda_runtime.h>
__global__ void hold(unsigned long long ns)
{
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
    do {
        __nanosleep(100000);
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    } while (t - t0 < ns);
}
// one CTA on each of `ctas` SMs, with the SM's shared memory, for `ns` ns
extern "C" int hold_sms(int ctas, unsigned long long ns, void *stream)
{
    const int smem = 200 * 1024;
    if (cudaFuncSetAttribute(hold, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return 1;
    hold<<<ctas, 32, smem, (cudaStream_t)stream>>>(ns);
    return cudaGetLastError() != cudaSuccess;
}
"""


def test_delayed_by_a_long_kernel(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import oracle
    import paper_1611_04959_gb300 as daq
    from paper_1611_04959_gb300 import build
    (tmp_path / "hold.cu").write_text(HOLD)
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-o", str(tmp_path / "hold.so"),
                    str(tmp_path / "hold.cu")], check=True)
    lib = ctypes.CDLL(str(tmp_path / "hold.so"))
    lib.hold_sms.argtypes = [ctypes.c_int, ctypes.c_uint64, ctypes.c_void_p]
    X, rows = 64, 100_000                     # 64 crystals: one CTA an SM
    pool = (1800 + np.random.default_rng(2).integers(-9, 10, size=(rows, X))).astype(np.int16)
    want = torch.from_numpy(oracle.pack(pool)).cuda()
    dev = torch.from_numpy(pool).cuda()
    got, n = daq.pack_pool(dev)
    assert n == want.numel() and torch.equal(got, want)
    side = torch.cuda.Stream()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    torch.cuda.synchronize()
    t0 = time.monotonic()
    assert lib.hold_sms(sms - 1, 4_700_000_000, side.cuda_stream) == 0
    time.sleep(0.05)
    got, n = daq.pack_pool(dev)
    took = time.monotonic() - t0
    assert took > 4.0                         # it was held up
    assert n == want.numel() and torch.equal(got, want)
