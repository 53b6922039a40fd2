"""The bounded wait of the tensor-core kernels, by itself: a barrier at which nobody arrives, on a plan whose status word says that
another CTA has given up (the wait ends after 1024 looks); and the report that a wait leaves, as the host reads it."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2507_05228_b200 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "tcgen05.cuh"
namespace tc = cascade::tc;
template <bool kPointer>
__global__ void wait_once(int32_t* status, int* out) {
  __shared__ int words[4];
  __shared__ uint64_t barrier;
  if (threadIdx.x == 0) {
    words[1] = 0;
    tc::mbar_init(tc::smem_u32(&barrier), 1);
    tc::WaitCtx<kPointer, 2> wc;
    if constexpr (kPointer) wc.words = words;
    else wc.misc = tc::smem_u32(words);
    wc.status = status;
    out[0] = tc::wait_bar(wc, tc::smem_u32(&barrier), 0u, 9, 3);
    out[1] = wc.load(1);
  }
}
extern "C" int run(int32_t* status, int* out) {
  wait_once<false><<<1, 32>>>(status, out);
  wait_once<true><<<1, 32>>>(status, out + 2);
  return (int)cudaDeviceSynchronize();
}
"""


def test_a_wait_that_ends_by_another_report_raises_the_abort_flag(tmp_path):
    source, lib = tmp_path / "wait.cu", tmp_path / "wait.so"
    source.write_text(SOURCE)
    subprocess.check_call([build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                           "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include"), str(source), "-o", str(lib)])
    status = torch.zeros(64, dtype=torch.int32, device="cuda")
    out = torch.full((4,), 7, dtype=torch.int32, device="cuda")
    status[0] = 5
    torch.cuda.synchronize()
    run = ctypes.CDLL(str(lib)).run
    run.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    assert run(status.data_ptr(), out.data_ptr()) == 0
    assert out.tolist() == [0, 1, 0, 1]  # not arrived, flag raised; by address and by pointer
    assert status.tolist() == [5] + [0] * 63  # the report that is there stays


def test_the_report_has_the_progress_of_every_warp():
    """Twenty words: the fp32 kernel has that many warps, and its loading ones, which keep them, come last."""
    import gpu_util as gu
    from paper_2507_05228_b200 import binding as cb
    plan = cb.cascade_shard_plan(np.zeros(8, np.int32), np.zeros(8, np.int32), 1, 1)
    words = torch.as_tensor(gu._DevicePointer(plan.dev_ptr("q_off") - 256, 28, "<i4"), device="cuda")  # first in the plan's memory
    words.copy_(torch.arange(28, dtype=torch.int32) * 1000 + 1)
    with pytest.raises(cb.CascadeError, match=r"word = 1: .*block 1001,2001,3001 tile 4001; .*progress 8001 9001 .* 19001 .* 26001 27001\)"):
        plan.device_status()
    words.zero_()
    assert plan.device_status() == 0
    plan.destroy()
