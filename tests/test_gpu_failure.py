"""Failure detection without a GPU fault: a device wait that nothing satisfies gives up after
its bounded limit, reports PTD_ERR_TIMEOUT through the status word, and the context keeps
working (the next calls run and give correct results)."""
import ctypes
import subprocess
import time

import numpy as np
import pytest
import torch

import oracle
from paper_2607_10661_gb300 import ptd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


VOTE_SOURCE = r"""
#include "ptd_device.cuh"
__global__ void vote_kernel(int gave_up, int any, int* out) {   // the thread numbers (-1: none)
  __shared__ int abort_flag;
  if (threadIdx.x == 0) abort_flag = 0;
  __syncthreads();
  if ((int)threadIdx.x == gave_up) *(volatile int*)&abort_flag = 1;   // as its wait leaves it
  out[threadIdx.x] = ptd::cta_any_unless_aborted((int)threadIdx.x == any, &abort_flag) ? 1 : 0;
}
extern "C" int vote(int gave_up, int any, int* out) {
  vote_kernel<<<1, 128>>>(gave_up, any, out);
  return (int)cudaGetLastError();
}
"""


def test_threads_agree_after_a_wait_that_one_of_them_gave_up_on(tmp_path):
    """What fp32 attention branches to a barrier on is the same for every thread of the CTA, also when
    only one thread's wait ran out."""
    from paper_2607_10661_gb300 import _build

    src, so = tmp_path / "vote.cu", tmp_path / "vote.so"
    src.write_text(VOTE_SOURCE)
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", "-I", _build.CSRC, str(src), "-o", str(so)],
                   check=True)
    vote = ctypes.CDLL(str(so)).vote
    vote.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    for gave_up, any_, want in ((-1, 9, 1), (-1, -1, 0), (5, 9, 0), (70, 9, 0), (9, 9, 0)):
        out = torch.full((128,), -1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert vote(gave_up, any_, out.data_ptr()) == 0
        torch.cuda.synchronize()
        assert out.unique().tolist() == [want], (gave_up, any_)


def test_bounded_wait_times_out_and_the_context_survives():
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    t0 = time.time()
    assert ptd.check_bounded_wait(status) == 1
    torch.cuda.synchronize()
    dt = time.time() - t0
    assert int(status.item()) == ptd.TIMEOUT
    assert 1.5 < dt < 30.0                      # the 2 s limit, not an endless wait
    # the context still works: a top-k call right after, checked against the oracle
    g = np.random.default_rng(3)
    x = g.normal(size=(5, 3000)).astype(np.float32)
    idx = torch.empty((5, 4), dtype=torch.int32, device="cuda")
    val = torch.empty((5, 4), dtype=torch.float32, device="cuda")
    ptd.topk_draft(torch.tensor(x, device="cuda"), 4, idx, val)
    torch.cuda.synchronize()
    assert np.array_equal(idx.cpu().numpy(), oracle.topk_rows(x, 4)[0])
