"""Calls on settled inputs behind a kernel that lets its successors start early and writes the logits of the call after the next: the call
in between may overlap with that kernel, the one that reads the logits may not."""
import ctypes
import subprocess

import pytest
import torch

import helpers
from paper_2502_01662_b200 import build, synth
from paper_2502_01662_b200.binding import COS_RUN_INPUTS_SETTLED

pytestmark = pytest.mark.gpu

PRODUCER = r"""
#include <cuda_runtime.h>
__global__ void produce(const uint4* from, uint4* to, long long n, int naps) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int k = 0; k < naps; ++k) __nanosleep(1000);
  for (long long i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) to[i] = from[i];
}
extern "C" int launch(const void* from, void* to, long long bytes, int naps, void* stream) {
  produce<<<2, 256, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<const uint4*>(from), static_cast<uint4*>(to), bytes / 16, naps);
  return static_cast<int>(cudaGetLastError());
}
"""


@pytest.fixture(scope="module")
def produce(tmp_path_factory):
    where = tmp_path_factory.mktemp("producer")
    src, lib = where / "produce.cu", where / "libproduce.so"
    src.write_text(PRODUCER)
    subprocess.run([build.nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-Xcompiler", "-fPIC", "-o", str(lib), str(src)],
                   check=True, capture_output=True)
    fn = ctypes.CDLL(str(lib)).launch
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong, ctypes.c_int, ctypes.c_void_p]

    def go(source, target, naps):
        assert source.is_contiguous() and target.is_contiguous() and source.nbytes == target.nbytes and source.nbytes % 16 == 0
        assert fn(source.data_ptr(), target.data_ptr(), source.nbytes, naps, torch.cuda.current_stream().cuda_stream) == 0
    return go


# in one launch, in several (a bound on the streaming launch), and with decisions in a launch of their own
@pytest.mark.parametrize("n,batch,cluster_size", [(2, 7, 0), (2, 33, 0), (2, 33, 16), (5, 33, 0)])
def test_logits_written_before_the_call_ahead_are_seen(produce, n, batch, cluster_size):
    weights = (0.6, 0.4) if n == 2 else (0.3, 0.25, 0.2, 0.15, 0.1)
    w = synth.Workload("order", n, synth.COMBINE_PROB_ENSEMBLE, weights, 1.0, batch, 4, 8000, "bf16", "gauss", sigma=2.5, rho=0.8, proposer_rule="cycle")
    inputs = synth.make_inputs(w, "cuda")
    fresh, live = inputs["logits"], torch.empty_like(inputs["logits"])
    args = (inputs["drafts"], inputs["proposer"], inputs["seed"])
    v = helpers.make_verifier(w, cluster_size=cluster_size)
    try:
        assert v.info()["rows_at_once"] == (n == 2 and cluster_size == 0)
        want = [v.run(fresh, *args, k) for k in range(8)]
        torch.cuda.synchronize()
        for k in range(8):
            live.copy_(torch.roll(fresh, 1000 + k, dims=-1))
            torch.cuda.synchronize()
            produce(fresh, live, 100)
            v.run(fresh, *args, 99, flags=COS_RUN_INPUTS_SETTLED)
            got = v.run(live, *args, k, flags=COS_RUN_INPUTS_SETTLED)
            torch.cuda.synchronize()
            for key in ("accept_count", "out_tokens", "row_status"):
                assert torch.equal(got[key], want[k][key]), (k, key)
    finally:
        v.close()
