"""The tiled tensor-core similarity kernel's CTAs wait for one another's norms, so they have to be
resident together.  While another stream's kernel holds some SMs for longer than the waits'
limit, a call must come later, not end with GPO_ERR_TIMEOUT; captured and replayed calls as well.
(The other kernel waits for nothing but the clock.)"""
import ctypes
import shutil
import subprocess

import pytest

from test_gpu_parity import batch_of, compare, gp_mod, oracle_params, oracle_run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

HOLDER = r"""
#include <cstdint>
__global__ void hold(uint64_t ns) {
  uint64_t t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  do {
    __nanosleep(100000);
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  } while (t - t0 < ns);
}
extern "C" int hold_sms(int blocks, int bytes, uint64_t ns, void* stream) {
  cudaError_t e = cudaFuncSetAttribute(hold, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) {
    hold<<<blocks, 32, bytes, static_cast<cudaStream_t>(stream)>>>(ns);
    e = cudaGetLastError();
  }
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def hold_sms(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("hold")
    (d / "hold.cu").write_text(HOLDER)
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-shared", "-Xcompiler", "-fPIC",
                           str(d / "hold.cu"), "-o", str(d / "libhold.so")])
    f = ctypes.CDLL(str(d / "libhold.so")).hold_sms
    f.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_uint64, ctypes.c_void_p]
    return f


def tiled(P, groups=40):
    b = batch_of("math", groups)  # 4 items per group, on more CTAs than the held GPU has free
    p = oracle_params(b)
    gp = P.GraphPO(kappa=p["kappa"], w=p["w"], lambda_eff=p["lambda_eff"], flags=P.binding.FLAG_TILED)
    db = P.Batch.from_arrays(b, device="cuda")
    return b, p, gp, db, gp.alloc_outputs(db, nodes=True)


def test_call_beside_a_kernel_that_holds_sms(gp_mod, hold_sms):
    import torch
    b, p, gp, db, out = tiled(gp_mod)
    gp.compute_into(db, out)
    gp.check()
    out["adv"].zero_()
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    # 24 SMs for 2.5 s (120 KB of shared memory: none of a similarity CTA's beside it)
    assert hold_sms(24, 120 << 10, 2_500_000_000, side.cuda_stream) == 0
    gp.compute_into(db, out)
    gp.check()
    compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, p), "held")
    side.synchronize()


def test_captured_tiled_call(gp_mod):
    import torch
    b, p, gp, db, out = tiled(gp_mod, 6)
    gp.compute_into(db, out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gp.compute_into(db, out)
    for _ in range(2):
        out["adv"].zero_()
        graph.replay()
        gp.check()
        compare({k: v.cpu().numpy() for k, v in out.items()}, oracle_run(b, p), "replay")
