"""What a GEMM CTA does once a wait of it has given up: it waits, boundedly, for its copies and MMAs in flight before it
gives up its shared memory and TMEM.  The bounded wait by itself on a GPU (a copy that lands, a phase that nothing
completes), and on the CPU that every GEMM kernel takes it between its last barrier and its deallocation."""
import ctypes
import os
import re
import subprocess

import pytest
import torch

from gpu_common import need_gpu

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2107_02103_gb300", "csrc")

SRC = r'''
#include "tc_gemm.cuh"
using namespace dpc;
// three stages of 256 bytes; barrier 1 asks for an arrival more than it gets
__global__ void probe(const unsigned char *src, int *out, unsigned char *copied) {
  __shared__ __align__(128) unsigned char stage[3][256];
  __shared__ __align__(8) uint64_t bar[3];
  if (threadIdx.x == 0) {
    for (int s = 0; s < 3; ++s)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc::smem_u32(bar + s)), "r"(s == 1 ? 2 : 1));
    asm volatile("fence.mbarrier_init.release.cluster;");
    for (int s = 0; s < 3; ++s) {
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_u32(bar + s)), "r"(256u) : "memory");
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                       tc::smem_u32(stage[s])), "l"(src + 256 * s), "r"(256u), "r"(tc::smem_u32(bar + s)) : "memory");
    }
    out[0] = tc::settle(tc::smem_u32(bar), 0u);
    out[1] = tc::settle(tc::smem_u32(bar + 1), 0u);
    out[2] = tc::settle(tc::smem_u32(bar + 2), 0u);
    out[3] = tc::settle_copies(tc::smem_u32(bar), 3, 1);  // the first stage alone
    out[4] = tc::settle_copies(tc::smem_u32(bar), 3, 3);
    out[5] = tc::settle_copies(tc::smem_u32(bar), 3, 0);  // none issued
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar + 1)) : "memory");
    out[6] = tc::settle_copies(tc::smem_u32(bar), 3, 3);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 768; i += blockDim.x) copied[i] = stage[i / 256][i % 256];
}
extern "C" int run(const unsigned char *src, int *out, unsigned char *copied) {
  probe<<<1, 32>>>(src, out, copied);
  return (int)cudaDeviceSynchronize();
}
'''


@pytest.mark.gpu
def test_bounded_wait(tmp_path):
    need_gpu()
    (tmp_path / "probe.cu").write_text(SRC)
    so = str(tmp_path / "probe.so")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "--expt-relaxed-constexpr", "-I", CSRC, "-I", os.path.join(CSRC, "..", "..", "include"),
                    str(tmp_path / "probe.cu"), os.path.join(CSRC, "dp_host.cu"), "-o", so], check=True)
    src = (torch.arange(768) % 251).to(torch.uint8).cuda()
    out, copied = torch.full((7,), -1, dtype=torch.int32, device="cuda"), torch.zeros(768, dtype=torch.uint8, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert ctypes.CDLL(so, mode=os.RTLD_LAZY).run(p(src), p(out), p(copied)) == 0
    assert out.tolist() == [1, 0, 1, 1, 0, 1, 1] and torch.equal(copied, src)


@pytest.mark.parametrize("name,stages", [("tab_gemm.cuh", "kStages"), ("tab_gemm_b8.cuh", "kStagesB"),
                                         ("fit_gemm.cuh", "kStagesF")])
def test_every_gemm_settles_before_it_deallocates(name, stages):
    src = open(os.path.join(CSRC, name)).read()
    body = src[:src.index("tcgen05.dealloc")]
    tail = re.sub(r"\s+", " ", body[body.rindex("tcgen05.fence::after_thread_sync"):])
    assert re.search(rf"if \(\*abortf\) {{ // uniform if \(tid == 0\) settle_copies\(smem_u32\(full\), {stages}, issued\); "
                     r"if \(tid == 32 && issued > 0\) settle\(smem_u32\(acc_full.*\); __syncthreads\(\); }", tail)
