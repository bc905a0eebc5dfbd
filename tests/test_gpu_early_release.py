"""A caller's kernel that releases its successor early (griddepcontrol.launch_dependents)
and writes a population or a fitness array only afterwards, with the old values in
every SM's L1: the call enqueued behind it on the same stream works on the new
values, whichever kernel is its first. The caller's kernel is compiled here; it reads,
waits a fixed time and writes inside its own arrays, one block per SM."""
import ctypes
import subprocess

import numpy as np
import pytest

from helpers import CHEB
from paper_1211_5481_gb300 import build, game
from paper_1211_5481_gb300 import datagen as dg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SOURCE = r"""
#include <cuda_runtime.h>
#include <stdint.h>
// dst = src (n words): every block first reads all of dst through L1, then lets the
// next launch start, waits 200 us and writes its share.
__global__ void late_write(uint32_t* dst, const uint32_t* src, long long n, uint32_t* seen) {
  uint32_t x = 0;
  for (long long i = threadIdx.x; i < n; i += blockDim.x) {
    uint32_t v;
    asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(v) : "l"(dst + i));
    x ^= v;
  }
  seen[blockIdx.x * blockDim.x + threadIdx.x] = x;
  __syncthreads();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
  do asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  while (t - t0 < 200000ull);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] = src[i];
}
extern "C" int run(void* dst, const void* src, long long n, void* seen, int blocks, void* st) {
  late_write<<<blocks, 256, 0, (cudaStream_t)st>>>((uint32_t*)dst, (const uint32_t*)src, n,
                                                   (uint32_t*)seen);
  return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def late_write(tmp_path_factory):
    d = tmp_path_factory.mktemp("late")
    (d / "late.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared",
                    "-o", str(d / "late.so"), str(d / "late.cu")], check=True)
    lib = ctypes.CDLL(str(d / "late.so"))
    blocks = torch.cuda.get_device_properties(0).multi_processor_count
    seen = torch.empty(blocks * 256, dtype=torch.int32, device="cuda")

    def run(dst, src, stream):
        assert dst.is_contiguous() and src.shape == dst.shape and src.dtype == dst.dtype
        p = lambda t: ctypes.c_void_p(t.data_ptr())
        words = dst.numel() * dst.element_size() // 4
        assert lib.run(p(dst), p(src), ctypes.c_longlong(words), p(seen), blocks,
                       ctypes.c_void_p(stream.cuda_stream)) == 0
    return run


@pytest.mark.parametrize("tied", [0, 1])
@pytest.mark.parametrize("form", ["fp32", "bf16", "bf16x3", "fp8", "gram"])
def test_evaluation_behind_an_early_release(late_write, form, tied):
    prec = {"fp32": game.GAME_PREC_FP32, "bf16": game.GAME_PREC_BF16, "fp8": game.GAME_PREC_FP8,
            "bf16x3": game.GAME_PREC_BF16X3, "gram": game.GAME_PREC_GRAM}[form]
    pr = dg.regression(7, 500, 6, 3, 0.05, degree=5)
    stream = torch.cuda.Stream()
    with game.Game(pr.X, pr.y, 5, CHEB, P=200, precision=prec, tied=tied, stream=stream) as g:
        old, new = (torch.from_numpy(dg.random_population(s, 200, g.K)).cuda() for s in (1, 2))
        pop, fit = old.clone(), torch.zeros(200, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        game.game_eval_fitness(g.h, new, fit)
        g.sync()
        want = fit.clone()
        torch.cuda.synchronize()
        late_write(pop, new, stream)
        game.game_eval_fitness(g.h, pop, fit)
        g.sync()
        assert torch.equal(fit, want)


@pytest.mark.parametrize("P", [300, 20_000])   # the two selection kernels
def test_candidates_behind_an_early_release(late_write, P):
    pr = dg.regression(7, 500, 3, 3, 0.05, degree=3)
    stream = torch.cuda.Stream()
    rng = np.random.default_rng(3)
    with game.Game(pr.X, pr.y, 3, CHEB, P=16, precision=game.GAME_PREC_BF16,
                   stream=stream) as g:
        pop = torch.from_numpy(dg.random_population(4, P, g.K)).cuda()
        old, new = (torch.from_numpy(rng.random(P)).cuda() for _ in range(2))
        idx = torch.zeros(16, dtype=torch.int32, device="cuda")
        fit = old.clone()
        torch.cuda.synchronize()
        game.game_rescore_top(g.h, pop, fit, 16, idx)   # allocations and G
        g.sync()
        fit.copy_(old)
        torch.cuda.synchronize()
        late_write(fit, new, stream)
        game.game_rescore_top(g.h, pop, fit, 16, idx)
        g.sync()
        assert np.array_equal(idx.cpu().numpy(), np.argsort(new.cpu().numpy(), kind="stable")[:16])
