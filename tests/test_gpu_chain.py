"""Hand-overs of running sums between the blocks of a cluster (simt::Chain, simt_pairs.cuh).

The chain is run by a kernel of its own with a wait of 20 ms: complete, and with one row's
hand-over never sent.  That row must end as not ok in the block that holds its last state,
whichever later blocks lie between, and without a wait for each of them.  (Rows beside it, held
up by its wait, may run out of theirs as well: each is either not ok or has its whole sum.)
The allocation-free order's second kernel must then give no order at all.
"""
import ctypes
import subprocess
import time

import numpy as np
import pytest
import torch

from paper_2608_27922_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = r"""
#include "k_noalloc.cu"
namespace dkv {
int sm_count() { return 1; }
namespace {
template <int RT>
__global__ void chain_probe(int tiles, int silent_tile, int silent_row, float* sums, int* ok, int* last) {
  __shared__ int4 mail[RT];
  uint32_t C, z;
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(C));
  asm("mov.u32 %0, %%cluster_ctaid.x;" : "=r"(z));
  simt::Chain<RT, 20000000ull> chain(mail, (int)z, (int)C, tiles);
  const int sr = simt::scan_row<RT>();
  float x = 0.f;
  int y = 0;
  for (int t = z; t < tiles; t += C) {
    if (sr >= 0) {
      chain.take(sr, t, x, y);
      x += (float)((sr + 1) * (t + 1));
      if (y != chain.LOST) y += 1;
      if (t != silent_tile || sr != silent_row) chain.give(sr, t, x, y);
    }
    __syncthreads();
  }
  chain.finish();
  if (chain.last() && sr >= 0) {
    sums[sr] = x;
    ok[sr] = y != chain.LOST;
    last[sr] = y;
  }
}
template <int RT>
int probe(int C, int tiles, int silent_tile, int silent_row, void* sums, void* ok, void* last) {
  return (int)launch_kernel(chain_probe<RT>, dim3(C), simt::NT, 0, C, false, (cudaStream_t)0, tiles, silent_tile,
                            silent_row, (float*)sums, (int*)ok, (int*)last);
}
}  // namespace
}  // namespace dkv
extern "C" int chain(int rows, int C, int tiles, int silent_tile, int silent_row, void* sums, void* ok, void* last) {
  return rows == 64   ? dkv::probe<64>(C, tiles, silent_tile, silent_row, sums, ok, last)
         : rows == 32 ? dkv::probe<32>(C, tiles, silent_tile, silent_row, sums, ok, last)
                      : dkv::probe<16>(C, tiles, silent_tile, silent_row, sums, ok, last);
}
extern "C" int order(const void* scores, int N, void* perm, void* out) {
  dkv::noalloc_order<<<(N + 31) / 32, 32 * dkv::ORD_GROUPS>>>((const float*)scores, N, 1, (int32_t*)perm, (float*)out);
  return (int)cudaGetLastError();
}
extern "C" unsigned no_score() { return dkv::NO_SCORE; }
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    d = tmp_path_factory.mktemp("chain")
    (d / "probe.cu").write_text(SRC)
    subprocess.check_call([B.nvcc(), *B.ARCH, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", B.ROOT + "/include",
                           "-I", B.CSRC, str(d / "probe.cu"), "-o", str(d / "probe.so")])
    return ctypes.CDLL(str(d / "probe.so"))


@pytest.mark.parametrize("rows,C,tiles", [(64, 2, 2), (64, 4, 11), (32, 8, 9), (32, 8, 3), (16, 2, 1), (16, 8, 40)])
def test_a_hand_over_that_never_comes_marks_its_row(probe, rows, C, tiles):
    sums = torch.empty(rows, device="cuda")
    ok = torch.empty(rows, dtype=torch.int32, device="cuda")
    last = torch.empty(rows, dtype=torch.int32, device="cuda")
    P = [ctypes.c_void_p(x.data_ptr()) for x in (sums, ok, last)]
    want = np.arange(1, rows + 1) * (tiles * (tiles + 1) / 2.0)
    silent = [(-1, -1)] + [(t, r) for t in {0, tiles // 2, tiles - 2} if 0 <= t < tiles - 1 for r in (0, rows - 1)]
    for t, r in silent:
        t0 = time.perf_counter()
        for x in (sums, ok, last):
            x.fill_(-7)
        torch.cuda.synchronize()
        assert probe.chain(rows, C, tiles, t, r, *P) == 0
        torch.cuda.synchronize()
        good = ok.cpu().numpy() == 1
        assert good.all() if r < 0 else not good[r], (t, r)
        assert np.all(ok.cpu().numpy() >= 0), (t, r)   # every row has been reported
        assert np.array_equal(sums.cpu().numpy()[good], want[good].astype(np.float32)), (t, r)
        assert np.all(last.cpu().numpy()[good] == tiles), (t, r)
        assert time.perf_counter() - t0 < 1.0   # a wait of 20 ms or a few, not one per tile


@pytest.mark.parametrize("N", [1, 31, 300, 2049, 16384])
def test_no_order_without_every_score(probe, N):
    rng = np.random.default_rng(N)
    probe.no_score.restype = ctypes.c_uint
    s = rng.integers(0, max(2, N // 3), N).astype(np.float32)
    s[N // 2] = np.nan   # a NaN of the inputs is a score like others: it has a place
    s.view(np.uint32)[N // 3] = 0xffffffff
    perm = torch.empty(N, dtype=torch.int32, device="cuda")
    out = torch.empty(N, device="cuda")

    def order(bits):
        dev = torch.from_numpy(bits.view(np.int32)).cuda()
        perm.fill_(-7)
        torch.cuda.synchronize()
        assert probe.order(ctypes.c_void_p(dev.data_ptr()), N, ctypes.c_void_p(perm.data_ptr()),
                           ctypes.c_void_p(out.data_ptr())) == 0
        torch.cuda.synchronize()
        return perm.cpu().numpy()

    assert np.array_equal(np.sort(order(s.view(np.uint32))), np.arange(N))
    for i in {0, N // 2, N - 1}:
        bad = s.view(np.uint32).copy()
        bad[i] = probe.no_score()
        assert np.all(order(bad) == -1), i
        assert bool(torch.isnan(out[i]))
