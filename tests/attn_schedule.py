"""The attention schedule's rule (csrc/attn_schedule.h) compiled for the host, and what the
share kernel left in the workspace: the tests assert with them which schedule a case takes."""
import ctypes
import os
import subprocess
import tempfile

import torch

from paper_2608_27922_gb300 import build as B

WHOLE, SHARES, TWO = 0, 1, 2
CTAS, PART_BYTES = 152, (128 * 128 + 128) * 4   # k_tc_attn.cu: SPLIT_CTAS, PART_FLOATS

_SRC = r"""
#include "attn_schedule.h"
using namespace dkv::attn;
extern "C" int pick(int heads, int nq, float nt, float longest, int n_sm, int scratch) {
  return schedule(Sizes{heads, (nq + 127) / 128, nt, longest}, nq, n_sm, scratch != 0);
}
extern "C" int pay(int heads, int nq, float nt, float longest, int ctas) {
  return shares_pay(Sizes{heads, (nq + 127) / 128, nt, longest}, ctas);
}
extern "C" int most_ctas() { return SPLIT_CTAS; }
"""
_lib = None


def _rule():
    global _lib
    if _lib is None:
        d = tempfile.mkdtemp()
        src, so = os.path.join(d, "rule.cpp"), os.path.join(d, "rule.so")
        with open(src, "w") as f:
            f.write(_SRC)
        subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", B.CSRC, src, "-o", so])
        _lib = ctypes.CDLL(so)
        assert _lib.most_ctas() == CTAS
    return _lib


def _sizes(rows, W):
    tiles = [max(1, (m + 127) // 128 + (W + 127) // 128) for m in rows]
    return ctypes.c_float(sum(tiles) / len(tiles)), ctypes.c_float(max(tiles))


def launched(budgets, Nq, W, n_sm, scratch=True):
    """The launcher's choice for a handle of these budgets."""
    return _rule().pick(len(budgets), Nq, *_sizes(budgets, W), n_sm, int(scratch))


def cuts(occ, Nq, W, n_sm):
    """Whether the share kernel cuts units with these occupancies (else it takes whole ones)."""
    return bool(_rule().pay(len(occ), Nq, *_sizes(occ, W), min(n_sm, CTAS)))


def units_list(bank):
    """The share kernel's list of units in the workspace (int32 [152][4], the last bytes)."""
    size = CTAS * (2 * PART_BYTES + 16)
    at = bank.workspace.numel() - (size + 255) // 256 * 256 + CTAS * 2 * PART_BYTES
    return bank.workspace[at:at + CTAS * 16].view(torch.int32).view(CTAS, 4)


def n_sm():
    return torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count


class taken:
    """with taken(bank) as t: ...one attend...; then t.shares (the share kernel ran) and t.cut
    (units it cut)."""

    def __init__(self, bank):
        self.bank = bank

    def __enter__(self):
        units_list(self.bank).fill_(-9)
        return self

    def __exit__(self, *exc):
        torch.cuda.synchronize()
        last = units_list(self.bank)[:, 3].cpu()
        self.shares = bool((last != -9).any())
        self.cut = int((last > 0).sum())
