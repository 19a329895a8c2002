"""The GEMM is part of a library that every rank of a job loads: its loads stay within one CTA's own shared memory (a
multicast load of memory on another GPU is not safe), and a call runs on the GPU that holds its operands. No GPU
needed."""
import contextlib
import glob
import os
import re

import pytest
import torch

from paper_2602_19775_gb300 import SSAError, ssa

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_source_loads_by_multicast():
    for path in glob.glob(os.path.join(ROOT, "paper_2602_19775_gb300", "csrc", "*.cu*")):
        assert not re.search(r"multicast", open(path).read()), path


class _On:
    """What bf16_gemm looks at of an operand before it enters the operand's device."""
    dtype, is_cuda = torch.bfloat16, True

    def __init__(self, device):
        self.device = torch.device(device)


def test_gemm_runs_on_the_device_of_its_operand(monkeypatch):
    seen = []

    @contextlib.contextmanager
    def device(d):
        seen.append(("enter", d))
        yield
        seen.append(("leave", d))

    monkeypatch.setattr(torch.cuda, "device", device)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(ssa, "_bf16_gemm_here", lambda *a: seen.append(("run", a[0].device)))
    here = torch.device("cuda:1")
    ssa.bf16_gemm(_On(here), _On(here))
    assert seen == [("enter", here), ("run", here), ("leave", here)]


def test_gemm_refuses_host_operands():
    a = torch.zeros((8, 8), dtype=torch.bfloat16)
    with pytest.raises(SSAError):
        ssa.bf16_gemm(a, a)


def test_rows_too_far_apart_for_the_call_are_copied():
    """The call's row strides are 32-bit: columns of a matrix with 2^31 of them are copied together."""
    x = torch.empty_strided((3, 64), (2 ** 31, 1), dtype=torch.bfloat16, device="meta")
    rows, ld = ssa._tma_rows(x)
    assert ld == 64 and rows.shape == (3, 64) and rows.stride(0) == 64
    x = torch.empty_strided((3, 64), (2 ** 31 - 8, 1), dtype=torch.bfloat16, device="meta")
    assert ssa._tma_rows(x)[1] == 2 ** 31 - 8
