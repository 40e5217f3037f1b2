"""The merge of split sequences by itself: what it does with what a decode kernel has left, or has not."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def merge_alone(tmp_path_factory):
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "merge_alone.cu")
    so = str(tmp_path_factory.mktemp("merge") / "libmerge.so")
    subprocess.check_call([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", src, "-o", so])
    f = ctypes.CDLL(so).merge_alone
    f.argtypes = [ctypes.c_void_p] * 7
    return f


def test_nothing_is_merged_after_a_wait_ran_out(merge_alone):
    # A decode kernel that gives up may not have said what there is to merge: the record then holds what was there before, and
    # the sequence and the partials that it names need not exist.  (Here they do, so that a merge would show.)
    import torch
    dev = torch.device("cuda", 0)
    info = torch.tensor([[0, 0, 4, 0]], dtype=torch.int32, device=dev)          # item 0, first partial in slot 0, four partials
    part_lse = torch.zeros((8, 32), dtype=torch.float32, device=dev)
    part_o = torch.ones((8, 32, 512), dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream().cuda_stream
    for status, merged in ((0, True), (1, False)):
        word = torch.tensor([status], dtype=torch.int32, device=dev)
        out = torch.full((16, 512), -7.0, dtype=torch.bfloat16, device=dev)
        lse = torch.full((16,), -7.0, dtype=torch.float32, device=dev)
        torch.cuda.synchronize()
        assert merge_alone(word.data_ptr(), info.data_ptr(), part_lse.data_ptr(), part_o.data_ptr(), out.data_ptr(), lse.data_ptr(), stream) == 0
        torch.cuda.synchronize()
        assert bool((out == (1.0 if merged else -7.0)).all())
        assert bool(torch.allclose(lse, torch.full_like(lse, 1.3862944 if merged else -7.0)))
