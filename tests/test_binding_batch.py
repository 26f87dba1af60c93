"""What the Python binding of seq_tree_verify_batch hands to the library, seen by a stand-in for it (no GPU)."""
import ctypes as C

import pytest
import torch

from paper_2402_12374_b200 import binding as B


class _Library:
    """Takes the parameters and writes nothing."""

    def seq_tree_verify_batch(self, ref, stream):
        self.params = C.cast(ref, C.POINTER(B.VerifyBatchParams)).contents
        return B.SEQ_OK


@pytest.fixture
def library(monkeypatch):
    lib = _Library()
    monkeypatch.setattr(B, "load", lambda: lib)
    monkeypatch.setattr(B, "_dev", lambda t, name, dtype=None: None if t is None else t.data_ptr())
    monkeypatch.setattr(B, "_stream", lambda stream: 0)
    return lib


def _args(R, n, V):
    return (torch.full((R, n), -1, dtype=torch.int32), torch.zeros((R, n), dtype=torch.int32), torch.zeros((R, n, V)), torch.zeros((R, n, V)),
            1.0, torch.zeros((R, n + 1)))


@pytest.mark.parametrize("columns", [8, 5, 1])
def test_paths_have_room_for_every_request(library, columns):
    """Request r's path is written at r * tree_stride, n entries of it, whatever view `parent` is."""
    R, n, V = 3, 8, 16
    parent, *rest = _args(R, n, V)
    path, path_len, bonus = B.seq_tree_verify_batch(parent[:, :columns], *rest)
    assert library.params.request0.path == path.data_ptr()
    assert path.shape == (R, n) and path.is_contiguous()
    assert path.untyped_storage().nbytes() >= ((R - 1) * library.params.tree_stride + n) * 4
    assert path_len.shape == bonus.shape == (R,) and path.dtype == path_len.dtype == bonus.dtype == torch.int32
