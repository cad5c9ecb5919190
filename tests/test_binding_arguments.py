"""What the native calls take and refuse, without a GPU: the arguments are looked at before anything is launched."""
import pytest
import torch

import paper_2408_06995_b200 as fpq


@pytest.fixture(scope="module")
def ext():
    return fpq._load_layers()


def _split_arguments(workspace, x1=None):
    x = torch.zeros(1, 4, 8, 8) if x1 is None else x1
    w = torch.zeros(16, dtype=torch.uint8)
    return (x, 1.0, torch.zeros(1, 4, 8, 8), 1.0, w, torch.ones(4), fpq.E4M3, fpq.E4M3, None, torch.zeros(1, 4, 8, 8), 3, 3, 1, 1,
            workspace)


class Scratch:
    """Memory that is no tensor."""

    def __init__(self, size):
        self.memory = torch.zeros(16, dtype=torch.uint8)
        self.size = size

    def data_ptr(self):
        return self.memory.data_ptr()

    def numel(self):
        if isinstance(self.size, Exception):
            raise self.size
        return self.size


def test_a_workspace_without_a_size_is_refused(ext):
    with pytest.raises(AttributeError, match="numel"):
        ext.conv2d_split(*_split_arguments(torch.zeros(16).untyped_storage()))


def test_a_workspace_is_asked_for_its_size(ext):
    with pytest.raises(KeyError, match="asked"):
        ext.conv2d_split(*_split_arguments(Scratch(KeyError("asked"))))


@pytest.mark.parametrize("size,error", [(-1, ValueError), ("16", TypeError), (1 << 70, OverflowError)])
def test_sizes_that_are_none(ext, size, error):
    with pytest.raises(error):
        ext.conv2d_split(*_split_arguments(Scratch(size)))


def test_tensors_without_sizes_raise(ext):
    # (an exception of torch's C++ side that left the call would end the process)
    ragged = torch.nested.nested_tensor([torch.zeros(4, 8, 8), torch.zeros(4, 8, 9)])
    with pytest.raises(RuntimeError, match="irregular"):
        ext.conv2d_split(*_split_arguments(torch.zeros(16, dtype=torch.uint8), ragged))


@pytest.mark.gpu
def test_sparse_tensors_raise():
    x = torch.zeros(4, 320, device="cuda").to_sparse()
    w = torch.zeros(1 << 16, dtype=torch.uint8, device="cuda")
    with pytest.raises((RuntimeError, AssertionError)):
        fpq.fpq_linear(x, w, torch.ones(64, device="cuda"), 1.0, fpq.E4M3, fpq.E4M3, None, 64, torch.empty(4, 64, device="cuda"), w)


@pytest.mark.gpu
def test_a_workspace_that_is_too_small_is_refused_whatever_holds_it():
    x = torch.randn(300, 320, device="cuda")
    w = torch.zeros(64, 320, dtype=torch.uint8, device="cuda")
    prep = fpq.fpq_prepare_weight(w, fpq.E4M3, fpq.LINEAR, 64, 320)
    need = fpq.fpq_linear_workspace_size(300, 64, 320, fpq.E4M3, fpq.E4M3)
    memory = torch.empty(need, dtype=torch.uint8, device="cuda")

    class Held(Scratch):
        def __init__(self, size):
            self.memory, self.size = memory, size

    scale = torch.ones(64, device="cuda")
    with pytest.raises(fpq.FpqError) as e:
        fpq.fpq_linear(x, prep, scale, 0.01, fpq.E4M3, fpq.E4M3, None, 64, workspace=Held(need - 1))
    assert e.value.code == fpq.ERR_WORKSPACE
    y = fpq.fpq_linear(x, prep, scale, 0.01, fpq.E4M3, fpq.E4M3, None, 64, workspace=Held(need))
    assert fpq.fpq_read_status() == fpq.OK and not bool(y.any())
