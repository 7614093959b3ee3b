"""Descriptors written by the native extension equal those of the Python code, and what the extension
leaves out (tensor subclasses, wrong arguments) ends as it does in Python."""
import ctypes
import sys
import types

import pytest
import torch

import paper_2202_07471_b200 as sq
from paper_2202_07471_b200 import binding


class Sub(torch.Tensor):
    pass


def buffers():
    out = []
    for i, shape in enumerate([(4, 3, 3, 3), (5, 7), (6, 2, 9), (1, 1, 1, 1), (8, 16, 1, 7)]):
        w = torch.randn(shape)
        b = sq.alloc_outputs(torch.nn.Parameter(w) if i == 1 else w, kernel_err=i != 2, channel_err=i != 3, pack_int4=i == 4,
                             dequant=i == 0, dequant_bf16=i in (0, 4))
        if i in (1, 4):
            b.scales_in = torch.ones(shape[0])
        out.append(b)
    out.insert(2, sq.alloc_outputs(torch.randn(3, 5).as_subclass(Sub)))
    return out


def test_native_descriptors_equal_the_python_ones():
    bufs = buffers()
    got = bytes(binding._descriptors(bufs))
    want = b"".join(bytes(binding._descriptor(b)) for b in bufs)
    assert got == want and len(got) == len(bufs) * ctypes.sizeof(binding.Layer)
    assert binding._marshal is None or binding._marshal.fill(bufs, 0, ctypes.addressof(binding._descriptors(bufs))) == 2   # stops at the subclass


@pytest.mark.parametrize("bad", [lambda b: setattr(b, "scales_in", torch.ones(5)), lambda b: setattr(b, "scales_in", torch.ones(4).double()),
                                 lambda b: setattr(b, "w", torch.randn(4)), lambda b: setattr(b, "w", torch.randn(1, 2, 3, 4, 5))])
def test_wrong_arguments_are_rejected_as_before(bad):
    b = sq.alloc_outputs(torch.randn(4, 3, 3, 3))
    bad(b)
    with pytest.raises((ValueError, IndexError)):
        sq.ModelCall([sq.alloc_outputs(torch.randn(2, 2)), b])


@pytest.mark.parametrize("name", ["w", "codes", "scales_in"])
def test_no_reference_is_kept_of_a_tensor_without_storage(name):
    """data_ptr() of a sparse tensor raises, here as in Python; the objects looked at before are released."""
    b = sq.alloc_outputs(torch.randn(4, 3, 3, 3))
    sparse = torch.zeros(4, 3, 3, 3).to_sparse()
    setattr(b, name, sparse)
    before = sys.getrefcount(sparse), sys.getrefcount(b.scales), sys.getrefcount(b.w)
    for _ in range(50):
        with pytest.raises((RuntimeError, ValueError)):
            sq.ModelCall([b])
    assert (sys.getrefcount(sparse), sys.getrefcount(b.scales), sys.getrefcount(b.w)) == before


def test_an_extension_with_another_layout_is_not_used():
    built = binding._native(types.SimpleNamespace(layout=None, fill=None))
    assert built is None and binding._native(None) is None
    assert binding._native(types.SimpleNamespace(fill=None)) is None   # built before it told its layout
    if binding._marshal is not None:
        layout = binding._marshal.layout
        assert binding._native(types.SimpleNamespace(layout=layout)) is not None
        for i in range(len(layout)):   # a field elsewhere, another size
            other = layout[:i] + (layout[i] + 8,) + layout[i + 1:]
            assert binding._native(types.SimpleNamespace(layout=other)) is None
