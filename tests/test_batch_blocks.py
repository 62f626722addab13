"""Batch calls refuse state blocks that the library would read or write past."""
from types import SimpleNamespace

import pytest
import torch

import paper_1501_05654_gb300 as rsg


class _Block(torch.Tensor):
    is_cuda = True   # stands in for a device tensor: the check looks at its kind and size only


def _block(*shape, dtype=torch.complex64):
    return torch.zeros(shape, dtype=dtype).as_subclass(_Block)


def _batch():
    b = rsg.Batch.__new__(rsg.Batch)
    b.hams = [SimpleNamespace(mesh=SimpleNamespace(P=10)), SimpleNamespace(mesh=SimpleNamespace(P=20))]
    b.S = [3, 4]
    return b


@pytest.mark.parametrize("blocks", [
    [_block(10, 4)], [_block(10, 3), _block(20, 4)], [_block(10, 4), _block(10, 4)],
    [_block(10, 4), _block(20, 4, dtype=torch.complex128)], [_block(10, 4), _block(4, 20).T], [torch.zeros(10, 4), _block(20, 4)]])
def test_refused(blocks):
    for call in (lambda: _batch().propagate(blocks, 1, 0.01), lambda: _batch().autotune(blocks, 0.01)):
        with pytest.raises(ValueError, match="block"):
            call()


def test_accepted():
    _batch()._check([_block(10, 4), _block(20, 4)])
    _batch()._check([_block(40), _block(20, 6)])   # the size counts
