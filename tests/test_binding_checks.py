"""Sizes and layouts that the Python binding refuses before the library, which
sees raw pointers, is called.  The tensors are stand-ins with what the checks
read, so no GPU is needed and nothing could be written."""

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def g():
    from paper_2109_01329_gb300 import build

    build.build()
    import paper_2109_01329_gb300 as grng

    return grng


class CudaTensor:
    """What the binding asks of a CUDA tensor."""

    is_cuda = True
    device = torch.device("cuda", 0)

    def __init__(self, numel, dtype=torch.float32, contiguous=True):
        self._numel, self.dtype, self._contiguous = numel, dtype, contiguous

    def numel(self):
        return self._numel

    def is_contiguous(self):
        return self._contiguous

    def element_size(self):
        return torch.empty(0, dtype=self.dtype).element_size()

    def get_device(self):
        return 0

    def data_ptr(self):
        return 0x10000


@pytest.mark.parametrize("dtype", [1, 2])
def test_transform_words_refuses_more_outputs_than_out_holds(g, dtype):
    d = g.Distribution(g.UNIFORM, dtype, 0.0, 1.0)
    out = CudaTensor(100, torch.float32 if dtype == 1 else torch.float64)
    with pytest.raises(ValueError, match="n exceeds the tensor size"):
        g.transform_words(d, CudaTensor(1000, torch.int32), out, n=101)


def test_batch_refuses_more_outputs_than_out_holds(g):
    d = g.Distribution.uniform(0.0, 1.0)
    fits = (g.Engine(g.PHILOX4X32X10, 1), d, CudaTensor(100), 100)
    with pytest.raises(ValueError, match="request 1: n exceeds the tensor size"):
        g.Batch([fits, (g.Engine(g.PHILOX4X32X10, 2), d, CudaTensor(100), 101)])


def test_batch_refuses_outputs_with_gaps(g):
    """A batch writes a request's outputs densely from its tensor's address."""
    d = g.Distribution.uniform(0.0, 1.0)
    with pytest.raises(ValueError, match="request 0: out must be contiguous"):
        g.Batch([(g.Engine(g.PHILOX4X32X10, 1), d, CudaTensor(100, contiguous=False), 100)])
