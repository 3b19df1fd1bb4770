"""The binding's one-pass layout check (rosko._mat) against its general parts
(_ptr, _ld): the same pointer, width and leading dimension for every layout
that a product accepts, and a refusal for those it does not.  GPU only."""
import pytest
import torch

from paper_2307_03930_gb300 import rosko

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [
    lambda x: x, lambda x: x[:, :5], lambda x: x[3:], lambda x: x[2:3], lambda x: x[:, :1],
    lambda x: x[2:3, :1], lambda x: x[::2], lambda x: x[:, 8:24], lambda x: x[:1, ::3][:, :1],
    lambda x: x.expand(1, 12, 32)[0], lambda x: x[:1].expand(4, 32),
])
def test_layouts(make):
    t = make(torch.arange(384, dtype=torch.float32, device="cuda").reshape(12, 32))
    assert rosko._mat(t) == (t.data_ptr(), t.shape[1], rosko._ld(t))


@pytest.mark.parametrize("make", [
    lambda x: x.t(), lambda x: x[:, ::2], lambda x: x[0], lambda x: x.reshape(3, 4, 32),
    lambda x: x.cpu(),
])
def test_refused(make):
    t = make(torch.zeros((12, 32), device="cuda"))
    with pytest.raises(ValueError):
        rosko._mat(t)


def test_without_elements_and_streams():
    assert rosko._mat(torch.zeros((0, 7), device="cuda")) == (0, 7, 7)
    assert rosko._mat(torch.zeros((7, 0), device="cuda")) == (0, 0, 1)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        assert rosko._stream(None) == s.cuda_stream
    assert rosko._stream(None) == torch.cuda.current_stream().cuda_stream
