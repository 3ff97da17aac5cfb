"""tr_put_words: host words written on the device by a kernel that carries
them, at the edges of its launch sizes (120 and 1000 words), and the binding's
choice between it and a copy."""
import ctypes

import pytest
import torch

from paper_2607_13500_gb300 import _build, _lib, api


@pytest.fixture(scope="module")
def lib():
    _build.build()
    return _lib.load()


def test_refuses_bad_arguments(lib):
    words = (ctypes.c_int32 * 4)()
    assert lib.tr_put_words(0x1000, ctypes.addressof(words), -1, None) == 1
    assert lib.tr_put_words(None, ctypes.addressof(words), 4, None) == 1
    assert lib.tr_put_words(0x1000, None, 4, None) == 1
    assert lib.tr_put_words(0x1002, ctypes.addressof(words), 4, None) == 4
    assert lib.tr_put_words(None, None, 0, None) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 119, 120, 121, 1000, 1001, 1120, 4000, 4001])
def test_words_arrive(lib, n):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    g = torch.Generator().manual_seed(n)
    words = torch.randint(-2 ** 31, 2 ** 31, (n,), generator=g).tolist()
    got = api._device_words(words, torch.device("cuda"))
    assert got.dtype == torch.int32 and got.tolist() == words


@pytest.mark.gpu
def test_one_line_call_with_many_images(lib):
    # budgets and offsets of more images than one launch carries
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2607_13500_gb300 as altr
    seqlens = [7 + i % 5 for i in range(900)]
    x, xp, xq = (torch.randn(sum(seqlens), 64, device="cuda").to(torch.bfloat16) for _ in range(3))
    one = altr.reduce(x, xp, xq, seqlens=seqlens, k=3, scores=True)
    kept = altr.Reducer(seqlens, 64, torch.bfloat16, "cuda", k=3, scores=True).run(x, xp, xq)
    assert torch.equal(one.idx, kept.idx) and torch.equal(one.y, kept.y) and one.cu_k == kept.cu_k
    assert one.status.tolist() == kept.status.tolist() and torch.equal(one.h2, kept.h2) and torch.equal(one.s, kept.s)
