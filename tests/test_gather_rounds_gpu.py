"""tr_gather over the row lengths its dispatch distinguishes: one to eight
16-byte loads a lane and round, whole and partial last rounds, one and more
rounds; a bit copy of the named rows."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, d) for d in (8, 256, 264, 512, 776, 1024, 1288, 1536, 1800, 2048, 2056,
                                                                   2304, 3584, 4096, 4360, 16384)] +
                                    [(torch.float32, d) for d in (4, 132, 1028, 2048)])
def test_rows_are_copied(dtype, d):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2607_13500_gb300 import _build, _lib
    from paper_2607_13500_gb300.api import _Tokens, _ptr, _stream
    _build.build()
    seqlens, ks = [37, 5, 60], [11, 0, 29]
    dev = torch.device("cuda")
    g = torch.Generator(device="cuda").manual_seed(d)
    x = torch.randn(sum(seqlens), d, generator=g, device=dev).to(dtype)
    idx, rows, off = [], [], 0
    for n, k in zip(seqlens, ks):
        i = torch.randperm(n, generator=g, device=dev)[:k].sort().values
        idx.append(i)
        rows.append(off + i)
        off += n
    idx, rows = torch.cat(idx).to(torch.int32), torch.cat(rows)
    y = torch.full((sum(ks) + 1, d), 7.0, dtype=dtype, device=dev)  # a guard row after the output
    d_cu = torch.tensor([0, 11, 11, 40], dtype=torch.int32, device=dev)
    tok = _Tokens(x, None, x, seqlens)
    _lib.check("tr_gather", _lib.load().tr_gather(tok.ref(), _ptr(d_cu), _ptr(idx), sum(ks), _ptr(y), _stream(dev)))
    torch.cuda.synchronize()
    assert torch.equal(y[:-1], x[rows]) and bool((y[-1] == 7.0).all())
