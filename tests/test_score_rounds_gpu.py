"""tr_score over the row lengths its last round distinguishes (2, 4, 6 or 8
16-byte chunks a lane, whole and partial, after none to two full rounds): the
sums of each record against float64 on the stored inputs, within the record's
fp32 rounding and the score pass's three fp32 roundings (2^-22, and their
products)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

CHUNKS = [1, 31, 32, 33, 63, 64, 65, 96, 97, 128, 129, 191, 192, 193, 255, 256, 257, 320, 353, 448, 449, 512, 513, 577]


@pytest.mark.parametrize("dtype,per", [(torch.bfloat16, 8), (torch.float16, 8), (torch.float32, 4)])
def test_records(dtype, per):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2607_13500_gb300 as altr
    from paper_2607_13500_gb300 import _build
    _build.build()
    for c in CHUNKS:
        d = c * per
        g = torch.Generator().manual_seed(c)
        x, xp, xq = (torch.randn(9, d, generator=g).to(dtype) for _ in range(3))
        st, h2, s = altr.score(x.cuda(), xp.cuda(), xq.cuda())
        st = st.double().cpu().numpy()
        v, p, q = (t.double().numpy() for t in (x, xp, xq))
        l1, s2 = np.abs(v).sum(1), (v * v).sum(1)
        a, b, pq = (p * p).sum(1), (q * q).sum(1), (p * q).sum(1)
        for col, want in ((0, l1), (1, s2), (2, a), (3, b)):
            assert np.allclose(st[:, col], want, rtol=2.0 ** -21.9, atol=0), (d, col)
        assert np.all(np.abs(st[:, 4] + st[:, 5] - pq) <= 1e-9 * np.sqrt(a * b)), d
        assert np.allclose(st[:, 6], l1 * l1 / s2, rtol=2.0 ** -20), d
        assert np.allclose(h2.cpu().numpy(), np.log(l1 * l1 / s2), rtol=1e-5, atol=2e-6), d
        assert np.allclose(s.cpu().numpy(), pq / np.sqrt(a * b), rtol=0, atol=1e-6), d
