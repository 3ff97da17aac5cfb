"""The encoder's final-layer MLP on the tensor cores with the scoring fused
into its second GEMM (tr_mlp_hidden, tr_mlp_score; Eq. 5, Section IV-B).

* H = sigma(x' W1^T + b1) and x'' = H W2^T + b2 against float64 references
  on the CPU (the x'' reference takes the kernel's own H, so each GEMM is
  checked alone).  Tolerance per element: 2^-8 |ref| (the bf16 rounding of
  the output, with a factor 2 of margin) + 2^-16 sum_k |a_k b_k| (fp32
  accumulation of K products; a pairwise or blocked fp32 sum of K = 4096
  terms stays near log2(K) u = 2^-20.4 of that, the bound leaves 16x) +
  for H, the same propagated through sigma (|sigma'| <= 1.13).
* x = bf16(resid + x'') bit for bit, recomputed from the stored x''.
* The statistics records against the exact sums of the stored x, x', x''.
* The selection that tr_select makes from these records: kept indices and
  gathered rows bit for bit against the oracle run on the stored tensors,
  and identical to the selection from tr_score's records.
"""
import math

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2607_13500_gb300 import _build
    _build.build()


def _alt():
    import paper_2607_13500_gb300 as altr
    return altr


def _f64(t):
    return t.float().cpu().numpy().astype(np.float64)


def _sigma(v, act):
    if act == "gelu":
        return 0.5 * v * (1.0 + torch.special.erf(v / math.sqrt(2.0)))
    if act == "quick_gelu":
        return v * torch.sigmoid(1.702 * v)
    return v


def _gemm_ref(a, b, bias):
    """a [m, k] b [n, k]^T (+ bias) and sum_k |a_k b_k| in float64 on the CPU."""
    a64, b64 = a.double().cpu(), b.double().cpu()
    v = a64 @ b64.T
    mag = a64.abs() @ b64.abs().T
    if bias is not None:
        v = v + bias.double().cpu()
    return v, mag


def _check_close(got, ref, mag, slope=1.0):
    got = got.double().cpu()
    tol = 2.0 ** -8 * ref.abs() + slope * 2.0 ** -16 * mag + 1e-6
    bad = (got - ref).abs() > tol
    assert not bad.any(), (int(bad.sum()), float(((got - ref).abs() / tol).max()))


def _inputs(t, d, dh, seed, resid=True, bias=True):
    g = torch.Generator().manual_seed(seed)
    x_pre = torch.randn(t, d, generator=g).to(torch.bfloat16)
    w1 = (torch.randn(dh, d, generator=g) / math.sqrt(d)).to(torch.bfloat16)
    w2 = (torch.randn(d, dh, generator=g) / math.sqrt(dh)).to(torch.bfloat16)
    b1 = 0.1 * torch.randn(dh, generator=g) if bias else None
    b2 = 0.1 * torch.randn(d, generator=g) if bias else None
    r = torch.randn(t, d, generator=g).to(torch.bfloat16) if resid else None
    dev = torch.device("cuda")
    mv = lambda v: None if v is None else v.to(dev)
    return mv(x_pre), mv(w1), mv(w2), mv(b1), mv(b2), mv(r)


CASES = [
    # name, rows, D, hidden, activation, residual, bias
    ("clip_l", 300, 1024, 4096, "gelu", True, True),           # 3 row blocks, the last ragged
    ("ragged_dims", 200, 1152, 4304, "quick_gelu", True, False),  # a half column block, a K tail of 16
    ("one_row", 1, 256, 512, "none", False, True),              # x = x'' (no residual)
    ("even_tiles_ragged", 600, 1296, 4400, "gelu", True, True),  # even column tile counts, every edge ragged
]


@pytest.mark.parametrize("name,t,d,dh,act,resid,bias", CASES, ids=[c[0] for c in CASES])
def test_mlp_outputs_and_records(name, t, d, dh, act, resid, bias):
    altr = _alt()
    xp, w1, w2, b1, b2, r = _inputs(t, d, dh, seed=len(name), resid=resid, bias=bias)
    m = altr.Mlp(t, w1, w2, b1, b2, act=act, scores=True)
    out = m.run(xp, r)
    torch.cuda.synchronize()
    assert out.error.item() == 0
    # H against float64, through sigma
    v1, mag1 = _gemm_ref(xp, w1, b1)
    _check_close(out.h, _sigma(v1, act), mag1, slope=1.13)
    # x'' against float64 on the kernel's own H
    v2, mag2 = _gemm_ref(out.h, w2, b2)
    _check_close(out.x_post, v2, mag2)
    # x = bf16(resid + x'') exactly
    want_x = (r.float() + out.x_post.float()).to(torch.bfloat16) if resid else out.x_post
    assert torch.equal(out.x.view(torch.int16), want_x.view(torch.int16))
    # records: the sums of the stored tensors
    st = out.stats.double().cpu().numpy()
    xx, pp, qq = _f64(out.x), _f64(xp), _f64(out.x_post)
    l1, s2 = np.abs(xx).sum(1), (xx * xx).sum(1)
    a, b, p = (pp * pp).sum(1), (qq * qq).sum(1), (pp * qq).sum(1)
    for col, want in ((0, l1), (1, s2), (2, a), (3, b)):
        assert np.allclose(st[:, col], want, rtol=2.0 ** -23, atol=0), col
    assert np.all(np.abs(st[:, 4] + st[:, 5] - p) <= 1e-9 * np.sqrt(a * b))
    assert np.allclose(st[:, 6], l1 * l1 / s2, rtol=2.0 ** -22)
    assert np.allclose(st[:, 7], p / np.sqrt(a * b), rtol=0, atol=2.0 ** -23)
    # the same records as the scoring pass over the stored tensors
    ref_stats, _, _ = altr.score(out.x, xp, out.x_post)
    torch.cuda.synchronize()
    rs = ref_stats.double().cpu().numpy()
    assert np.allclose(st[:, :4], rs[:, :4], rtol=4e-7, atol=0)
    # a second call gives the same bits
    h0, q0, x0, s0 = (v.clone() for v in (out.h, out.x_post, out.x, out.stats))
    out2 = m.run(xp, r)
    torch.cuda.synchronize()
    for u, w in ((h0, out2.h), (q0, out2.x_post), (x0, out2.x), (s0, out2.stats)):
        assert torch.equal(u, w)
    assert out2.error.item() == 0


def _select_and_check(altr, out, xp, seqlens, budget, images):
    """tr_select on the fused records: indices and gathered rows against the
    oracle on the stored tensors, and equal to the selection on tr_score's."""
    ks, k1s, cu = budget
    idx, _, _, status = altr.select(out.x, xp, out.x_post, out.stats, seqlens=seqlens, budget=budget)
    stats2, _, _ = altr.score(out.x, xp, out.x_post, seqlens=seqlens)
    idx2, _, _, _ = altr.select(out.x, xp, out.x_post, stats2, seqlens=seqlens, budget=budget)
    torch.cuda.synchronize()
    st = status.cpu().tolist()
    assert st[1] == 0 and st[3] == 0, st
    assert torch.equal(idx, idx2)
    from paper_2607_13500_gb300 import _lib
    from paper_2607_13500_gb300.api import _Tokens, _ptr, _stream
    tok = _Tokens(out.x, xp, out.x_post, seqlens)
    y = torch.empty(max(cu[-1], 1), out.x.shape[1], dtype=torch.bfloat16, device=out.x.device)
    d_cu = torch.tensor(cu, dtype=torch.int32, device=out.x.device)
    _lib.check("tr_gather", _lib.load().tr_gather(tok.ref(), _ptr(d_cu), _ptr(idx), cu[-1], _ptr(y),
                                                  _stream(out.x.device)))
    torch.cuda.synchronize()
    idx_h, y_h = idx.cpu().numpy(), y.cpu()
    offs = np.concatenate([[0], np.cumsum(seqlens)]).astype(np.int64)
    for b in images:
        o0, o1 = int(offs[b]), int(offs[b + 1])
        ref = oracle.select_image(_f64(out.x[o0:o1]), _f64(xp[o0:o1]), _f64(out.x_post[o0:o1]), ks[b], k1s[b])
        assert np.array_equal(idx_h[cu[b]:cu[b + 1]], ref["kept"]), b
        rows = out.x[o0:o1].cpu()[torch.from_numpy(ref["kept"].astype(np.int64))]
        assert torch.equal(y_h[cu[b]:cu[b + 1]].view(torch.int16), rows.view(torch.int16)), b


def test_fused_selection_small():
    # Three 576-token images of the CLIP-L-shaped workload (cluster mixture,
    # activation outliers), K = 192 and K = 64.
    altr = _alt()
    w = synth.make_mlp(seed=3, device="cuda", batch=3)
    m = altr.Mlp(w.total, w.w1, w.w2, w.b1, w.b2, act="gelu")
    out = m.run(w.x_pre, w.resid)
    torch.cuda.synchronize()
    assert out.error.item() == 0
    for k in (192, 64):
        budget = altr.budgets(w.seqlens, k=k)
        _select_and_check(altr, out, w.x_pre, w.seqlens, budget, range(w.batch))


def test_fused_selection_full_size():
    # The full CLIP-L-shaped batch (64 images x 576 tokens, D = 1024,
    # hidden 4096): GEMM outputs on sampled rows, the selection of sampled
    # images against the oracle.
    altr = _alt()
    w = synth.make_mlp(seed=0, device="cuda")
    m = altr.Mlp(w.total, w.w1, w.w2, w.b1, w.b2, act="gelu")
    out = m.run(w.x_pre, w.resid)
    torch.cuda.synchronize()
    assert out.error.item() == 0
    rows = torch.tensor([0, 1, 577, 9000, 20000, w.total - 1])
    v1, mag1 = _gemm_ref(w.x_pre[rows], w.w1, w.b1)
    _check_close(out.h[rows], _sigma(v1, "gelu"), mag1, slope=1.13)
    v2, mag2 = _gemm_ref(out.h[rows], w.w2, w.b2)
    _check_close(out.x_post[rows], v2, mag2)
    want_x = (w.resid.float() + out.x_post.float()).to(torch.bfloat16)
    assert torch.equal(out.x.view(torch.int16), want_x.view(torch.int16))
    budget = altr.budgets(w.seqlens, k=w.k)
    _select_and_check(altr, out, w.x_pre, w.seqlens, budget, [0, 37, 63])


# ---------------------------------------------------------------- projector on the kept tokens
@pytest.mark.parametrize("name,over,bud,d_out,act", [
    ("llava576", dict(batch=3, d=1024), dict(k=192), 4096, "gelu"),           # LLaVA-1.5's 1024 -> 4096 layer
    ("ragged_dynres", dict(batch=5, n=(256, 3000), d=1152), dict(ratio=(2, 9)), 1280, "quick_gelu"),
    ("llava576", dict(batch=2, d=1040), dict(k=64), 512, "gelu"),              # a partial last k-block
], ids=["llava576", "ragged_dynres", "partial_kblock"])
def test_project_kept(name, over, bud, d_out, act):
    # Selection, then the projector's first layer on the kept tokens read
    # from x by index: bit for bit tr_project on the gathered copy y (the
    # hidden-GEMM kernel with plain TMA loads), and within the GEMM tolerance
    # of float64 on the kept rows.
    altr = _alt()
    w_in = synth.make(name, seed=17, device="cuda", **over)
    budget = altr.budgets(w_in.seqlens, **bud)
    r = altr.reduce(w_in.x, w_in.x_pre, w_in.x_post, seqlens=w_in.seqlens, budget=budget)
    g = torch.Generator(device="cuda").manual_seed(5)
    w = (torch.randn(d_out, w_in.d, generator=g, device="cuda") / math.sqrt(w_in.d)).to(torch.bfloat16)
    bias = 0.05 * torch.randn(d_out, generator=g, device="cuda")
    z, err = altr.project_kept(w_in.x, r.idx, budget[2], w, bias, act=act, seqlens=w_in.seqlens)
    zh, err_h = altr.project(r.y, w, bias, act=act)
    torch.cuda.synchronize()
    assert err.item() == 0 and err_h.item() == 0
    assert torch.equal(z.view(torch.int16), zh.view(torch.int16))
    v, mag = _gemm_ref(r.y, w, bias)
    _check_close(z, _sigma(v, act), mag, slope=1.13)


def test_project_kept_index_outside_its_image():
    # A kept index past its image's tokens (or negative) feeds a zero row:
    # its output row is sigma(bias), the other rows are untouched by it.
    altr = _alt()
    x = _inputs(100, 256, 512, seed=9, resid=False, bias=False)[0]
    idx = torch.tensor([0, 10, 55, -3, 1, 49, 50], dtype=torch.int32, device="cuda")
    cu = [0, 4, 7]
    g = torch.Generator(device="cuda").manual_seed(6)
    w = (torch.randn(256, 256, generator=g, device="cuda") / 16).to(torch.bfloat16)
    bias = 0.1 * torch.randn(256, generator=g, device="cuda")
    z, err = altr.project_kept(x, idx, cu, w, bias, act="gelu", seqlens=[50, 50])
    torch.cuda.synchronize()
    assert err.item() == 0
    rows = torch.zeros(7, 256, dtype=torch.bfloat16, device="cuda")  # slots 2, 3, 6 stay zero rows
    for slot, row in [(0, 0), (1, 10), (4, 51), (5, 99)]:
        rows[slot] = x[row]
    v, mag = _gemm_ref(rows, w, bias)
    _check_close(z, _sigma(v, "gelu"), mag, slope=1.13)


def _columns(rows, n, k, kind):
    from paper_2607_13500_gb300 import _lib
    return _lib.load().tr_gemm_columns(rows, n, k, kind)


# The layouts a GEMM may take, by size: tile columns of the hidden and the
# score GEMM (asserted), with ragged rows, columns and k-blocks.
LAYOUT_CASES = [
    ((256, 64), 1000, 1024, 16400, "none", True, True),     # 4 x 16 score tiles, 256.25 k-blocks
    ((128, 64), 1, 256, 6144, "none", False, True),         # one row, 4 score tiles, 96 k-blocks
    ((128, 64), 300, 528, 4464, "gelu", True, True),        # 2 x 9 score tiles, the last 16 columns
    ((192, 128), 1500, 1024, 4400, "gelu", True, True),     # 6 x 8 score tiles, 68.75 k-blocks
    ((256, 128), 2048, 784, 4112, "gelu", False, True),     # 8 x 7 score tiles, the last 16 columns
    ((192, 128), 1200, 1024, 4096, "quick_gelu", True, True),  # 5 row tiles
    ((256, 64), 1000, 1024, 4160, "quick_gelu", True, False),  # 4 x 16 score tiles, 65 k-blocks
    ((64, 64), 129, 1056, 1472, "quick_gelu", True, True),  # 17 score tiles, the last half empty
    ((256, 192), 2885, 1152, 4304, "gelu", True, True),     # 12 x 6 score tiles
    ((256, 128), 2048, 784, 2064, "gelu", False, True),     # 8 x 7 score tiles, the last 16 columns
    ((256, 192), 2049, 1152, 1600, "none", True, True),     # 9 x 6 score tiles
    ((128, 256), 3000, 1296, 528, "gelu", True, True),      # 12 x 6 score tiles, the last 16 columns
]


@pytest.mark.parametrize("columns,t,d,dh,act,resid,bias", LAYOUT_CASES,
                         ids=["%d-%d-%d" % c[1:4] for c in LAYOUT_CASES])
def test_mlp_layouts(columns, t, d, dh, act, resid, bias):
    assert columns == (_columns(t, dh, d, 0), _columns(t, d, dh, 1))
    test_mlp_outputs_and_records("%d-%d" % columns, t, d, dh, act, resid, bias)
    # a second call reproduces every bit: the row partials are merged in a fixed order
    altr = _alt()
    xp, w1, w2, b1, b2, r = _inputs(t, d, dh, seed=3, resid=resid, bias=bias)
    m = altr.Mlp(t, w1, w2, b1, b2, act=act)
    first = [v.clone() for v in (lambda o: (o.h, o.x_post, o.x, o.stats))(m.run(xp, r))]
    again = (lambda o: (o.h, o.x_post, o.x, o.stats))(m.run(xp, r))
    torch.cuda.synchronize()
    for u, v in zip(first, again):
        assert torch.equal(u.view(torch.int16), v.view(torch.int16))


def _project_direct(x, idx, cu_k, w, bias, seqlens):
    """tr_project_kept itself, which the binding's project_kept calls for few
    rows and for images above 16384 tokens."""
    from paper_2607_13500_gb300 import _lib
    from paper_2607_13500_gb300.api import _Tokens, _ptr, _stream
    tok = _Tokens(x, None, x, seqlens)
    z = torch.empty(cu_k[-1], w.shape[0], dtype=torch.bfloat16, device=x.device)
    err = torch.zeros(1, dtype=torch.int32, device=x.device)
    d_cu = torch.tensor(cu_k, dtype=torch.int32, device=x.device)
    _lib.check("tr_project_kept", _lib.load().tr_project_kept(
        tok.ref(), _ptr(d_cu), _ptr(idx), cu_k[-1], _ptr(w), _ptr(bias), w.shape[0], 0, _ptr(z), _ptr(err),
        _stream(x.device)))
    return z, err


@pytest.mark.parametrize("columns,d,d_out,k,n,b", [
    (64, 8208, 528, 40, 300, 3), (128, 4096, 2560, 200, 300, 3), (64, 784, 1296, 50, 300, 3), (128, 272, 528, 200, 300, 16),
    (64, 256, 272, 1025, 1300, 3), (192, 272, 528, 350, 400, 12), (256, 272, 1040, 1025, 1300, 3),
    (256, 784, 1040, 1025, 1300, 3)])
def test_project_layouts(columns, d, d_out, k, n, b):
    # every tile width: the dense projector within the GEMM tolerance of
    # float64, and the rows read by index bit for bit the same
    assert columns == _columns(b * k, d_out, d, 0) == _columns(b * k, d_out, d, 2)
    altr = _alt()
    g = torch.Generator(device="cuda").manual_seed(9)
    x = torch.randn(b * n, d, generator=g, device="cuda").to(torch.bfloat16)
    idx = torch.rand(b, n, generator=g, device="cuda").argsort(1)[:, :k].sort(1).values.to(torch.int32)
    w = (torch.randn(d_out, d, generator=g, device="cuda") / math.sqrt(d)).to(torch.bfloat16)
    bias = 0.05 * torch.randn(d_out, generator=g, device="cuda")
    y = torch.cat([x[i * n:(i + 1) * n][idx[i].long()] for i in range(b)]).contiguous()
    idx, cu_k = idx.reshape(-1).contiguous(), [i * k for i in range(b + 1)]
    z, err = altr.project(y, w, bias, act="gelu")
    zk, err_k = altr.project_kept(x, idx, cu_k, w, bias, act="gelu", seqlens=[n] * b)
    zd, err_d = _project_direct(x, idx, cu_k, w, bias, [n] * b)
    torch.cuda.synchronize()
    assert err.item() == 0 and err_k.item() == 0 and err_d.item() == 0
    assert torch.equal(z.view(torch.int16), zk.view(torch.int16))
    assert torch.equal(z.view(torch.int16), zd.view(torch.int16))
    v, mag = _gemm_ref(y, w, bias)
    _check_close(z, _sigma(v, "gelu"), mag, slope=1.13)


@pytest.mark.parametrize("d_out,copied", [(1008, False), (1024, True)])
def test_project_kept_of_many_rows_of_a_ragged_batch(d_out, copied, monkeypatch):
    # both routes on either side of the width from which the rows are copied
    # first: images of several sizes, one empty and one that keeps nothing,
    # and indices outside their images, which feed rows of zeros
    altr = _alt()
    from paper_2607_13500_gb300 import _lib
    lib, copies = _lib.load(), []
    gather = lib.tr_gather
    monkeypatch.setattr(lib, "tr_gather", lambda *a: copies.append(a) or gather(*a))
    seqlens, ks, d = [1500, 0, 2600, 7, 900], [1200, 0, 1900, 0, 200], 272
    g = torch.Generator(device="cuda").manual_seed(4)
    x = torch.randn(sum(seqlens), d, generator=g, device="cuda").to(torch.bfloat16)
    w = (torch.randn(d_out, d, generator=g, device="cuda") / math.sqrt(d)).to(torch.bfloat16)
    bias = 0.05 * torch.randn(d_out, generator=g, device="cuda")
    idx, rows, cu, off = [], [], [0], 0
    for n, k in zip(seqlens, ks):
        i = torch.randperm(max(n, 1), generator=g, device="cuda")[:k].sort().values
        idx.append(i)
        rows.append(off + i)
        off += n
        cu.append(cu[-1] + k)
    idx, rows = torch.cat(idx).to(torch.int32), torch.cat(rows)
    y = x[rows]
    for slot, bad in ((0, -1), (1199, 1500), (1200, 2600), (3099, 2 ** 31 - 1), (3100, -2 ** 31), (3299, 900)):
        idx[slot] = bad
        y[slot] = 0
    z, err = altr.project_kept(x, idx, cu, w, bias, act="gelu", seqlens=seqlens)
    assert bool(copies) == copied
    zd, err_d = _project_direct(x, idx, cu, w, bias, seqlens)
    zy, err_y = altr.project(y, w, bias, act="gelu")
    torch.cuda.synchronize()
    assert err.item() == 0 and err_d.item() == 0 and err_y.item() == 0
    assert torch.equal(z.view(torch.int16), zd.view(torch.int16))
    assert torch.equal(z.view(torch.int16), zy.view(torch.int16))


def test_project_kept_of_an_image_past_the_gather_limit():
    # more tokens in an image than tr_gather takes: the direct kernel
    altr = _alt()
    g = torch.Generator(device="cuda").manual_seed(2)
    n, d, d_out, k = 20000, 64, 96, 4000
    x = torch.randn(n, d, generator=g, device="cuda").to(torch.bfloat16)
    idx = torch.randperm(n, generator=g, device="cuda")[:k].sort().values.to(torch.int32)
    w = (torch.randn(d_out, d, generator=g, device="cuda") / 8).to(torch.bfloat16)
    z, err = altr.project_kept(x, idx, [0, k], w, act="none", seqlens=[n])
    zd, err_d = altr.project(x[idx.long()].contiguous(), w, act="none")
    torch.cuda.synchronize()
    assert err.item() == 0 and err_d.item() == 0 and torch.equal(z.view(torch.int16), zd.view(torch.int16))


@pytest.mark.parametrize("t,d,dh", [(2048, 1024, 4096), (192, 1024, 256), (1, 272, 512)])
def test_mlp_score_with_a_smaller_workspace(t, d, dh):
    # what 256-column tiles need, less than the layout chosen otherwise, is
    # enough; a block fewer is refused
    altr = _alt()
    xp, w1, w2, b1, b2, r = _inputs(t, d, dh, seed=4)
    m = altr.Mlp(t, w1, w2, b1, b2, act="gelu", scores=True)
    m.run(xp, r)
    least = -(-t // 128) * -(-d // 256) * 10240
    assert m._ws_bytes > least
    m._ws = torch.full((least + 4096,), 0xff, dtype=torch.uint8, device="cuda")
    m._ws_bytes = least
    o = m.run(xp, r)
    v, mag = _gemm_ref(o.h, w2, b2)
    _check_close(o.x_post, v, mag)
    assert o.error.item() == 0 and bool((m._ws[least:] == 0xff).all())
    st, h2, s = altr.score(o.x, xp, o.x_post)
    assert torch.allclose(o.stats[:, :4], st[:, :4], rtol=2.0 ** -21, atol=0)
    assert torch.allclose(o.h2, h2, rtol=1e-5, atol=2e-6) and torch.allclose(o.s, s, rtol=0, atol=1e-5)
    m._ws_bytes = least - 256
    with pytest.raises(Exception, match="tr_mlp_score"):
        m.run(xp, r)


@pytest.mark.parametrize("t,d,dh", [(576, 1024, 4096), (48, 1024, 4096), (129, 1056, 1472), (1, 256, 6144)])
def test_rows_do_not_depend_on_the_batch(t, d, dh):
    # An image's rows alone, in a batch whose GEMMs are laid out differently,
    # and with the least scratch: K is summed in one order, so H, x'' and x are
    # the same bit for bit, and so is the projector's z.  The records' sums are
    # grouped by the tile columns: the same to their fp32 rounding, and the
    # certified selection the same.
    altr = _alt()
    most = 12 * t if t > 1 else 3000
    xp, w1, w2, b1, b2, r = _inputs(most, d, dh, seed=12)
    m = altr.Mlp(most, w1, w2, b1, b2, act="quick_gelu")
    whole = m.run(xp, r)
    alone = altr.Mlp(t, w1, w2, b1, b2, act="quick_gelu")
    rows = [(a.clone(), b[:t].clone()) for o in [alone.run(xp[:t].contiguous(), r[:t].contiguous())]
            for a, b in ((o.h, whole.h), (o.x_post, whole.x_post), (o.x, whole.x), (o.stats, whole.stats))]
    alone._ws_bytes = -(-t // 128) * -(-d // 256) * 10240
    least = alone.run(xp[:t].contiguous(), r[:t].contiguous())
    torch.cuda.synchronize()
    for a, b in rows[:3]:
        assert torch.equal(a.view(torch.int16), b.view(torch.int16))
    for a, b in zip((least.x_post, least.x), (rows[1][0], rows[2][0])):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16))
    sa, sb = rows[3]
    assert torch.allclose(sa[:, :4], sb[:, :4], rtol=2.0 ** -23, atol=0)
    z, _ = altr.project(whole.x, w1, b1)
    za, _ = altr.project(whole.x[:t].contiguous(), w1, b1)
    zk, _ = altr.project_kept(whole.x, torch.arange(t, dtype=torch.int32, device="cuda"), [0, t], w1, b1)
    assert torch.equal(z[:t].view(torch.int16), za.view(torch.int16))
    assert torch.equal(z[:t].view(torch.int16), zk.view(torch.int16))
