"""The few-row GEMM (csrc/fewrow.cu), and the choice between it and the tile kernel
below two waves of 128 x 256 tiles.  Row counts at the edges of its row groups (16 to 256) and 16-row
blocks, K ranges cut over 1 to 8 CTAs of a cluster, head dims 64 and 128 and
column counts that end inside a 128-column tile, against the oracle; and the
general tile kernel (CC_GEMM_PAIRS=0) over every form both take."""
import numpy as np
import pytest
import torch

import oracle
import synth
from synth.configs import ModelShape
from tests._util import causal_cache, rel_err, to_device, to_np

pytestmark = pytest.mark.gpu

# d_ff 4160 = 65 k-blocks of the down projection over 5 column tiles (the last
# 32 wide): cut over 8 CTAs; q_dim 192 and 640: a last tile half past N, and whole
SHAPES = {64: ModelShape(2, 544, 3, 1, 64, 4160, 700, 1e4, 1e-5, qkv_bias=True),
          128: ModelShape(2, 544, 5, 1, 128, 4160, 700, 1e4, 1e-6)}


@pytest.fixture(scope="module")
def pkg():
    import paper_2607_27600_gb300 as p
    p.load_library()
    return p


def _score(pkg, shape, w, c, mode, full):
    from paper_2607_27600_gb300 import cc
    b, cap = c["tokens"].shape
    ws = cc.alloc_workspace(cc.cc_score_workspace_size(shape, b, cap, mode))
    s = torch.full((b, cap), float("nan"), dtype=torch.float32, device="cuda")
    (cc.cc_score_full if full else cc.cc_score_layer)(shape, pkg.Weights(w), pkg.Cache(c), mode, s, ws)
    got = s.cpu().numpy()
    assert cc.cc_get_status() == cc.CC_OK
    return got


@pytest.mark.parametrize("dh", [64, 128])
@pytest.mark.parametrize("lens,cap", [([1], 1), ([15], 16), ([17], 17), ([129], 160), ([255], 257),
                                      ([300, 2, 16, 0], 300), ([530], 600)])
def test_scores_at_the_edges_of_groups_and_blocks(pkg, dh, lens, cap):
    """Precise operands (every product twice as long: [hi | lo] rows): the
    stated 2e-3 of that mode on every row of the fast pass."""
    from paper_2607_27600_gb300 import cc
    shape = SHAPES[dh]
    w_np = to_np(synth.model_weights(shape, 5, with_kv_proj=True))
    c_np = causal_cache(shape, w_np, lens, cap, 6)
    got = _score(pkg, shape, to_device(w_np), to_device(c_np), cc.SCORE_LOGIT | cc.SCORE_PRECISE, False)
    want = oracle.score_layer(shape, w_np, c_np)
    for b, n in enumerate(lens):
        if n > 1:
            assert rel_err(got[b, :n], want[b, :n]) < 2e-3, (b, n)
        if n > 0:
            assert got[b, n - 1] == np.inf
        assert np.all(got[b, n:] == -np.inf)


@pytest.mark.parametrize("dh", [64, 128])
@pytest.mark.parametrize("mode", ["bf16", "f16", "precise"])
@pytest.mark.parametrize("full", [False, True])
def test_scores_equal_the_tile_kernel(pkg, monkeypatch, dh, mode, full):
    """Both kernels multiply the same operands and sum in fp32, so they differ
    by summation order: 1e-6 relative per sum, and by what one rounding of a
    16-bit activation that falls the other way moves (2^-9 bf16, 2^-12 fp16, of
    one of 544 terms); bounded here by a tenth of the mode's own error."""
    from paper_2607_27600_gb300 import cc
    shape, lens, cap = SHAPES[dh], [300, 33, 129], 320
    flag = {"bf16": 0, "f16": cc.SCORE_F16, "precise": cc.SCORE_PRECISE}[mode]
    w_np = to_np(synth.model_weights(shape, 7, with_kv_proj=True))
    w, c = to_device(w_np), to_device(causal_cache(shape, w_np, lens, cap, 8))
    if mode == "f16":
        w = cc.f16_weights(w)
    got = _score(pkg, shape, w, c, cc.SCORE_LOGIT | flag, full)
    monkeypatch.setenv("CC_GEMM_PAIRS", "0")
    ref = _score(pkg, shape, w, c, cc.SCORE_LOGIT | flag, full)
    tol = {"bf16": 5e-3, "f16": 1e-3, "precise": 1e-4}[mode]
    for b, n in enumerate(lens):
        f = np.isfinite(ref[b, :n])
        assert np.array_equal(f, np.isfinite(got[b, :n]))
        assert rel_err(got[b, :n], ref[b, :n]) < tol, b


@pytest.mark.parametrize("d,f,n", [(2048, 16384, 129), (2048, 16384, 250), (2048, 16384, 256),
                                   (3424, 12288, 250), (3424, 12288, 257), (3424, 12288, 511)])
def test_wide_layer_equals_the_tile_kernel(pkg, monkeypatch, d, f, n):
    """One gate/up group of up to 256 rows over a single accumulator pair, and
    a down projection whose partial rows are exchanged in two rounds: d_model
    2048 over 8 CTAs, 3424 (27 column tiles, the last partial) as CTA pairs, the
    last without its second tile, over 4 splits, and two groups over 2.  fp16
    operands: the sums' order and roundings that fall the other way move a row
    by 2^-12 of single terms (bf16, 2^-9: 6e-3 of the largest of 511 rows, so
    8e-4 here): the 1e-3 of the test above."""
    from paper_2607_27600_gb300 import cc
    shape = ModelShape(1, d, 4, 2, 128, f, 700, 1e4, 1e-5)
    w = cc.f16_weights(synth.model_weights(shape, 5, device="cuda", with_kv_proj=True))
    c = synth.synthetic_cache(shape, [n], n + 4 - n % 4, 6, device="cuda")
    mode = cc.SCORE_LOGIT | cc.SCORE_F16
    got = _score(pkg, shape, w, c, mode, False)
    monkeypatch.setenv("CC_GEMM_PAIRS", "0")
    ref = _score(pkg, shape, w, c, mode, False)
    fin = np.isfinite(ref[0])
    assert np.array_equal(fin, np.isfinite(got[0])) and fin.sum() == n - 1
    assert rel_err(got[0, :n], ref[0, :n]) < 1e-3


@pytest.mark.parametrize("dh", [64, 128])
@pytest.mark.parametrize("layout", ["slot", "head", "paged", "e4m3"])
@pytest.mark.parametrize("counts", [[1, 0, 1], [37, 128, 5]])
def test_appends_equal_the_tile_kernel(pkg, monkeypatch, dh, layout, counts):
    """Appended K/V rows, H^(L-1), tokens and positions in every cache layout,
    and nothing written outside the appended slots.  bf16 rows: 2^-8 of a value
    per rounding that falls the other way (over two layers: 4e-2 of a row's
    largest); e4m3: one code step (2^-3)."""
    import bench
    from paper_2607_27600_gb300 import cc
    shape, lens, cap = SHAPES[dh], [200, 130, 0], 512
    w_np = to_np(synth.model_weights(shape, 9, with_kv_proj=True))
    c_np = causal_cache(shape, w_np, lens, cap, 10)
    w = pkg.Weights(to_device(w_np))
    toks = synth.tokens((3, max(counts)), shape.vocab, 3).cuda()
    cnt = torch.tensor(counts, dtype=torch.int32, device="cuda")
    out = []
    for env in (None, "0"):
        if env:
            monkeypatch.setenv("CC_GEMM_PAIRS", env)
        c = to_device(c_np)
        if layout == "e4m3":
            bench.to_e4m3_cache(c)
        elif layout == "paged":
            bench.to_paged_cache(c, 128, 11)
        elif layout == "head":
            for key in ("k", "v"):
                c[key] = [x.permute(0, 2, 1, 3).contiguous() for x in c[key]]
            c["kv_layout"] = 1
        before = [x.clone() for x in c["k"] + c["v"]]
        ws = cc.alloc_workspace(cc.cc_append_workspace_size(shape, 3, cap))
        cc.cc_append_chunk(shape, w, pkg.Cache(c), toks, None, cnt, max(counts), ws)
        assert cc.cc_get_status() == cc.CC_OK
        out.append((c, before))
    (c0, b0), (c1, _) = out
    assert torch.equal(c0["seq_len"], c1["seq_len"]) and torch.equal(c0["tokens"], c1["tokens"])
    assert torch.equal(c0["pos"], c1["pos"])

    def val(x):
        return (x.view(torch.float8_e4m3fn) if layout == "e4m3" else x).float()

    def changed(x, b):   # per head_dim vector
        return (x.view(torch.uint8) != b.view(torch.uint8)).reshape(*x.shape[:-1], -1).any(-1)

    for x, y, b in zip(c0["k"] + c0["v"], c1["k"] + c1["v"], b0):
        rows = changed(y, b)
        assert torch.equal(changed(x, b), rows)
        assert int(rows.sum()) == sum(counts) * shape.n_kv_heads
        tol = 0.13 if layout == "e4m3" else 4e-2
        assert (val(x) - val(y)).abs().max() <= tol * val(y)[rows].abs().max()
    assert (c0["h_last"].float() - c1["h_last"].float()).abs().max() <= 4e-2 * c1["h_last"].float().abs().max()


@pytest.mark.parametrize("lens,counts", [([0], [257]), ([64], [520]), ([0], [600]), ([300], [1100]),
                                         ([0, 5, 100], [700, 40, 1]), ([0, 0], [640, 639])])
def test_appends_of_every_form_equal_the_tile_kernel(pkg, monkeypatch, lens, counts):
    """Row counts past one group, where a product goes to the few-row kernel, to
    single CTAs of 128 or 256 columns or to CTA pairs: against single CTAs for
    all of them.  bf16 rows through two layers: 4e-2 of the largest, as above."""
    from paper_2607_27600_gb300 import cc
    shape, cap = ModelShape(2, 2048, 16, 8, 128, 6144, 700, 1e4, 1e-5), 1408
    w = synth.model_weights(shape, 9, device="cuda", with_kv_proj=True)
    toks = synth.tokens((len(lens), max(counts)), shape.vocab, 3).cuda()
    cnt = torch.tensor(counts, dtype=torch.int32, device="cuda")
    ws = cc.alloc_workspace(cc.cc_append_workspace_size(shape, len(lens), cap))
    out = []
    for env in (None, None, "0"):
        if env:
            monkeypatch.setenv("CC_GEMM_PAIRS", env)
        c = synth.synthetic_cache(shape, lens, cap, 10, device="cuda")
        cc.cc_append_chunk(shape, pkg.Weights(w), pkg.Cache(c), toks, None, cnt, max(counts), ws)
        assert cc.cc_get_status() == cc.CC_OK
        out.append(c["k"] + c["v"] + [c["h_last"]])
    for x, again, y in zip(*out):
        assert torch.equal(x, again)
        for b, (n, m) in enumerate(zip(lens, counts)):
            assert torch.equal(x[b, :n], y[b, :n]) and torch.equal(x[b, n + m:], y[b, n + m:])
            a, r = x[b, n:n + m].float(), y[b, n:n + m].float()
            assert (a - r).abs().max() <= 4e-2 * r.abs().max(), b
