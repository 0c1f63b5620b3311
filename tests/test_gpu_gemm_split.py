"""The K split of a CTA-pair launch's last wave (csrc/gemm.cu, split_wave), which
the down projections of appends take: two to four parts per tile, ragged row
tiles (an odd last tile, tiles of one row, empty sequences), counters left zero
for the next launch, against the unpaired tile kernel on the same operands."""
import pytest
import torch

import synth
from synth.configs import ModelShape

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2607_27600_gb300 as p
    p.load_library()
    return p


# (d_model, d_ff): the down projection's 6, 24 and 15 tiles (600 rows) in 4, 2
# and 3 parts; the last K ends inside a barrier stage and a k-block
@pytest.mark.parametrize("d,f", [(512, 16384), (2048, 8192), (1280, 10784)])
@pytest.mark.parametrize("lens,counts", [([100], [600]), ([100, 0, 7, 3], [500, 129, 12, 0]),
                                         ([0, 9], [513, 1])])
def test_appends_equal_the_tile_kernel(pkg, monkeypatch, d, f, lens, counts):
    """H^(L-1) and K/V rows of a packed chunk through three layers: bf16, 2^-8 per
    rounding that falls the other way, 4e-2 of the largest over the layers; two
    runs give the same bits (a fixed order of sums)."""
    from paper_2607_27600_gb300 import cc
    cap = 720
    shape = ModelShape(3, d, 16, 8, 128 if d > 512 else 64, f, 700, 1e4, 1e-5)
    w = synth.model_weights(shape, 9, device="cuda", with_kv_proj=True)
    toks = synth.tokens((len(lens), max(counts)), shape.vocab, 3).cuda()
    cnt = torch.tensor(counts, dtype=torch.int32, device="cuda")
    ws = cc.alloc_workspace(cc.cc_append_workspace_size(shape, len(lens), cap))
    out = []
    for env in ("2", "2", "0"):
        monkeypatch.setenv("CC_GEMM_PAIRS", env)
        c = synth.synthetic_cache(shape, lens, cap, 10, device="cuda")
        cc.cc_append_chunk(shape, pkg.Weights(w), pkg.Cache(c), toks, None, cnt, max(counts), ws)
        assert cc.cc_get_status() == cc.CC_OK
        out.append(c["k"] + c["v"] + [c["h_last"]])
    for x, again, y in zip(*out):
        assert torch.equal(x, again)
        for b, (n, m) in enumerate(zip(lens, counts)):
            assert torch.equal(x[b, :n], y[b, :n]) and torch.equal(x[b, n + m:], y[b, n + m:])
            if m:
                a, r = x[b, n:n + m].float(), y[b, n:n + m].float()
                assert (a - r).abs().max() <= 4e-2 * r.abs().max(), b
