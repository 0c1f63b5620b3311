"""The K split of a CTA-pair launch's last wave (csrc/gemm.cu, split_wave):
two to four (precise: eight) parts per tile, ragged row tiles (an odd last
tile, tiles of one row, empty sequences), the residual epilogues, and counters
left zero for the next launch, against the unpaired tile kernel on the same
operands."""
import numpy as np
import pytest
import torch

import synth
from synth.configs import ModelShape
from tests._util import rel_err

pytestmark = pytest.mark.gpu

# (d_model, d_ff): the down projection's 6, 24 and 15 tiles (600 rows) in 4, 2
# and 3 parts; the last K ends inside a barrier stage and a k-block
SIZES = [(512, 16384), (2048, 8192), (1280, 10784)]


@pytest.fixture(scope="module")
def pkg():
    import paper_2607_27600_gb300 as p
    p.load_library()
    return p


def _shape(d, f, layers=1):
    return ModelShape(layers, d, 16, 8, 128 if d > 512 else 64, f, 700, 1e4, 1e-5)


@pytest.mark.parametrize("d,f", SIZES)
@pytest.mark.parametrize("mode", ["bf16", "f16", "precise", "logprob", "full"])
@pytest.mark.parametrize("lens,cap", [([600], 600), ([513, 0, 1, 129], 520)])
def test_scores_equal_the_tile_kernel(pkg, monkeypatch, d, f, mode, lens, cap):
    """Same operands, fp32 sums in another order (1e-6 relative) and 16-bit
    activations whose rounding falls the other way (2^-9 bf16, 2^-12 fp16, of
    single terms): a tenth of each mode's own error.  full: over two layers the
    first roundings that differ move every later value a little, so the second
    layer's fall independently; with [hi | lo] activations (2^-17 each) ten
    products' independent roundings give sqrt(10) 2^-17 / sqrt(3), at 5 sigma
    over the rows 7e-5: stated 2e-4."""
    from paper_2607_27600_gb300 import cc
    shape = _shape(d, f, 2 if mode == "full" else 1)
    w = synth.model_weights(shape, 5, device="cuda", with_kv_proj=True)
    c = synth.synthetic_cache(shape, lens, cap, 6, device="cuda")
    flag = {"f16": cc.SCORE_F16, "precise": cc.SCORE_PRECISE, "full": cc.SCORE_PRECISE}.get(mode, 0)
    base = cc.SCORE_LOGPROB if mode == "logprob" else cc.SCORE_LOGIT
    if mode == "f16":
        w = cc.f16_weights(w)
    fn = cc.cc_score_full if mode == "full" else cc.cc_score_layer
    ws = cc.alloc_workspace(cc.cc_score_workspace_size(shape, len(lens), cap, base | flag))
    out = []
    for env in ("2", "2", "0"):
        monkeypatch.setenv("CC_GEMM_PAIRS", env)
        s = torch.full((len(lens), cap), float("nan"), dtype=torch.float32, device="cuda")
        fn(shape, pkg.Weights(w), pkg.Cache(c), base | flag, s, ws)
        assert cc.cc_get_status() == cc.CC_OK
        out.append(s.cpu().numpy())
    got, again, ref = out
    assert np.array_equal(got, again)   # a fixed order of sums
    tol = {"f16": 1e-3, "precise": 1e-4, "full": 2e-4}.get(mode, 5e-3)
    for b, n in enumerate(lens):
        fin = np.isfinite(ref[b])
        assert np.array_equal(fin, np.isfinite(got[b])) and fin.sum() == max(0, n - 1)
        if n > 1:
            assert rel_err(got[b, :n], ref[b, :n]) < tol, b


@pytest.mark.parametrize("d,f", SIZES[1:])
def test_appends_equal_the_tile_kernel(pkg, monkeypatch, d, f):
    """K/V rows of a packed chunk (fused projections where the widths allow):
    bf16, 2^-8 per rounding that falls the other way, 4e-2 of the largest over
    two layers."""
    from paper_2607_27600_gb300 import cc
    shape, lens, counts, cap = _shape(d, f, 2), [100, 0, 7], [500, 129, 12], 700
    w = synth.model_weights(shape, 9, device="cuda", with_kv_proj=True)
    toks = synth.tokens((3, max(counts)), shape.vocab, 3).cuda()
    cnt = torch.tensor(counts, dtype=torch.int32, device="cuda")
    out = []
    for env in ("2", "0"):
        monkeypatch.setenv("CC_GEMM_PAIRS", env)
        c = synth.synthetic_cache(shape, lens, cap, 10, device="cuda")
        ws = cc.alloc_workspace(cc.cc_append_workspace_size(shape, 3, cap))
        cc.cc_append_chunk(shape, pkg.Weights(w), pkg.Cache(c), toks, None, cnt, max(counts), ws)
        assert cc.cc_get_status() == cc.CC_OK
        out.append(c)
    for x, y in zip(out[0]["k"] + out[0]["v"], out[1]["k"] + out[1]["v"]):
        for b in range(3):
            r = slice(lens[b], lens[b] + counts[b])
            assert torch.equal(x[b, :lens[b]], y[b, :lens[b]])
            assert (x[b, r].float() - y[b, r].float()).abs().max() <= 4e-2 * y[b, r].float().abs().max()
