"""The decode attention kernel (csrc/attn.cu, attn_decode_kernel and its
combine) at the edges of its 64-key chunks, splits and pages: key counts 1 to
700, one split and many, 1 to 8 query heads per KV head, both head dims, the
K/V layouts, and a batch past the 64 sequences whose activations travel as
bf16 pairs.  Checked on H^(L-1), the residual stream after the first layer,
against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from synth.configs import ModelShape
from tests._util import to_device, to_np

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 62, 63, 64, 65, 127, 128, 191, 447, 699]   # (+ the step's own key)


@pytest.fixture(scope="module")
def pkg():
    import paper_2607_27600_gb300 as p
    p.load_library()
    return p


@pytest.mark.parametrize("dh,hkv,g,lens,cap,layout", [
    (64, 2, 1, EDGES, 704, "slot"), (64, 1, 3, EDGES, 704, "head"), (64, 2, 8, EDGES, 768, "paged"),
    (128, 2, 1, EDGES, 768, "paged"), (128, 1, 5, EDGES, 704, "slot"), (128, 2, 8, EDGES, 704, "head"),
    (128, 1, 2, [0, 1, 30, 62, 63], 64, "slot"),              # one split
    (64, 2, 2, [(7 * i) % 140 for i in range(70)], 140, "slot"),   # single bf16 activations
])
def test_step_matches_oracle(pkg, dh, hkv, g, lens, cap, layout):
    """The new K/V rows and the record are bf16 (2^-9 each, of values up to the
    row's largest) and pass through one O projection and MLP: 2^-7 of the row's
    largest; single bf16 activations add five roundings of 2^-9: 2^-6."""
    import bench
    from paper_2607_27600_gb300 import cc
    shape = ModelShape(2, 256, hkv * g, hkv, dh, 512, 300, 1e4, 1e-5)
    b = len(lens)
    w_np = to_np(synth.model_weights(shape, 3, with_kv_proj=True))
    c_np = to_np(synth.synthetic_cache(shape, lens, cap, 4))
    c = to_device(c_np)
    if layout == "paged":
        bench.to_paged_cache(c, 128, 11)
    elif layout == "head":
        for key in ("k", "v"):
            c[key] = [x.permute(0, 2, 1, 3).contiguous() for x in c[key]]
        c["kv_layout"] = 1
    tok = np.random.default_rng(5).integers(0, shape.vocab, size=b)
    nxt = torch.empty(b, dtype=torch.int32, device="cuda")
    ws = cc.alloc_workspace(cc.cc_decode_workspace_size(shape, b, cap))
    cc.cc_decode_step(shape, pkg.Weights(to_device(w_np)), pkg.Cache(c),
                      torch.from_numpy(tok.astype(np.int32)).cuda(), nxt, None, ws)
    assert cc.cc_get_status() == cc.CC_OK
    cn = {k: ([np.asarray(x, np.float64).copy() for x in v] if isinstance(v, list) else
              np.asarray(v).copy()) for k, v in c_np.items()}
    oracle.decode_step(shape, w_np, cn, tok)
    got, tol = c["h_last"].float().cpu().numpy(), 2.0 ** (-6 if b > 64 else -7)
    for i, n in enumerate(lens):
        want = cn["h_last"][i, n]
        assert np.abs(got[i, n] - want).max() <= tol * np.abs(want).max(), (i, n)
