"""The weight-streaming GEMVs of one to four decode rows (csrc/gemv.cu): K of one
to many 256-element boxes with and without a remainder, column counts that end
inside a group of 16 or a box of 8, every cache layout, biases, rows with and
without a token, and launches that mix them with the few-row GEMM."""
import numpy as np
import pytest
import torch

import oracle
import synth
from synth.configs import ModelShape
from tests._util import causal_cache, rel_err, to_device, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2607_27600_gb300 as p
    p.load_library()
    return p


def _launches(cc):
    """Launches per kernel kind since timing was enabled."""
    return {k: n for k, (n, _) in cc.cc_timing_collect().items()}


# d_model and d_ff: 256 exactly, 288 (a box and 32), 608, 2592 (ten boxes and 32)
SHAPES = {
    "small": ModelShape(3, 288, 8, 2, 64, 608, 300, 1e4, 1e-5, qkv_bias=True),
    "head128": ModelShape(2, 512, 5, 1, 128, 2592, 300, 1e4, 1e-6),
    # more query heads per KV head than the decode attention takes: single bf16 rows
    "g12": ModelShape(2, 256, 12, 1, 64, 320, 300, 1e4, 1e-5),
    "g1": ModelShape(2, 256, 4, 4, 64, 256, 300, 1e4, 1e-5, qkv_bias=True),
}


@pytest.mark.parametrize("name", list(SHAPES))
@pytest.mark.parametrize("layout", ["slot", "head", "paged", "e4m3"])
@pytest.mark.parametrize("lens", [[70], [0, 64], [5, 127, 63], [1, 200, 33, 0]])
def test_steps_match_the_oracle(pkg, name, layout, lens):
    """Two steps, K/V rows of every layer, H^(L-1) and the logits.  The rows
    written are bf16 (2^-9 of a value) and feed two to three layers of pairs and
    fp32 sums: 2^-6 of a row's largest (e4m3: a code step, 2^-3)."""
    import bench
    from paper_2607_27600_gb300 import cc
    from tests.test_gpu_fp8 import fp8_views
    shape, cap, b = SHAPES[name], 256, len(lens)
    w_np = to_np(synth.model_weights(shape, 3, with_kv_proj=True))
    c_np = causal_cache(shape, w_np, lens, cap, 4)
    if layout == "e4m3":
        on, c = fp8_views(c_np)
    else:
        on, c = c_np, to_device(c_np)
    if layout == "paged":
        bench.to_paged_cache(c, 128, 11)
    elif layout == "head":
        for key in ("k", "v"):
            c[key] = [x.permute(0, 2, 1, 3).contiguous() for x in c[key]]
        c["kv_layout"] = 1
    on = {k: ([np.asarray(x, np.float64).copy() for x in v] if isinstance(v, list) and k in "kv" else
              v if isinstance(v, list) else np.asarray(v).copy()) for k, v in on.items()}
    weights, cache = pkg.Weights(to_device(w_np)), pkg.Cache(c)
    ws = cc.alloc_workspace(cc.cc_decode_workspace_size(shape, b, cap))
    nxt = torch.empty(b, dtype=torch.int32, device="cuda")
    best = torch.empty(b, dtype=torch.float32, device="cuda")
    tok = np.random.default_rng(5).integers(0, shape.vocab, size=b)
    tol = 2.0 ** (-3 if layout == "e4m3" else -6)
    for step in range(2):
        cc.cc_timing_enable(True)
        cc.cc_decode_step(shape, weights, cache, torch.from_numpy(tok.astype(np.int32)).cuda(), nxt, best, ws)
        kinds = _launches(cc)
        cc.cc_timing_enable(False)
        assert cc.cc_get_status() == cc.CC_OK
        # q, k and v in one launch, whatever their columns: the GEMV ran
        assert kinds.get("gemm_qkv", 0) == shape.n_layers and not kinds.get("gemm_kv", 0)
        o_next, _, o_logits = oracle.decode_step(shape, w_np, on, tok)
        for i, n0 in enumerate(lens):
            n = n0 + step
            h = c["h_last"][i, n].float().cpu().numpy()
            assert np.abs(h - on["h_last"][i, n]).max() <= tol * np.abs(on["h_last"][i, n]).max()
            for key in ("k", "v"):
                for l in range(shape.n_layers):
                    x = bench.logical_kv(c, key, l)[i, n]
                    if layout == "e4m3":
                        x = x.view(torch.float8_e4m3fn).float() * on["kv_scale"][l]["kv".index(key)]
                    want = np.asarray(on[key][l][i, n], np.float64)
                    assert np.abs(x.float().cpu().numpy() - want).max() <= tol * np.abs(want).max(), (key, l, i)
            top = np.sort(o_logits[i])[-1]
            assert abs(float(best[i]) - top) <= 2e-2 * np.abs(o_logits[i]).max()
        tok = o_next
    assert c["seq_len"].tolist() == [n + 2 for n in lens]


def test_a_full_sequence_appends_nothing(pkg):
    """The second of three sequences has no room: reported, its token -1, no slot
    of it written, and the others' bits those of a batch without it."""
    from paper_2607_27600_gb300 import cc
    shape, cap = SHAPES["small"], 64
    w = to_device(to_np(synth.model_weights(shape, 3, with_kv_proj=True)))
    tok = torch.tensor([3, 5, 9], dtype=torch.int32, device="cuda")
    out = []
    for keep, lens in (([0, 1, 2], [20, 64, 7]), ([0, 2], [20, 7])):
        full = synth.synthetic_cache(shape, [20, 64, 7], cap, 4, device="cuda")
        c = {k: [x[keep].contiguous() for x in v] if isinstance(v, list) else v[keep].contiguous()
             for k, v in full.items()}
        before = [x.clone() for x in c["k"] + c["v"]]
        b = len(keep)
        nxt = torch.empty(b, dtype=torch.int32, device="cuda")
        best = torch.empty(b, dtype=torch.float32, device="cuda")
        ws = cc.alloc_workspace(cc.cc_decode_workspace_size(shape, b, cap))
        cc.cc_decode_step(shape, pkg.Weights(w), pkg.Cache(c), tok[keep].contiguous(), nxt, best, ws)
        assert cc.cc_get_status() == (cc.CC_ERR_DEVICE_ARG if b == 3 else cc.CC_OK)
        out.append((c, before, nxt.tolist(), best.tolist()))
    (c3, b3, n3, f3), (c2, _, n2, f2) = out
    assert n3[1] == -1 and [n3[0], n3[2]] == n2 and [f3[0], f3[2]] == f2
    assert c3["seq_len"].tolist() == [21, 64, 8]
    for x, y in zip(c3["k"] + c3["v"], b3):
        assert torch.equal(x[1], y[1])
    for x, y in zip(c3["k"] + c3["v"] + [c3["h_last"]], c2["k"] + c2["v"] + [c2["h_last"]]):
        assert torch.equal(x[[0, 2]], y)


@pytest.mark.parametrize("d,f,batch", [(4096, 14336, 1), (3584, 18944, 1), (3584, 18944, 2), (2048, 8192, 4)])
def test_layers_mix_with_the_few_row_gemm(pkg, monkeypatch, d, f, batch):
    """Shapes whose products divide between the two kernels, the norms' sums
    passing from one to the other: against the tile kernel for all of them, whose
    activations are single bf16 rows (five roundings of 2^-9 over two layers)."""
    from paper_2607_27600_gb300 import cc
    shape, cap = ModelShape(2, d, d // 128, 4, 128, f, 1000, 5e5, 1e-5), 512
    w = synth.model_weights(shape, 9, device="cuda", with_kv_proj=True)
    lens = [300 + 7 * i for i in range(batch)]
    tok = synth.tokens((batch,), shape.vocab, 3).cuda().to(torch.int32)
    out = []
    for env in (None, None, "0"):
        if env:
            monkeypatch.setenv("CC_GEMM_PAIRS", env)
        c = synth.synthetic_cache(shape, lens, cap, 10, device="cuda")
        nxt = torch.empty(batch, dtype=torch.int32, device="cuda")
        best = torch.empty(batch, dtype=torch.float32, device="cuda")
        ws = cc.alloc_workspace(cc.cc_decode_workspace_size(shape, batch, cap))
        cc.cc_decode_step(shape, pkg.Weights(w), pkg.Cache(c), tok, nxt, best, ws)
        assert cc.cc_get_status() == cc.CC_OK
        out.append(c["k"] + c["v"] + [c["h_last"], best])
    for x, again, y in zip(*out):
        assert torch.equal(x, again)
        for i, n in enumerate(lens):
            a, r = (x[i, n], y[i, n]) if x.dim() > 1 else (x[i], y[i])
            assert (a.float() - r.float()).abs().max() <= 2e-2 * r.float().abs().max(), i
