"""The decode attention kernel (csrc/attn.cu, attn_decode_kernel and its
combine): key counts 1 to 700 at the edges of 64-key chunks and pages, one split
and many of one chunk, splits of several chunks, 1 to 8 query heads per KV head,
both head dims, the K/V layouts and types, what it reports and what NaN and
infinity do; and decode batches around the sizes at which the activations'
bf16 pairs change layout (16, 32) and end (64).  Checked on H^(L-1), the residual
stream after the first layer, against the oracle."""
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


def keys_per_split(shape, lens, cap):
    """Keys of a split as the kernel plans them (csrc/attn.cu, dec_split_keys)
    for the longest of sequences of `lens` keys."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    units = len(lens) * shape.n_kv_heads
    ctas = max(sms, 3 * sms - units // 2)
    splits = max(1, min(128, -(-cap // 64), 160 * 256 // 8 // units, 4 * ctas // units))
    even = int(sum(lens) * shape.n_kv_heads / ctas)
    return -(-max(even, -(-max(lens) // splits)) // 64) * 64


def decode(pkg, shape, w, c):
    from paper_2607_27600_gb300 import cc
    b, cap = c["tokens"].shape
    nxt = torch.empty(b, dtype=torch.int32, device="cuda")
    best = torch.empty(b, dtype=torch.float32, device="cuda")
    ws = cc.alloc_workspace(cc.cc_decode_workspace_size(shape, b, cap))
    tok = np.random.default_rng(5).integers(0, shape.vocab, size=b)
    cc.cc_decode_step(shape, pkg.Weights(w), pkg.Cache(c),
                      torch.from_numpy(tok.astype(np.int32)).cuda(), nxt, best, ws)
    return cc.cc_get_status(), tok, nxt.cpu().numpy(), best.cpu().numpy()


@pytest.mark.parametrize("kv", ["bf16", "e4m3"])
@pytest.mark.parametrize("entry", [1 << 20, -1])
def test_bad_page_inside_a_split_is_reported(pkg, kv, entry):
    """A block-table entry outside the pool whose slots start no split: its
    keys are skipped and CC_ERR_DEVICE_ARG recorded; the other sequences'
    tokens and logits keep their bits and the context stays usable."""
    import bench
    from paper_2607_27600_gb300 import cc
    from tests.test_gpu_fp8 import fp8_views
    shape = ModelShape(2, 128, 4, 1, 64, 256, 300, 1e4, 1e-5)
    lens, cap = [3900 + i for i in range(32)], 4096
    per = keys_per_split(shape, [n + 1 for n in lens], cap)
    page = next(i for i in range(1, 20) if (128 * i) % per >= 64 and (128 * i) // per == (128 * i + 127) // per)
    w = to_device(to_np(synth.model_weights(shape, 3, with_kv_proj=True)))
    c_np = to_np(synth.synthetic_cache(shape, lens, cap, 4))
    good = bench.to_paged_cache(fp8_views(c_np)[1] if kv == "e4m3" else to_device(c_np), 128, 11)
    bad = {k: v.clone() if isinstance(v, torch.Tensor) else v for k, v in good.items()}
    bad.update({k: [x.clone() for x in good[k]] for k in ("k", "v")})
    bad["block_table"][7, page] = entry
    status, _, nxt, best = decode(pkg, shape, w, good)
    assert status == cc.CC_OK
    bad_status, _, bad_nxt, bad_best = decode(pkg, shape, w, bad)
    assert bad_status == cc.CC_ERR_DEVICE_ARG
    others = np.arange(len(lens)) != 7
    np.testing.assert_array_equal(bad_nxt[others], nxt[others])
    np.testing.assert_array_equal(bad_best[others], best[others])
    assert np.isfinite(bad_best[7])
    assert cc.cc_get_status() == cc.CC_OK


@pytest.mark.parametrize("slot", [0, 1400, 2999])
@pytest.mark.parametrize("rows", [1, 40])
def test_nan_key_gives_zero_rows(pkg, rows, slot):
    """A row that attends a NaN key comes out 0, whichever key split holds the
    key: a decode step (rows 1) and a chunk append, both with their keys split,
    against the same call over zero values.  (Zero new values too: Wv = 0.)"""
    from paper_2607_27600_gb300 import cc
    shape = ModelShape(2, 128, 4, 1, 64, 256, 300, 1e4, 1e-5)
    n, cap = 3000, 3200
    w_np = to_np(synth.model_weights(shape, 3, with_kv_proj=True))
    w_np["layers"][0]["wv"] = np.zeros_like(w_np["layers"][0]["wv"])
    out = []
    for nan in (True, False):
        c = to_device(to_np(synth.synthetic_cache(shape, [n], cap, 4)))
        if nan:
            c["k"][0][0, slot] = float("nan")
        else:
            c["v"][0].zero_()
        weights, cache = pkg.Weights(to_device(w_np)), pkg.Cache(c)
        tok = torch.arange(rows, dtype=torch.int32, device="cuda").reshape(1, rows)
        if rows == 1:
            ws = cc.alloc_workspace(cc.cc_decode_workspace_size(shape, 1, cap))
            nxt = torch.empty(1, dtype=torch.int32, device="cuda")
            cc.cc_decode_step(shape, weights, cache, tok[0], nxt, None, ws)
        else:
            ws = cc.alloc_workspace(cc.cc_append_workspace_size(shape, 1, cap))
            count = torch.tensor([rows], dtype=torch.int32, device="cuda")
            cc.cc_append_chunk(shape, weights, cache, tok, None, count, rows, ws)
        assert cc.cc_get_status() == cc.CC_OK
        out.append(c["h_last"][0, n:n + rows].float().cpu().numpy())
    np.testing.assert_array_equal(out[0], out[1])
    assert np.isfinite(out[0]).all()


@pytest.mark.parametrize("batch", [1, 20])
def test_infinite_activation_stays_infinite(pkg, batch):
    """One SwiGLU activation past fp32's range: the residual stream takes the
    sign of its down weights, as with single bf16 activations; the remainder of
    an infinite value in a bf16 pair is 0, not a NaN."""
    shape = ModelShape(2, 128, 4, 1, 64, 256, 300, 1e4, 1e-5)
    w_np = to_np(synth.model_weights(shape, 3, with_kv_proj=True))
    w_np["embed"][:, 0] = 1.0
    for key in ("w_gate", "w_up"):
        w_np["layers"][0][key][0] = 0.0
        w_np["layers"][0][key][0, 0] = 3e19
    down = w_np["layers"][0]["w_down"][:, 0]
    down[down == 0.0] = 0.01
    lens = [3 + i for i in range(batch)]
    c = to_device(to_np(synth.synthetic_cache(shape, lens, 64, 4)))
    status = decode(pkg, shape, to_device(w_np), c)[0]
    assert status == 0
    got = c["h_last"].float().cpu().numpy()
    for i, n in enumerate(lens):
        np.testing.assert_array_equal(got[i, n], np.sign(down) * np.float32(np.inf))


@pytest.mark.parametrize("dh,hkv,g,layout", [(64, 1, 4, "slot"), (128, 1, 8, "head"), (128, 2, 3, "paged"),
                                             (64, 1, 8, "e4m3"), (128, 1, 2, "e4m3")])
def test_splits_of_several_chunks(pkg, dh, hkv, g, layout):
    """Splits of three chunks and more: stages refilled, pages changing inside a
    split, and a reference max that later chunks raise (keys grow sixtyfold along
    the cache).  The tolerance of test_step_matches_oracle (e4m3: the new row's
    codes may round the other way, one key of thousands: 2^-6)."""
    import bench
    from tests.test_gpu_fp8 import fp8_views
    from tests._util import bf16_round
    shape = ModelShape(2, 256, hkv * g, hkv, dh, 512, 300, 1e4, 1e-5)
    lens, cap = [3900 - 27 * i for i in range(32 // hkv)], 4096
    lens += [2500 + i for i in range(16)] if hkv > 1 else []
    assert keys_per_split(shape, [n + 1 for n in lens], cap) >= 3 * 64
    w_np = to_np(synth.model_weights(shape, 3, with_kv_proj=True))
    c_np = to_np(synth.synthetic_cache(shape, lens, cap, 4))
    ramp = np.linspace(1.0, 60.0, cap, dtype=np.float32)[None, :, None, None]
    c_np["k"] = [bf16_round(x * ramp) for x in c_np["k"]]
    on, c = fp8_views(c_np) if layout == "e4m3" else (c_np, to_device(c_np))
    on = {k: ([np.asarray(x, np.float64).copy() for x in v] if k in ("k", "v") else
              v if isinstance(v, list) else np.asarray(v).copy()) for k, v in on.items()}
    if layout == "paged":
        bench.to_paged_cache(c, 128, 11)
    elif layout == "head":
        for key in ("k", "v"):
            c[key] = [x.permute(0, 2, 1, 3).contiguous() for x in c[key]]
        c["kv_layout"] = 1
    status, tok, _, _ = decode(pkg, shape, to_device(w_np), c)
    assert status == 0
    oracle.decode_step(shape, w_np, on, tok)
    got, tol = c["h_last"].float().cpu().numpy(), 2.0 ** (-6 if layout == "e4m3" else -7)
    for i, n in enumerate(lens):
        want = on["h_last"][i, n]
        assert np.abs(got[i, n] - want).max() <= tol * np.abs(want).max(), (i, n)


@pytest.mark.parametrize("batch", [5, 16, 17, 32, 33, 64, 65])
def test_batches_around_the_pair_layouts(pkg, batch):
    """Every sequence's appended K/V rows, H^(L-1), next token and logit, over a
    vocabulary that ends inside a column tile; the third sequence has no room, so
    the packed rows after it move up.  Pairs: 2^-7 of a row's largest; 65
    sequences travel as single bf16 rows: 2^-6."""
    shape = ModelShape(2, 256, 8, 2, 64, 512, 300, 1e4, 1e-5)
    cap = 160
    lens = [(37 * i) % 150 for i in range(batch)]
    lens[2] = cap
    w_np = to_np(synth.model_weights(shape, 3, with_kv_proj=True))
    c_np = to_np(synth.synthetic_cache(shape, lens, cap, 4))
    c = to_device(c_np)
    status, tok, nxt, best = decode(pkg, shape, to_device(w_np), c)
    assert status == 7 and nxt[2] == -1   # CC_ERR_DEVICE_ARG: the full sequence
    assert c["seq_len"].tolist() == [n + (i != 2) for i, n in enumerate(lens)]
    tol = 2.0 ** (-6 if batch > 64 else -7)
    cn = {k: ([np.asarray(x, np.float64).copy() for x in v] if isinstance(v, list) else
              np.asarray(v).copy()) for k, v in c_np.items()}
    for i, n in enumerate(lens):
        if i == 2:
            for key in ("k", "v"):
                for l in range(2):
                    assert np.array_equal(c[key][l][i].float().cpu().numpy(), c_np[key][l][i])
            continue
        one = {k: [x[i:i + 1] for x in v] if isinstance(v, list) else v[i:i + 1] for k, v in cn.items()}
        _, _, logits = oracle.decode_step(shape, w_np, one, tok[i:i + 1])
        rows = [(c["h_last"][i, n], one["h_last"][0, n])]
        rows += [(c[key][l][i, n], one[key][l][0, n]) for key in ("k", "v") for l in range(2)]
        for got, want in rows:
            want = np.asarray(want, np.float64)
            assert np.abs(got.float().cpu().numpy() - want).max() <= tol * np.abs(want).max(), i
        top = logits[0].max()
        assert logits[0][nxt[i]] >= top - tol * np.abs(logits[0]).max(), i
        assert abs(best[i] - top) <= tol * np.abs(logits[0]).max(), i
