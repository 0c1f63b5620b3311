"""cc_compact_kv_static: compaction for callers that cannot allocate device
memory (for example a serving loop whose whole device pool is already the KV
cache).  It must give exactly what cc_compact_kv gives with a workspace, on
two calls in a row, because its scratch is one fixed array shared by every
call on the device and keeping the previous call's contents.

This file is collected last so that a run stopping at the first failure has
already run every other test."""
import numpy as np
import pytest
import torch

import synth
from synth.configs import ModelShape

pytestmark = pytest.mark.gpu

SHAPE = ModelShape(n_layers=3, d_model=256, n_q_heads=8, n_kv_heads=2, head_dim=64,
                   d_ff=384, vocab=1000, rope_theta=1e4, rms_eps=1e-5)


def _keep(seq, cap, seed):
    r = np.random.default_rng(seed)
    idx = np.full((len(seq), cap), -1, np.int32)
    cnt = np.zeros(len(seq), np.int32)
    for b, n in enumerate(seq):
        k = np.sort(r.choice(n, size=max(1, n // 3), replace=False))
        idx[b, :len(k)] = k
        cnt[b] = len(k)
    return torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda()


def _snapshot(c):
    return [t.clone() for t in c["k"] + c["v"]] + [c["h_last"].clone(), c["tokens"].clone(),
                                                   c["pos"].clone(), c["seq_len"].clone()]


def test_static_scratch_compaction_matches_workspace_version_twice():
    import paper_2607_27600_gb300 as pkg
    from paper_2607_27600_gb300 import cc
    pkg.load_library()
    seq, cap = [3000, 1777], 3072
    ref = synth.synthetic_cache(SHAPE, seq, cap, seed=41, device="cuda")
    stat = {k: ([t.clone() for t in v] if isinstance(v, list) else v.clone())
            for k, v in ref.items()}
    ref_c, stat_c = pkg.Cache(ref), pkg.Cache(stat)
    ws = cc.alloc_workspace(cc.cc_compact_workspace_size(SHAPE, ref_c))
    for call, seed in enumerate((1, 2)):
        idx, cnt = _keep([int(x) for x in ref["seq_len"].tolist()], cap, seed)
        cc.cc_compact_kv(SHAPE, ref_c, idx, cnt, ws)
        cc.cc_compact_kv_static(SHAPE, stat_c, idx, cnt)
        assert cc.cc_get_status() == cc.CC_OK
        for a, b in zip(_snapshot(ref), _snapshot(stat)):
            assert torch.equal(a, b), f"call {call}"
        assert stat["seq_len"].tolist() == cnt.tolist()


def test_static_scratch_rejects_caches_beyond_its_size():
    import paper_2607_27600_gb300 as pkg
    from paper_2607_27600_gb300 import cc
    big = ModelShape(n_layers=64, d_model=256, n_q_heads=8, n_kv_heads=2, head_dim=64, d_ff=384,
                     vocab=1000, rope_theta=1e4, rms_eps=1e-5)
    # 128 K/V arrays of 256-byte rows move in 4 KB units of 16 slots: 2^19 / 16 = 32768
    # units per array, so about 4.2 M four-byte unit flags (16 MiB) > the 1 MiB array
    cap = 1 << 19
    tiny = torch.zeros(16, dtype=torch.bfloat16, device="cuda")   # pointers are not dereferenced
    c = {"k": [tiny] * 64, "v": [tiny] * 64, "h_last": None,
         "tokens": torch.zeros(1, 1, dtype=torch.int32, device="cuda"),
         "pos": torch.zeros(1, 1, dtype=torch.int32, device="cuda"),
         "seq_len": torch.zeros(1, dtype=torch.int32, device="cuda")}
    cache = pkg.Cache(c)
    cache.c.cap = cap      # host-side plan only: rejected before anything is enqueued
    idx = torch.zeros(1, dtype=torch.int32, device="cuda")
    with pytest.raises(cc.CCError) as e:
        cc.cc_compact_kv_static(big, cache, idx, idx)
    assert e.value.code == cc.CC_ERR_WORKSPACE


@pytest.mark.parametrize("layout", ["slot", "paged", "head"])
@pytest.mark.parametrize("d_model", [256, 4096])
def test_units_of_more_rows_than_lanes(layout, d_model):
    """64-byte K/V rows (one head of 64 e4m3 values): units of 64 rows, or 128
    beside 8 KB H rows.  Exact against a gather; an entry below its slot in a
    unit's second half is reported and its row left alone."""
    import bench
    import paper_2607_27600_gb300 as pkg
    from paper_2607_27600_gb300 import cc
    pkg.load_library()
    shape = ModelShape(2, d_model, 8, 1, 64, 384, 1000, 1e4, 1e-5)
    seq, cap = [2000, 777], 2048
    c = synth.synthetic_cache(shape, seq, cap, seed=7, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(3)
    for key in ("k", "v"):
        c[key] = [torch.randint(0, 120, x.shape, dtype=torch.uint8, device="cuda", generator=g)
                  for x in c[key]]
    c["kv_scale"] = [(1.0, 1.0)] * 2
    before = {k: [x.clone() for x in c[k]] for k in ("k", "v")}
    if layout == "paged":
        bench.to_paged_cache(c, 128, 5)
    elif layout == "head":
        for key in ("k", "v"):
            c[key] = [x.permute(0, 2, 1, 3).contiguous() for x in c[key]]
        c["kv_layout"] = 1
    idx, cnt = _keep(seq, cap, 9)
    bad = 50                               # the second half of the first unit
    idx[0, bad] = bad - 1
    cache = pkg.Cache(c)
    ws = cc.alloc_workspace(cc.cc_compact_workspace_size(shape, cache))
    cc.cc_compact_kv(shape, cache, idx, cnt, ws)
    assert cc.cc_get_status() == cc.CC_ERR_DEVICE_ARG
    idx[0, bad] = bad
    for key in ("k", "v"):
        for l in range(2):
            got = bench.logical_kv(c, key, l)
            for b in range(2):
                n = int(cnt[b])
                assert torch.equal(got[b, :n], before[key][l][b, idx[b, :n].long()])


def test_static_scratch_takes_short_rows():
    """64-byte rows move in units of 64 slots: 128 (array, sequence) pairs of
    98304 slots need 0.8 MiB of scratch, within the fixed array."""
    import paper_2607_27600_gb300 as pkg
    from paper_2607_27600_gb300 import cc
    pkg.load_library()
    shape = ModelShape(8, 256, 8, 1, 64, 384, 1000, 1e4, 1e-5)
    b, cap = 8, 98304
    c = {k: [torch.randint(0, 120, (b, cap, 1, 64), dtype=torch.uint8, device="cuda")
             for _ in range(8)] for k in ("k", "v")}
    c.update(h_last=None, kv_scale=[(1.0, 1.0)] * 8,
             tokens=torch.arange(b * cap, dtype=torch.int32, device="cuda").reshape(b, cap),
             pos=torch.zeros((b, cap), dtype=torch.int32, device="cuda"),
             seq_len=torch.full((b,), cap, dtype=torch.int32, device="cuda"))
    cache = pkg.Cache(c)
    assert cc.cc_compact_workspace_size(shape, cache) <= 1 << 20
    idx, cnt = _keep([cap] * b, cap, 4)
    want = {k: [x[1, idx[1, :int(cnt[1])].long()] for x in c[k]] for k in ("k", "v")}
    cc.cc_compact_kv_static(shape, cache, idx, cnt)
    assert cc.cc_get_status() == cc.CC_OK
    for key in ("k", "v"):
        for x, y in zip(c[key], want[key]):
            assert torch.equal(x[1, :int(cnt[1])], y)
