"""The keep-set select's segments (csrc/select.cu): a sequence over 1, 2, 4 or
8 CTAs by cap and batch, keys kept in shared memory up to 45056 slots of a
segment and re-read above.  Lengths around those lines and around segment
ends, ties that straddle segments, sinks, and batches whose sequences end in
different segments: exact against the oracle's select."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap,lens", [
    (2048, [2048, 1, 2047]), (8192, [8192, 33, 8191]), (8193, [8193, 5, 8, 9]),
    (9000, [8997, 33, 4500, 9000]),
    (131072, [131071, 16385, 0]), (8 * 45056 + 64, [8 * 45056 + 61])])
@pytest.mark.parametrize("kind", ["normal", "ties", "special", "one value"])
@pytest.mark.parametrize("n_sink", [0, 5])
def test_select_matches_the_oracle(cap, lens, kind, n_sink):
    _check(cap, lens, kind, n_sink, (0.003, 0.5, 0.97))


@pytest.mark.parametrize("cap", [9001, 16384, 50000])
@pytest.mark.parametrize("batch", [12, 17, 40, 80, 160])
@pytest.mark.parametrize("kind", ["normal", "ties"])
def test_select_of_a_batch(cap, batch, kind):
    """Batches whose clusters of eight would queue for the SMs take fewer CTAs
    per sequence, down to one, with keys held and re-read."""
    r = np.random.default_rng(batch)
    lens = r.integers(1, cap + 1, batch).tolist()
    lens[:3] = [cap, cap - 1, 1]
    _check(cap, lens, kind, 2, (0.3,))


def _check(cap, lens, kind, n_sink, parts):
    from paper_2607_27600_gb300 import cc
    cc.load_library()
    r = np.random.default_rng(cap + len(kind) + n_sink)
    b = len(lens)
    s = r.standard_normal((b, cap)).astype(np.float32)
    if kind == "ties":
        s = np.round(s)
    elif kind == "special":
        for v in (np.nan, np.inf, -np.inf, 0.0, -0.0):
            s[r.random((b, cap)) < 0.15] = v
    elif kind == "one value":
        s[:] = -1.5
    for part in parts:
        budget = [max(int(n * part), min(n, 1 + n_sink)) for n in lens]
        idx = torch.full((b, cap), -7, dtype=torch.int32, device="cuda")
        cnt = torch.zeros(b, dtype=torch.int32, device="cuda")
        cc.cc_select_keep(torch.from_numpy(s).cuda(), torch.tensor(lens, dtype=torch.int32, device="cuda"),
                          b, cap, torch.tensor(budget, dtype=torch.int32, device="cuda"), n_sink, idx, cnt)
        assert cc.cc_get_status() == cc.CC_OK
        want, count = oracle.select_keep(s, lens, budget, n_sink)
        got = idx.cpu().numpy()
        assert np.array_equal(cnt.cpu().numpy(), count)
        for i in range(b):
            assert np.array_equal(got[i, :count[i]], want[i, :count[i]]), (i, part)
            assert np.all(got[i, count[i]:] == -7)   # entries past the count are not written
