"""The one-launch bucketing of small calls: where its CTA count, its queries per
thread or its shared-memory limit change, and just past its largest size (the
three-kernel path), the permutation, the tile list, Eq. 1's sum and the copy
decision are the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2608_27888_gb300 import workloads as W
from tests.util import QD, tiny_assets

pytestmark = pytest.mark.gpu


def check(D, S, q, m):
    import torch
    from paper_2608_27888_gb300 import ntc
    a = tiny_assets([[(2, 2), (1, 1)]] * S, hidden=64, out_dim=3, num_sets=S, num_decoders=D, set_to_decoder=m)
    dec = ntc.Decoder(a, "fp16")
    perm, counts, tiles, (copied, div) = dec.bucket(ntc.queries_to_device(q), divergence=True)
    p, c, _, t = oracle.bucket(q["set_id"], m, D)
    assert np.array_equal(perm.cpu().numpy().astype(np.uint32), p)
    assert np.array_equal(counts.cpu().numpy().astype(np.uint32), c)
    assert np.array_equal(tiles.cpu().numpy().astype(np.uint32), t)
    key = np.where(q["set_id"] < S, m[np.minimum(q["set_id"], S - 1)], D)
    want = sum(len(np.unique(key[i:i + 32])) - 1 for i in range(0, len(q), 32))
    assert (copied, div) == (int(want > 4 * ((len(q) + 31) // 32)), want)
    # the records in bucket order, through a decode of the same call
    out = dec.decode(ntc.queries_to_device(q))
    torch.cuda.synchronize()
    assert torch.isnan(out).any(1).cpu().numpy().tolist() == (q["set_id"] >= S).tolist()
    dec.close()


def stream(n, S, runs, seed):
    rng = np.random.default_rng(seed)
    q = np.zeros(n, dtype=QD)
    if runs:  # long runs of one set, ragged
        cut = np.sort(rng.integers(0, n, max(1, n // 700)))
        q["set_id"] = rng.integers(0, S + 1, len(cut) + 1)[np.searchsorted(cut, np.arange(n), side="right")]
    else:
        q["set_id"] = rng.integers(0, S + 1, n)  # S: out of range
    q["u"], q["v"] = rng.random(n), rng.random(n)
    return q


@pytest.mark.parametrize("runs", [False, True])
@pytest.mark.parametrize("n", [1, 32, 33, 1024, 1025, 4096, 4097, 8193, 16384, 16385, 32768, 32769, 40001, 65536, 65537, 131072, 131073])
def test_sizes(n, runs):
    S, D = 40, 23
    check(D, S, stream(n, S, runs, n), W.map_random_partition(5, S, D))


@pytest.mark.parametrize("D", [2, 586, 930, 950, 1380, 1420, 4095])
@pytest.mark.parametrize("n", [900, 5000, 65536])
def test_decoder_counts(n, D):
    check(D, D, stream(n, D, False, D), np.arange(D, dtype=np.uint32)[::-1].copy())
