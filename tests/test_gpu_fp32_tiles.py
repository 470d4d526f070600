"""The fp32 decode's tiles of every kind of length: where a warp's queries begin
and where its second half does (32, 64, 96), and one row either side."""
import numpy as np
import pytest

import oracle
from paper_2608_27888_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LENGTHS = [1, 2, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 191, 193, 0, 256]


@pytest.mark.parametrize("hidden", [64, 128])
@pytest.mark.parametrize("out_dim", [3, 8, 9, 16])
def test_lengths(hidden, out_dim):
    from paper_2608_27888_gb300 import ntc
    D = len(LENGTHS)
    a = W.make_assets(41, D, 32, 2, D, W.map_identity(D), hidden=hidden, out_dim=out_dim)
    rng = np.random.default_rng(hidden + out_dim)
    q = np.zeros(sum(LENGTHS), dtype=W.QUERY_DTYPE)
    q["set_id"] = rng.permutation(np.repeat(np.arange(D), LENGTHS))
    q["u"], q["v"], q["lod"] = rng.random(len(q)), rng.random(len(q)), rng.random(len(q))
    dec = ntc.Decoder(a, "fp32")
    got = dec.decode(ntc.queries_to_device(q)).cpu().numpy()
    ref, _ = oracle.decode(a, q)
    assert np.abs(got - ref).max() <= 1e-5  # the fp32 tolerance of the parity tests
    assert dec.error_count() == 0
    dec.close()
