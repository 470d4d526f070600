"""Output rows of every channel count, in both element types: rows side by side in
the caller's order and scattered ones, ragged last tiles, and nothing written
outside the rows."""
import numpy as np
import pytest

import oracle
from paper_2608_27888_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL_MAX, TOL_MEAN = 2e-2, 2e-3  # the tensor-core tolerance of the parity tests
GUARD = 64  # elements before and after the rows


@pytest.mark.parametrize("hidden", [64, 128])
@pytest.mark.parametrize("output", ["fp32", "fp16"])
@pytest.mark.parametrize("out_dim", [1, 3, 8, 9, 10, 12, 15, 16])
def test_rows_of_every_width(out_dim, output, hidden):
    import torch
    from paper_2608_27888_gb300 import ntc
    a = W.make_assets(31, 6, 64, 2, 5, np.array([0, 1, 2, 3, 4, 1]), hidden=hidden, out_dim=out_dim)
    coherent = W.queries_gbuffer(32, 64, 44, 5, 6, 64)        # long runs of one decoder: rows side by side
    mixed = W.queries_uniform(33, 1500 + 77, 6)               # scattered rows, ragged tiles
    mixed["set_id"][::97] = 6                                 # bad rows: NaN
    q = np.concatenate([coherent, mixed])
    dec = ntc.Decoder(a, "fp16", output)
    dq = ntc.queries_to_device(q)
    for shift in (0, 1):  # a base aligned for vector rows, and one that is not
        buf = torch.full((GUARD + shift + len(q) * out_dim + GUARD,), 7.0, dtype=dec.out_dtype(), device="cuda")
        rows = buf[GUARD + shift:GUARD + shift + len(q) * out_dim].view(len(q), out_dim)
        dec.decode(dq, rows)
        got = rows.float().cpu().numpy()
        assert (buf[:GUARD + shift] == 7.0).all() and (buf[-GUARD:] == 7.0).all()
        ref, _ = oracle.decode(a, q)
        bad = q["set_id"] >= 6
        assert np.isnan(got[bad]).all()
        err = np.abs(got[~bad] - ref[~bad])
        assert err.max() <= TOL_MAX and err.mean() <= TOL_MEAN
    dec.close()
