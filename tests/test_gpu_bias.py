"""Biases of any size that fp32 holds and the logits keep in range: they count in
fp32 in the tensor-core decodes too, also where an fp16 part alone would overflow."""
import numpy as np
import pytest

import oracle
from tests.util import queries, split_weights, tiny_assets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp16", "bf16"])
@pytest.mark.parametrize("hidden,channels,layers", [(64, 8, 2), (128, 8, 2), (16, 4, 2), (64, 4, 3), (128, 4, 4)])
def test_large_biases_that_cancel(precision, hidden, channels, layers):
    from paper_2608_27888_gb300 import ntc
    a = tiny_assets([[(4, 4), (2, 2)]], channels=channels, hidden=hidden, layers=layers, out_dim=4)
    w = split_weights(a)
    w[1][:] = 128.0                          # the first hidden layer's values: 128, exact in both types
    for l in range(1, layers):               # further ones: -2^17 + (2^17 + 128) = 128 again
        w[2 * l][:, 0], w[2 * l + 1][:] = -1024.0, 2.0 ** 17 + 128.0
    w[-2][:, 1] = -1024.0                    # logits: -2^17 + 2^17 + x
    x = np.array([1.0, -1.0, 0.25, -2.0], np.float32)
    w[-1][:] = np.float32(2.0 ** 17) + x
    dec = ntc.Decoder(a, precision)
    q = queries([(0, 0.3, 0.7, 0.0)] * 200)
    got = dec.decode(ntc.queries_to_device(q)).cpu().numpy()
    ref, _ = oracle.decode(a, q)
    assert np.abs(ref - 1.0 / (1.0 + np.exp(-x))).max() < 1e-6
    assert np.abs(got - ref).max() <= 2e-3   # tanh.approx (2^-11) and a 2^-6 step of the fp32 logit's terms
    dec.close()
