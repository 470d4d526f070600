"""Long tile lists: where a CTA's groups of neighbouring tiles become two and four
tiles long, with few and many decoders, the tensor-core pipelines agree with the
per-lane decode of the same context (another kernel, unsorted)."""
import numpy as np
import pytest

from paper_2608_27888_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def check(hidden, general, precision, decoders, n):
    import torch
    from paper_2608_27888_gb300 import ntc
    a = W.make_assets(17, 97, 16, 2, decoders, np.arange(97) % decoders, hidden=hidden, out_dim=9, **general)
    rng = np.random.default_rng(n)
    q = np.zeros(n, dtype=W.QUERY_DTYPE)
    cut = np.sort(rng.integers(0, n, 3000))
    q["set_id"] = rng.integers(0, 97, 3001)[np.searchsorted(cut, np.arange(n), side="right")]
    q["u"], q["v"], q["lod"] = rng.random(n), rng.random(n), rng.random(n)
    dec = ntc.Decoder(a, precision)
    dq = ntc.queries_to_device(q)
    err = (dec.decode(dq) - dec.decode(dq, mode="divergent_fma")).abs()
    assert torch.isfinite(err).all()
    assert err.max() <= 2e-2 and err.mean() <= 2e-3  # the tensor-core tolerance of the parity tests
    assert dec.error_count() == 0
    dec.close()


@pytest.mark.parametrize("n", [466_945, 1_245_185 + 77])  # 24 and 64 tiles of 128 per CTA (152 CTAs), and a ragged end
@pytest.mark.parametrize("decoders", [3, 97])
@pytest.mark.parametrize("shape", ["64", "128", "general-64", "general-128"])
def test_groups(shape, decoders, n):
    hidden = int(shape.split("-")[-1])
    general = dict(levels=1, channels=4, pe_frequencies=4, activation=1, layers=3) if "general" in shape else {}
    check(hidden, general, "fp16", decoders, n)


@pytest.mark.parametrize("hidden", [16, 32, 64, 128])
@pytest.mark.parametrize("levels,channels,pe,layers,precision", [
    (2, 8, 0, 3, "fp16"), (2, 8, 6, 1, "bf16"), (1, 8, 3, 4, "fp16"), (2, 4, 5, 2, "bf16"), (1, 4, 0, 1, "fp16")])
def test_every_general_layout(levels, channels, pe, layers, precision, hidden):
    """Each instantiation of the general pipeline on lists of 24 and more tiles per
    CTA, so that its stages, slots, images and output-row ring are all used again."""
    general = dict(levels=levels, channels=channels, pe_frequencies=pe, layers=layers, activation=layers % 2)
    check(hidden, general, precision, 97, 466_945)
