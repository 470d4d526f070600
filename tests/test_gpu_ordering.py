"""Calls whose kernels start before their predecessor on the stream has ended:
queries written by a kernel just before the call, two contexts on two streams, and
captured calls on changing queries. The rows are those of the same queries decoded
on an idle GPU, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2608_27888_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# n: one-launch bucketing, three kernels; 1 decoder: no bucketing
CASES = [(900, 7, {}), (65_000, 7, {}), (200_000, 7, {}), (200_000, 300, {}), (30_000, 1, {}),
         (50_000, 5, dict(levels=1, channels=4, pe_frequencies=3, layers=3))]


def setup(n, D, general, hidden=64):
    from paper_2608_27888_gb300 import ntc
    S = max(16, D)
    a = W.make_assets(9, S, 32, 1, D, W.map_random_partition(3, S, D), hidden=hidden, out_dim=9, **general)
    dec = ntc.Decoder(a, "fp16")
    qs = [ntc.queries_to_device(W.queries_uniform(70 + i, n, S)) for i in range(6)]
    want = []
    for q in qs:
        torch.cuda.synchronize()
        want.append(dec.decode(q))
    torch.cuda.synchronize()
    return dec, qs, want


@pytest.mark.parametrize("n,D,general", CASES)
def test_queries_written_just_before(n, D, general):
    dec, qs, want = setup(n, D, general)
    q = torch.empty_like(qs[0])
    got = []
    for rep in range(4):
        for s in qs:
            torch.add(s, 0, out=q)  # (a kernel; a copy would be a memcpy)
            got.append(dec.decode(q))
    assert all(torch.equal(g, want[i % len(qs)]) for i, g in enumerate(got))
    dec.close()


@pytest.mark.parametrize("n,D,general", CASES)
def test_two_contexts_on_two_streams(n, D, general):
    both = [setup(n, D, general), setup(n, D, general, hidden=128)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = [[], []]
    for rep in range(3):
        for i in range(6):
            for k, (dec, qs, _) in enumerate(both):
                with torch.cuda.stream(streams[k]):
                    got[k].append(dec.decode(qs[i]))
    torch.cuda.synchronize()
    for k, (dec, qs, want) in enumerate(both):
        assert all(torch.equal(g, want[i % 6]) for i, g in enumerate(got[k]))
        dec.close()


@pytest.mark.parametrize("n,D,general", CASES)
def test_captured(n, D, general):
    dec, qs, want = setup(n, D, general)
    q, out = torch.empty_like(qs[0]), torch.empty_like(want[0])
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):
        dec.decode(q, out, stream=s)
    for rep in range(2):
        for src, w in zip(qs, want):
            torch.add(src, 0, out=q)
            g.replay()
            assert torch.equal(out, w)
    dec.close()
