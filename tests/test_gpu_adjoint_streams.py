"""Adjoints of one handle on two streams: both use the scratch that stays with it."""
import pytest

from paper_2502_01496_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_two_streams_one_handle(precision):
    """Alternating cotangents on two streams, nothing waited for between the calls,
    against one stream: equal up to the order of float64 atomics (1e-12 of the
    largest component); a second, larger set grows the scratch in between."""
    import torch
    from paper_2502_01496_gb300 import native
    f = native.KdFmm(theta=0.5, eps=0.01, n_leaf=16, precision=precision)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for n in (30000, 100000):
        ps = W.plummer(n, n)
        x = torch.tensor(ps.x, device="cuda")
        f.build(x, torch.tensor(ps.m, device="cuda")).accel()
        g = torch.Generator("cuda").manual_seed(n)
        b = [torch.randn(x.shape, dtype=torch.float64, device="cuda", generator=g) for _ in range(8)]
        want = []
        for v in b:
            want.append(f.vjp(v))
            torch.cuda.synchronize()
        got = []
        for k, v in enumerate(b):
            with torch.cuda.stream(streams[k & 1]):
                got.append(f.vjp(v))
        torch.cuda.synchronize()
        for p, q in zip(got, want):
            for u, v in zip(p, q):
                assert (u - v).abs().max() <= 1e-12 * v.abs().max()
