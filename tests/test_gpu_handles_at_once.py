"""Small handles stepped at once on streams of their own share the GPU: a short call does not wait
for the long calls of the others to end."""
import numpy as np
import pytest

from paper_1707_00198_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,others", [("fp64", 1), ("fp32", 3)])
def test_a_short_call_beside_long_ones(prec, others):
    import torch
    from paper_1707_00198_gb300.lbcg import Lattice
    g, p = I.config_static_droplet()
    streams = [torch.cuda.Stream() for _ in range(others + 1)]
    hs = [Lattice(g, p, prec, stream=s.cuda_stream) for s in streams]
    one = Lattice(g, p, prec)
    one.step(100)
    one.step(40)
    want = one.populations()
    one.close()
    for L in hs:
        L.step(100)
    torch.cuda.synchronize()
    ends = []
    for L, s in zip(hs, streams):
        L.step(40 if L is hs[-1] else 8000)      # (one cooperative launch each)
        ends.append(torch.cuda.Event(enable_timing=True))
        ends[-1].record(s)
    torch.cuda.synchronize()
    # the short call was launched last and ended first
    assert all(ends[-1].elapsed_time(e) > 0 for e in ends[:-1])
    assert np.array_equal(hs[-1].populations(), want)
    for L in hs:
        L.close()
