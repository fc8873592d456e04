"""Calls from a torch stream that is not the default one: the context's stream waits for what the
caller's stream holds (stokes_wait_for) and the caller's stream for the result (stokes_release_to)."""
import pytest
import torch

from paper_2311_06926_gb300 import Stokes

pytestmark = pytest.mark.gpu


def test_calls_are_ordered_with_the_callers_stream():
    """Inputs written late and outputs read early on side streams, alternating between two of them;
    the same numbers as with every step waited for."""
    G = Stokes(24, 2, max_order=2, max_steps=0, autotune=False)
    g = torch.Generator(device="cuda").manual_seed(1)
    base = torch.randn(G.size, dtype=torch.float64, device="cuda", generator=g)
    m = torch.randn(2048, 2048, device="cuda", generator=g)
    expected = []
    for k in range(6):
        y = G.apply_K(base * float(k + 1))
        torch.cuda.synchronize()
        expected.append(y.clone())
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for s in streams:
        s.wait_stream(torch.cuda.current_stream())
    x = [torch.zeros_like(base) for _ in range(6)]
    y = [torch.zeros_like(base) for _ in range(6)]
    out = [torch.zeros_like(base) for _ in range(6)]
    torch.cuda.synchronize()
    for k in range(6):
        with torch.cuda.stream(streams[k % 2]):
            t = m
            for _ in range(20):   # a few milliseconds before the input is there
                t = torch.tanh(t @ m)
            x[k].copy_(base * float(k + 1) + 0.0 * t[0, 0].double())
            G.apply_K(x[k], out=y[k])
            out[k].copy_(y[k])
            x[k].fill_(float("nan"))   # after the call in the caller's order
    torch.cuda.synchronize()
    for k in range(6):
        assert torch.equal(out[k], expected[k])
    G.close()


def test_a_context_on_the_callers_stream_needs_no_order():
    """The library's C calls with the context's own stream, and from the legacy default stream."""
    G = Stokes(8, 2, max_order=2, max_steps=0, autotune=False)
    x = torch.randn(G.size, dtype=torch.float64, device="cuda")
    ref = G.apply_K(x)
    torch.cuda.synchronize()
    assert G.lib.stokes_wait_for(G.h, G.stream.cuda_stream) == 0
    assert G.lib.stokes_release_to(G.h, G.stream.cuda_stream) == 0
    assert G.lib.stokes_wait_for(G.h, None) == 0
    assert G.lib.stokes_release_to(G.h, None) == 0
    assert G.lib.stokes_wait_for(None, None) < 0
    assert G.lib.stokes_release_to(None, None) < 0
    with torch.cuda.stream(G.stream):
        y = G.apply_K(x)
    torch.cuda.synchronize()
    assert torch.equal(y, ref)
    G.close()
