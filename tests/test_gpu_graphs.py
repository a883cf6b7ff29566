"""A captured graph of an even number of steps stays valid when steps are taken outside it
between its replays: whatever those steps share launches with, they leave the state in the
buffers that the graph reads. Against the same number of steps in a state of its own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _capture(side, step):
    import torch
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=side):
        step(4)
    return g


def _replay(g, side):
    import torch
    with torch.cuda.stream(side):       # the state's stream, in order with its other steps
        g.replay()


# held on the SMs; taken two at a time; a lattice whose second strip is two columns wide
@pytest.mark.parametrize("nx,ny", [(96, 300), (1024, 768), (122, 4400)])
@pytest.mark.parametrize("trace", [0, 3, 4])
@pytest.mark.parametrize("between", [2, 3, 4, 6, 7])
def test_steps_between_replays(nx, ny, trace, between):
    import torch
    from paper_1008_2865_gb300 import Lattice, inputs
    rho0 = inputs.noisy_density(nx, ny, seed=1, mean=0.7, amp=0.01, mode="rel")
    kw = dict(G1=-5.0, G2=0.6, trace_every=trace)
    side = torch.cuda.Stream()
    steps = 2 * between + 2 * 4
    with Lattice(rho0, **kw) as lat:
        lat.step(steps)
        ref = lat.fields()
    with Lattice(rho0, stream=side.cuda_stream, **kw) as lat:
        g = _capture(side, lat.step)
        lat.step(between)
        if between % 2:
            lat.step(1)                 # back in the graph's buffers
        _replay(g, side)
        lat.step(between - between % 2)
        _replay(g, side)
        torch.cuda.synchronize()
        got = lat.fields()
    for a, b in zip(ref, got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("trace", [0, 3, 10])
@pytest.mark.parametrize("between", [2, 6, 22])
def test_batch_steps_between_replays(trace, between):
    import torch
    from paper_1008_2865_gb300 import Batch, inputs
    rhos = [inputs.noisy_density(nx, ny, seed=nx, mean=0.7, amp=0.01, mode="rel")
            for nx, ny in ((96, 80), (131, 67))]
    kw = dict(G1=-5.0, G2=[0.6, 0.3], trace_every=trace)
    side = torch.cuda.Stream()
    with Batch(rhos, **kw) as b:
        b.step(2 * between + 8)
        ref = [b.fields(i) for i in range(2)]
    with Batch(rhos, stream=side.cuda_stream, **kw) as b:
        b.step(1)                       # its launches are ready before the capture
        b.step(1)
        g = _capture(side, b.step)
        b.step(between - 2)
        _replay(g, side)
        b.step(between)
        _replay(g, side)
        torch.cuda.synchronize()
        got = [b.fields(i) for i in range(2)]
    for one, two in zip(ref, got):
        for a, c in zip(one, two):
            assert np.array_equal(a, c)
