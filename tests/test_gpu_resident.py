"""Many steps of a small lattice in one launch (k_resident) against the same steps one
at a time (lb_step(1) is a single launch of k_step): fields, trace and saved state must
agree bit for bit, from the smallest lattice (one tile whose halo wraps around) over
odd sizes and narrow last tiles to the largest that fits, in both storage types, with
and without omega = 1, for trace periods that leave rows at the ends of a call and more
rows than one launch keeps; a bounded wait that runs out; and a captured graph."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(5, 5), (6, 7), (7, 300), (300, 6), (17, 9), (64, 32), (65, 33), (70, 45), (127, 129),
         (250, 187), (333, 50), (512, 384)]


def _run(nx, ny, prec, omega, trace, calls, shape=None):
    from paper_1008_2865_gb300 import Lattice, capi, inputs
    rho0 = inputs.noisy_density(nx, ny, seed=nx + ny, mean=0.7, amp=0.01, mode="rel")
    with Lattice(rho0, omega=omega, G1=-5.0, G2=0.6, prec=prec, trace_every=trace) as lat:
        if shape:
            lat.set_launch(*shape)
        for n in calls:
            lat.step(n)
        assert capi.lb_check_guards(lat.handle) == 0
        return (*lat.fields(), lat.trace(), lat.save())


def _same(one, two):
    for a, b in zip(one, two):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("prec,omega", [("fp32", 1.0), ("fp32", 0.8), ("fp16_delta", 1.0),
                                        ("fp16_delta", 1.3)])
def test_resident_steps_equal_single_steps(nx, ny, prec, omega):
    ref = _run(nx, ny, prec, omega, 6, [1] * 25)
    _same(ref, _run(nx, ny, prec, omega, 6, [25]))
    _same(ref, _run(nx, ny, prec, omega, 6, [2, 1, 13, 9]))


@pytest.mark.parametrize("trace", [0, 1, 7, 100])
@pytest.mark.parametrize("shape", [None, (128, 72, 0), (96, 4, 0), (256, 64, 0)])
def test_trace_rows_of_resident_steps(trace, shape):
    """Every launch shape's own summation order, chunks above and below 64 rows, and 40
    rows in one call (more than one launch keeps)."""
    ref = _run(130, 150, "fp32", 1.0, trace, [1] * 40, shape)
    _same(ref, _run(130, 150, "fp32", 1.0, trace, [40], shape))


@pytest.mark.parametrize("n,omega", [(640, 1.0), (680, 1.0), (720, 1.0), (560, 0.9), (600, 0.9)])
def test_either_side_of_the_largest_resident_lattice(n, omega):
    ref = _run(n, n + 3, "fp32", omega, 3, [1] * 7)
    _same(ref, _run(n, n + 3, "fp32", omega, 3, [7]))


def test_a_wait_that_runs_out():
    """The first tile marks its halo values with a step nobody waits for: its neighbours'
    waits run out, the next synchronising call reports it, and the context lives on."""
    from paper_1008_2865_gb300 import LBError, Lattice, capi, inputs
    rho0 = inputs.noisy_density(96, 80, seed=1, mean=0.7, amp=0.01, mode="rel")
    with Lattice(rho0, G1=-5.0, G2=0.6) as lat:
        capi.lb_set_wait_limit(lat.handle, 2_000_000, 1)
        lat.step(5)
        with pytest.raises(LBError) as e:
            lat.fields()
        assert e.value.status == capi.LB_ERR_TIMEOUT
        with pytest.raises(LBError):
            lat.step(1)
    with Lattice(rho0, G1=-5.0, G2=0.6) as lat:
        lat.step(5)
        assert np.isfinite(lat.energy()).all()


@pytest.mark.parametrize("nx", [96, 1024])
def test_captured_steps_replay(nx):
    """A captured even number of steps advances the state on every replay, as single
    launches that swap the buffers once each."""
    import torch
    from paper_1008_2865_gb300 import Lattice, inputs
    rho0 = inputs.noisy_density(nx, 300, seed=1, mean=0.7, amp=0.01, mode="rel")
    side = torch.cuda.Stream()
    with Lattice(rho0, G1=-5.0, G2=0.6, trace_every=0) as lat:
        lat.step(12)
        ref = lat.fields()
    with Lattice(rho0, G1=-5.0, G2=0.6, trace_every=0, stream=side.cuda_stream) as lat:
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=side):
            lat.step(4)
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        _same(ref, lat.fields())


def test_held_lattices_on_streams_of_their_own_threads():
    """Lattices of different sizes (so different tiles and shared memory), and an adjoint,
    each stepped by its own thread on its own stream at the same time, against the same
    work one after another."""
    import threading

    import torch
    from paper_1008_2865_gb300 import Lattice, inputs
    jobs = [(512, 384, 0), (96, 80, 0), (300, 301, 0), (128, 128, 40)]

    def work(nx, ny, adjoint, stream):
        rho0 = inputs.noisy_density(nx, ny, seed=nx, mean=0.7, amp=0.01, mode="rel")
        out = []
        for _ in range(6):
            with Lattice(rho0, G1=-5.0, G2=0.6, trace_every=7, stream=stream) as lat:
                if adjoint:
                    J, g, gG = lat.adjoint(adjoint, np.ascontiguousarray(rho0[::-1]))
                    out += [np.array([J, *gG]), g]
                else:
                    for _ in range(5):
                        lat.step(20)
                out += [*lat.fields(), lat.trace()]
        return out

    ref = [work(*j, 0) for j in jobs]
    got, bad = [None] * len(jobs), []

    def run(i):
        try:
            s = torch.cuda.Stream()
            got[i] = work(*jobs[i], s.cuda_stream)
        except Exception as exc:      # shown by the main thread
            bad.append((i, exc))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
    for one, two in zip(ref, got):
        _same(one, two)
