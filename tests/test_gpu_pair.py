"""Steps taken two at a time (k_step2, lattices of 2^18 sites on) against the same
steps taken one at a time (lb_step(1) never pairs): the fields and the trace must
agree bit for bit, from the narrowest and the flattest lattices to several strips
and row chunks, with odd and even sizes, at the strip width (120 columns) and one
to either side, in both storage types, with and without omega = 1."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(5, 52429), (8, 32768), (119, 2203), (120, 2185), (121, 2170), (122, 2149), (241, 1088),
         (512, 512), (1023, 257), (2050, 131), (52430, 5)]


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("prec,omega", [("fp32", 1.0), ("fp32", 0.8), ("fp16_delta", 1.0),
                                        ("fp16_delta", 1.3)])
def test_paired_steps_equal_single_steps(nx, ny, prec, omega):
    from paper_1008_2865_gb300 import Lattice, capi, inputs
    rho0 = inputs.noisy_density(nx, ny, seed=nx + ny, mean=0.7, amp=0.01, mode="rel")
    got = []
    for chunks in ([1] * 13, [13], [4, 9]):
        with Lattice(rho0, omega=omega, G1=-5.0, G2=0.6, prec=prec, trace_every=6) as lat:
            for n in chunks:
                lat.step(n)
            got.append((*lat.fields(), lat.trace(), lat.save()))
            assert lat.t == 13
            assert capi.lb_check_guards(lat.handle) == 0
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("sizes", [[(5, 5)], [(96, 80), (121, 33), (240, 17)],
                                   [(64, 700), (5, 9), (1500, 12), (120, 120)]])
@pytest.mark.parametrize("prec,omega", [("fp32", 1.0), ("fp32", 0.9), ("fp16_delta", 1.0),
                                        ("fp16_delta", 1.2)])
@pytest.mark.parametrize("trace", [0, 6, 20])
def test_paired_batch_steps_equal_single_steps(sizes, prec, omega, trace):
    """A batch stepped in one call (pairs, graph replay, odd numbers of buffer swaps per
    period) against one step per call (no pairs), and two calls that split a period."""
    from paper_1008_2865_gb300 import Batch, inputs
    rhos = [inputs.noisy_density(nx, ny, seed=nx + ny, mean=0.7, amp=0.01, mode="rel")
            for nx, ny in sizes]
    om = [omega] + [1.0] * (len(sizes) - 1)
    got = []
    for chunks in ([1] * 47, [47], [3, 37, 7]):
        with Batch(rhos, omega=om, G1=-5.0, G2=0.6, prec=prec, trace_every=trace) as b:
            for n in chunks:
                b.step(n)
            got.append([(*b.fields(i), b.trace(i)) for i in range(len(b))])
            assert b.t == 47
    for other in got[1:]:
        for one, two in zip(got[0], other):
            for p, q in zip(one, two):
                assert np.array_equal(p, q)
