"""k_step2 of a single lattice against single steps, bit for bit (fields, trace, saved state), on
lattices that no launch can hold on the SMs (700,000 sites on): widths around one and two
strips of 120 columns, odd and even, the narrowest and the flattest lattices, both storage types,
with and without omega = 1; with a trace (in pairs beyond L2, between them below) and without."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(64, 11001), (119, 6001), (120, 6000), (239, 3001), (240, 3000), (357, 2003), (1023, 700),
         (5, 340001), (8, 212501), (340001, 5), (20003, 36), (1800, 1000)]


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("prec,omega", [("fp32", 1.0), ("fp32", 0.8), ("fp16_delta", 1.0),
                                        ("fp16_delta", 1.3)])
@pytest.mark.parametrize("trace", [0, 4])
def test_pairs_equal_single_steps(nx, ny, prec, omega, trace):
    from paper_1008_2865_gb300 import Lattice, capi, inputs
    rho0 = inputs.noisy_density(nx, ny, seed=nx + ny, mean=0.7, amp=0.01, mode="rel")
    got = []
    for each in (1, 9):
        with Lattice(rho0, omega=omega, G1=-5.0, G2=0.6, prec=prec, trace_every=trace) as lat:
            for _ in range(9 // each):
                lat.step(each)
            assert capi.lb_check_guards(lat.handle) == 0
            got.append((*lat.fields(), lat.trace(), lat.save()))
    for a, b in zip(*got):
        assert np.array_equal(a, b)
