"""The adjoint on lattices with an odd number of sites (and one even one next to them):
checkpoints and segment states follow one another in memory, and each must start where
its population pairs are aligned. Bars as in test_gpu_adjoint.py (J 1e-6, gradients
1e-4), several segments long."""
import numpy as np
import pytest

import oracle
from paper_1008_2865_gb300 import Lattice, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(5, 5), (17, 13), (33, 21), (34, 21)])
@pytest.mark.parametrize("every", [0, 3])
def test_adjoint_of_odd_lattices(nx, ny, every):
    r0 = inputs.noisy_density(nx, ny, 11, mean=0.7, amp=0.01, mode="rel")
    tgt = inputs.noisy_density(nx, ny, 12, mean=0.7, amp=0.01, mode="rel")
    Jo, go, gGo = oracle.gradient(r0, tgt, 20, G1=-5.0, G2=0.5)
    with Lattice(r0, G1=-5.0, G2=0.5, trace_every=0) as lat:
        J, g, gG = lat.adjoint(20, tgt, checkpoint_every=every)
    assert abs(J - Jo) <= 1e-6 * abs(Jo)
    assert np.linalg.norm(g - go) <= 1e-4 * np.linalg.norm(go)
    for k in range(2):
        assert abs(gG[k] - gGo[k]) <= 1e-4 * abs(gGo[k])


@pytest.mark.parametrize("nx,ny", [(5, 5), (6, 40), (64, 33), (250, 187), (512, 96)])
def test_held_reverse_equals_the_two_passes(nx, ny):
    """omega = 1 on a lattice that fits the SMs takes a segment back in one launch; the
    two-pass path takes one step at a time. 1 - 2^-24 rounds to an FP32 omega other than 1,
    so it takes the two passes with couplings and arithmetic that differ by one rounding:
    the results agree far inside the FP32 error of either (bar 2e-6 in J, 1e-4 in the
    gradients, as against the oracle), for one segment, several and a short last one."""
    r0 = inputs.noisy_density(nx, ny, 11, mean=0.7, amp=0.01, mode="rel")
    tgt = inputs.noisy_density(nx, ny, 12, mean=0.7, amp=0.01, mode="rel")
    got = {}
    for omega in (1.0, 1.0 - 2.0 ** -24):
        for every in (0, 7, 30):
            with Lattice(r0, omega=omega, G1=-5.0, G2=0.5, trace_every=4) as lat:
                J, g, gG = lat.adjoint(30, tgt, checkpoint_every=every)
                got[omega, every] = (J, g, gG, lat.trace(), lat.fields())
    for omega in (1.0, 1.0 - 2.0 ** -24):
        for every in (7, 30):                      # any spacing, the same bits
            one, two = got[omega, 0], got[omega, every]
            assert one[0] == two[0] and one[2] == two[2] and np.array_equal(one[1], two[1])
            assert np.array_equal(one[3], two[3])
            assert all(np.array_equal(p, q) for p, q in zip(one[4], two[4]))
    (J, g, gG, *_), (Jt, gt, gGt, *_) = got[1.0, 0], got[1.0 - 2.0 ** -24, 0]
    assert abs(J - Jt) <= 2e-6 * abs(Jt)
    assert np.linalg.norm(g - gt) <= 1e-4 * np.linalg.norm(gt)
    for k in range(2):
        assert abs(gG[k] - gGt[k]) <= 1e-4 * abs(gGt[k])


def test_held_segment_of_more_steps_than_a_grid_dimension():
    """One segment of 70,000 steps (more than a grid may have rows) against segments of
    265: the same bits. The lattice has no unstable mode, so nothing overflows."""
    r0 = inputs.noisy_density(5, 5, 11, mean=0.7, amp=0.01, mode="rel")
    tgt = inputs.noisy_density(5, 5, 12, mean=0.7, amp=0.01, mode="rel")
    got = []
    for every in (0, 70000):
        with Lattice(r0, G1=-3.0, G2=0.2, trace_every=0) as lat:
            got.append(lat.adjoint(70000, tgt, checkpoint_every=every))
    assert got[0][0] == got[1][0] and got[0][2] == got[1][2]
    assert np.array_equal(got[0][1], got[1][1])
