"""Memory that only faster ways to step need (the density deviations of traced states, the
halo words and kept states of a held lattice): where it cannot be had, the state is made all
the same, and its steps give the same fields and trace bit for bit."""
import numpy as np
import pytest

from paper_1008_2865_gb300 import Batch, Lattice, capi, inputs

pytestmark = pytest.mark.gpu

NEEDED = 11      # control words (5), partial sums, trace ring, populations and psi (4)


@pytest.fixture
def fail_alloc():
    yield capi.lb_debug_fail_alloc
    capi.lb_debug_fail_alloc(-1)


@pytest.mark.parametrize("nx,ny", [(96, 80), (1000, 700), (1500, 1300)])
@pytest.mark.parametrize("prec,omega", [("fp32", 1.0), ("fp16_delta", 0.9)])
@pytest.mark.parametrize("after", [NEEDED, NEEDED + 1, NEEDED + 4])
def test_a_state_without_scratch(nx, ny, prec, omega, after, fail_alloc):
    rho0 = inputs.noisy_density(nx, ny, seed=3, mean=0.7, amp=0.01, mode="rel")
    got = []
    for fail in (-1, after):
        fail_alloc(fail)
        with Lattice(rho0, omega=omega, G1=-5.0, G2=0.6, prec=prec, trace_every=4) as lat:
            fail_alloc(-1)
            lat.step(11)
            got.append((*lat.fields(), lat.trace(), lat.save()))
            assert capi.lb_check_guards(lat.handle) == 0
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_a_batch_without_scratch(fail_alloc):
    rhos = [inputs.noisy_density(nx, ny, seed=nx, mean=0.7, amp=0.01, mode="rel")
            for nx, ny in ((96, 80), (131, 67))]
    got = []
    for fail in (-1, NEEDED, 2 * NEEDED + 1):
        fail_alloc(fail)
        with Batch(rhos, G1=-5.0, G2=[0.6, 0.3], trace_every=4) as b:
            fail_alloc(-1)
            b.step(27)
            got.append([(*b.fields(i), b.trace(i)) for i in range(2)])
    for other in got[1:]:
        for one, two in zip(got[0], other):
            for a, c in zip(one, two):
                assert np.array_equal(a, c)


def test_an_adjoint_without_scratch(fail_alloc):
    """Takes the two passes instead of the held reverse sweep: equal within the FP32 error of
    either (bars as between the two in test_gpu_adjoint_odd.py)."""
    rho0, target = (inputs.noisy_density(96, 80, s, mean=0.7, amp=0.01, mode="rel") for s in (1, 2))
    got = []
    for fail in (-1, NEEDED):
        fail_alloc(fail)
        with Lattice(rho0, G1=-5.0, G2=0.5, trace_every=0) as lat:
            fail_alloc(-1)
            got.append(lat.adjoint(30, target))
    (J, g, gG), (Jt, gt, gGt) = got
    assert abs(J - Jt) <= 2e-6 * abs(Jt)
    assert np.linalg.norm(g - gt) <= 1e-4 * np.linalg.norm(gt)
    for k in range(2):
        assert abs(gG[k] - gGt[k]) <= 1e-4 * abs(gGt[k])
