"""The adjoint of lattices that the small ones do not stand for: too large for the SMs with omega
= 1 (paired forward steps, single recomputation, two passes whose grids stride over the sites)
and with another omega, an odd width, and the largest that are held. Bars as in test_gpu_adjoint.py
(J 1e-6, gradients 1e-4); any checkpoint spacing gives the same bits."""
import numpy as np
import pytest

import oracle
from paper_1008_2865_gb300 import Lattice, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,omega", [(901, 760, 1.0), (600, 641, 0.8), (680, 684, 1.0)])
def test_adjoint_of_a_large_lattice(nx, ny, omega):
    steps = 10
    r0 = inputs.noisy_density(nx, ny, 11, mean=0.7, amp=0.01, mode="rel")
    tgt = inputs.noisy_density(nx, ny, 12, mean=0.7, amp=0.01, mode="rel")
    Jo, go, gGo = oracle.gradient(r0, tgt, steps, omega=omega, G1=-5.0, G2=0.5)
    with Lattice(r0, omega=omega, G1=-5.0, G2=0.5, trace_every=0) as lat:
        lat.step(steps)
        forward, J0 = lat.fields(), lat.objective(tgt)
    got = []
    for every in (0, 5, 10):
        with Lattice(r0, omega=omega, G1=-5.0, G2=0.5, trace_every=0) as lat:
            J, g, gG = lat.adjoint(steps, tgt, checkpoint_every=every)
            for a, b in zip(lat.fields(), forward):
                assert np.array_equal(a, b)
        assert J == J0
        got.append((J, g, gG))
        assert abs(J - Jo) <= 1e-6 * abs(Jo)
        assert np.linalg.norm(g - go) <= 1e-4 * np.linalg.norm(go)
        for k in range(2):
            assert abs(gG[k] - gGo[k]) <= 1e-4 * abs(gGo[k])
    for J, g, gG in got[1:]:
        assert J == got[0][0] and gG == got[0][2] and np.array_equal(g, got[0][1])
