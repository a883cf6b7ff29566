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
