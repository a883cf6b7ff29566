"""Energies, objective and its derivatives of states whose psi is far beyond the range in which
FP32 carries products of two (|psi| of 1e20 and 1e-20, couplings of 1e30), and of a state with an
infinite psi: the sums have the range of FP64. The reference takes the same FP32 psi in FP64
throughout; the kernels' class sums are FP32 sums of at most 9 values of one sign and the
couplings are FP32, so the sums agree to (8 + 1) 2^-24 < 1e-6. The misfit of the state's own
density, which the objective forms again from FP32 populations, is at most N (9 2^-24 rho)^2."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1008_2865_gb300 import Lattice, capi, inputs

pytestmark = pytest.mark.gpu

NX, NY = 70, 45
BAR = 1e-6


def _psi_bytes(saved):
    """The view of a saved state's psi deviations (its last N floats)."""
    return saved[-4 * NX * NY:].view(np.float32).reshape(NY, NX)


def _state(scale, G1, G2, prec):
    """A state at t = 0 with psi = scale (1 + 1%), and that psi."""
    rho0 = inputs.noisy_density(NX, NY, seed=4, mean=min(scale, 0.7), amp=0.01, mode="rel")
    lat = Lattice(rho0, G1=G1, G2=G2, prec=prec, trace_every=0)
    mean = float(np.float32(rho0.mean()))
    psi_ref = np.float32(-np.expm1(-mean))
    saved = np.frombuffer(bytes(lat.save()), dtype=np.uint8).copy()
    dpsi = _psi_bytes(saved)
    if scale > 1.0:
        dpsi[...] = (scale * (1.0 + 0.01 * np.random.default_rng(1).uniform(-1, 1, (NY, NX))))
        lat.load(saved)
    return lat, rho0, float(psi_ref) + dpsi.astype(np.float64)


@pytest.mark.parametrize("prec", ["fp32", "fp16_delta"])
@pytest.mark.parametrize("scale,G1,G2", [(0.5, -5.0, 0.6), (1e20, -5.0, 0.6), (1e-20, -5.0, 0.6),
                                         (0.5, -5e30, 6e29), (0.5, -5e-30, 6e-31),
                                         (1e20, -5e-18, 6e-19), (1e-20, -5e18, 6e17)])
def test_energy_and_objective_have_the_range_of_fp64(scale, G1, G2, prec):
    lat, rho0, psi = _state(scale, G1, G2, prec)
    with lat:
        es, em, eb, mass = lat.energy()
        want = oracle.energy(psi, G1, G2)
        for got, ref in zip((es, em, eb), want):
            assert abs(got - ref) <= BAR * abs(ref)
        rho = lat.fields()[0]
        assert abs(mass - rho.sum()) <= BAR * rho.sum()
        J = lat.objective(rho)
        misfit = NX * NY * (9 * 2.0 ** -24 * rho.max()) ** 2
        E = want[0] + want[1]
        assert abs(J - E) <= BAR * (abs(want[0]) + abs(want[1])) + misfit
        if prec == "fp32":
            # without steps the adjoint gives the objective and its explicit derivatives
            Ja, _, gG = lat.adjoint(0, rho)
            assert Ja == J
            for got, (a, b) in zip(gG, ((1.0, 0.0), (0.0, 1.0))):
                s, m, _ = oracle.energy(psi, a, b)
                assert abs(got - (s + m)) <= BAR * (abs(s) + abs(m))
    # the sums of a state in range are unchanged by one that was not
    lat, rho0, psi = _state(0.5, -5.0, 0.6, prec)
    with lat:
        assert lat.energy() == lat.energy()


@pytest.mark.parametrize("prec", ["fp32", "fp16_delta"])
def test_an_infinite_psi_gives_infinite_energies(prec):
    lat, _, _ = _state(0.5, -5.0, 0.6, prec)
    with lat:
        saved = np.frombuffer(bytes(lat.save()), dtype=np.uint8).copy()
        _psi_bytes(saved)[7, 9] = np.inf
        lat.load(saved)
        out = (ctypes.c_double * 4)()
        st = capi.load().lb_energy(ctypes.c_void_p(lat.handle), out)
        assert st == capi.LB_ERR_NONFINITE
        assert out[0] == -np.inf and out[1] == np.inf and out[2] == -np.inf
        assert np.isfinite(out[3])
