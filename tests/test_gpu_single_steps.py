"""The kernels of steps that are a launch of their own (k_step, k_step_total, k_step_batch with
k_batch_reduce): one step a call, which never shares a launch, at every CTA width, on grids
of many short and of few long CTA rows, against the oracle (bars as in test_gpu_parity.py) and bit for
bit against the same steps in one call."""
import numpy as np
import pytest

import oracle
from paper_1008_2865_gb300 import Batch, Lattice, capi, inputs

pytestmark = pytest.mark.gpu


def _err(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


def _rows_err(tr, ref):
    return float(np.max(np.abs(tr[:, 1:] - ref[:, 1:]) / np.abs(ref[:, 1:])))


def _run(make, steps, each, launch=None):
    with make() as lat:
        if launch:
            lat.set_launch(*launch)
        for _ in range(steps // each):
            lat.step(each)
        lat.step(steps % each)
        assert lat.t == steps and capi.lb_check_guards(lat.handle) == 0
        return (*lat.fields(), lat.trace(), lat.save())


def _same(one, two):
    for a, b in zip(one, two):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("nx,ny,launch", [
    (301, 170, (64, 16, 0)), (301, 170, (96, 17, 0)), (301, 170, (128, 16, 0)),
    (301, 170, (192, 40, 0)), (301, 170, (256, 33, 0)),
    (130, 2000, (64, 4, 0)), (61, 997, (64, 5, 0)), (4000, 9, (256, 4, 0)), (4000, 9, (192, 4, 0))])
def test_single_steps_at_every_launch_shape(nx, ny, launch):
    rho0 = inputs.noisy_density(nx, ny, seed=9, mean=0.7, amp=0.01, mode="rel")
    ref = oracle.run(rho0, 30, G1=-5.0, G2=0.6, trace_every=10)

    def make():
        return Lattice(rho0, G1=-5.0, G2=0.6, trace_every=10)

    got = _run(make, 30, 1, launch)
    rho, ux, uy, tr, _ = got
    assert _err(rho, ref[0]) <= 1e-5 and _err(ux, ref[1]) <= 1e-5 and _err(uy, ref[2]) <= 1e-5
    assert len(tr) == 3 and np.array_equal(tr[:, 0], ref[3][:, 0])
    assert _rows_err(tr, ref[3]) <= 1e-4
    assert np.max(np.abs(tr[:, 1] - ref[3][:, 1]) / ref[3][:, 1]) <= 1e-6
    _same(got, _run(make, 30, 30, launch))


@pytest.mark.parametrize("launch", [None, (64, 8, 0), (96, 16, 0), (128, 72, 0), (192, 40, 0),
                                    (256, 33, 0)])
@pytest.mark.parametrize("nx,ny,prec,omega", [(2050, 1000, "fp32", 1.0), (1301, 1400, "fp32", 0.8),
                                              (1301, 1400, "fp16_delta", 1.0)])
def test_trace_rows_of_an_alternating_march(nx, ny, prec, omega, launch):
    """A lattice beyond L2 marches down in even row chunks and up in odd ones; its paired steps'
    trace rows (trace_tile, both directions) against those of k_step's reduction steps."""
    rho0 = inputs.noisy_density(nx, ny, seed=nx, mean=0.7, amp=0.01, mode="rel")

    def make():
        return Lattice(rho0, omega=omega, G1=-5.0, G2=0.6, prec=prec, trace_every=4)

    _same(_run(make, 11, 1, launch), _run(make, 11, 11, launch))


@pytest.mark.parametrize("launch", [(64, 16), (96, 24), (128, 72), (192, 40), (256, 48)])
@pytest.mark.parametrize("prec,om", [("fp32", 1.0), ("fp16_delta", 0.9)])
def test_batch_at_every_launch_shape(launch, prec, om):
    """Replicas stepped one step a call (k_step_batch), in one call (pairs and the period's
    graph), and alone one step a call (k_step): the same bits; one replica alternates."""
    shapes = [(64, 48), (131, 67), (1537, 1200), (300, 40), (5, 5)]
    g2 = [0.0, 0.3, 0.6, 0.9, 0.45]
    rhos = [inputs.noisy_density(nx, ny, seed=nx, mean=0.7, amp=0.01, mode="rel") for nx, ny in shapes]
    omega = [om] + [1.0] * 4
    got = []
    for each in (1, 13):
        with Batch(rhos, omega=omega, G1=-5.0, G2=g2, prec=prec, trace_every=4) as b:
            b.set_launch(launch[0], launch[1], 1)
            for _ in range(13 // each):
                b.step(each)
            assert capi.lb_batch_check_guards(b.handle) == 0
            got.append([(*b.fields(i), b.trace(i)) for i in range(5)])
    for one, two in zip(*got):
        _same(one, two)
    for i, rho0 in enumerate(rhos):
        alone = _run(lambda: Lattice(rho0, omega=omega[i], G1=-5.0, G2=g2[i], prec=prec,
                                     trace_every=4), 13, 1, (launch[0], launch[1], 0))
        _same(got[0][i], alone[:4])
