"""A stream that has only some of the GPU's SMs (of a green context) refuses the cooperative
launch that holds a small lattice: the steps are taken all the same, with the same fields and
trace bit for bit, and the adjoint takes its two passes."""
import ctypes

import numpy as np
import pytest

from paper_1008_2865_gb300 import Lattice, inputs

pytestmark = pytest.mark.gpu


class _Resource(ctypes.Structure):
    _fields_ = [("type", ctypes.c_int), ("pad", ctypes.c_ubyte * 92), ("sm_count", ctypes.c_uint),
                ("rest", ctypes.c_ubyte * 512)]


@pytest.fixture(scope="module")
def share():
    """A stream with 16 SMs."""
    import torch
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")

    def call(name, *args):
        if getattr(cu, name)(*args) != 0:
            pytest.skip(f"{name}: no green contexts here")

    dev = ctypes.c_int()
    whole, part, rest = _Resource(), _Resource(), _Resource()
    groups = ctypes.c_uint(1)
    desc, ctx, stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    call("cuDeviceGet", ctypes.byref(dev), 0)
    call("cuDeviceGetDevResource", dev, ctypes.byref(whole), 1)
    call("cuDevSmResourceSplitByCount", ctypes.byref(part), ctypes.byref(groups), ctypes.byref(whole),
         ctypes.byref(rest), 0, 16)
    call("cuDevResourceGenerateDesc", ctypes.byref(desc), ctypes.byref(part), 1)
    call("cuGreenCtxCreate", ctypes.byref(ctx), desc, dev, 1)
    call("cuGreenCtxStreamCreate", ctypes.byref(stream), ctx, 1, 0)
    yield stream.value
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("nx,ny,prec,omega", [(300, 200, "fp32", 1.0), (640, 600, "fp32", 1.0),
                                              (301, 199, "fp16_delta", 0.9)])
def test_steps_on_a_share_of_the_sms(share, nx, ny, prec, omega):
    rho0 = inputs.noisy_density(nx, ny, seed=5, mean=0.7, amp=0.01, mode="rel")
    got = []
    for stream in (0, share):
        with Lattice(rho0, omega=omega, G1=-5.0, G2=0.6, prec=prec, trace_every=5,
                     stream=stream) as lat:
            lat.step(11)
            lat.step(10)
            assert lat.t == 21
            got.append((*lat.fields(), lat.trace(), lat.save()))
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_adjoint_on_a_share_of_the_sms(share):
    """Bars as between the held reverse sweep and the two passes (test_gpu_adjoint_odd.py)."""
    rho0, target = (inputs.noisy_density(300, 200, s, mean=0.7, amp=0.01, mode="rel") for s in (1, 2))
    got = []
    for stream in (0, share):
        with Lattice(rho0, G1=-5.0, G2=0.5, trace_every=0, stream=stream) as lat:
            got.append(lat.adjoint(20, target))
    (J, g, gG), (Jt, gt, gGt) = got
    assert abs(J - Jt) <= 2e-6 * abs(Jt)
    assert np.linalg.norm(g - gt) <= 1e-4 * np.linalg.norm(gt)
    for k in range(2):
        assert abs(gG[k] - gGt[k]) <= 1e-4 * abs(gGt[k])
