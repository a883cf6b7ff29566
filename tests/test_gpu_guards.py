"""Every device buffer of a state has guards of its own: the control words (results, error
flags, trace count, input flag, arrival counters), partial sums, trace ring, populations, psi
and, where the state has them, its density deviations, the halo words and the buffers of kept
states. One damaged guard after another is reported, and no buffer shares another's."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,prec,omega,trace,buffers", [
    (96, 80, "fp32", 1.0, 0, 13),           # 5 control words, 2, 4 fields, 2 sets of halo words
    (96, 80, "fp16_delta", 0.9, 5, 17),     # deviations, counters, partial sums, kept states
    (1000, 700, "fp32", 1.0, 5, 12),        # not held
    (96, 80, "fp64", 1.0, 5, 11)])
def test_every_buffer_is_guarded(nx, ny, prec, omega, trace, buffers):
    from paper_1008_2865_gb300 import LBError, Lattice, capi, inputs
    rho0 = inputs.noisy_density(nx, ny, seed=1, mean=0.7, amp=0.01, mode="rel")
    with Lattice(rho0, omega=omega, prec=prec, trace_every=trace) as lat:
        lat.step(12)
        lat.energy()
        assert capi.lb_check_guards(lat.handle) == 0
        for k in range(buffers):
            capi.lb_debug_damage_guard(lat.handle, k)
            assert capi.lb_check_guards(lat.handle) == k + 1
        with pytest.raises(LBError):
            capi.lb_debug_damage_guard(lat.handle, buffers)
