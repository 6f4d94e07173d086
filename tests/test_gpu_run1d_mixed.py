"""1D mixed runs in one launch (csrc/run1d32.cu): the oracle's result at the
edges of the kernel's range (n = 8 has one transform pass and no barrier in it,
16 two, 8192 the largest) and the same bits however the steps are split into
calls."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _solve(inst, order, calls):
    from paper_2001_06113_gb300 import Problem
    with Problem(inst.shape, inst.dt, inst.nsteps, order=order, batch=3, precision="mixed") as p:
        p.set_potential(inst.V0, inst.vfac_table())
        q = inst.pulse
        p.set_pulse(q.A0, q.omega, q.T_pulse, q.direction)
        p.set_initial(inst.u0)
        for k in calls:
            p.step(k)
        return p.read_u()


@pytest.mark.parametrize("n,order", [(8, 8), (8, 4), (16, 8), (16, 2), (8192, 8)])
def test_run_matches_oracle_and_its_pieces(n, order):
    import synth
    from oracle.periodic import oracle_for, rel_l2
    inst = synth.random_periodic((n,), 11 + n, 2e-3, 40, pulse=synth.Pulse(2.0, 10.0, 0.05, (1.0,)))
    u = _solve(inst, order, [40])
    ref = oracle_for(inst, order=order).solve(inst.u0, 40)
    assert rel_l2(u[0], ref) <= 1e-5
    assert np.array_equal(u[0], u[1]) and np.array_equal(u[0], u[2])
    v = _solve(inst, order, [1, 2, 5, 1, 3, 20, 8])
    assert np.array_equal(u, v)
