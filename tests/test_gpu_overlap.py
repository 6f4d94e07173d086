"""Passes that do not overlap (tdse_set_overlap) give the same bits: one FP64 and one
mixed problem in 2D and 3D, and the four-step 1D layout."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,kw", [((64, 128), {}), ((16, 32, 16), {}), ((1024,), {"layout_1d": "passes"})])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_overlap_keeps_bits(shape, kw, precision):
    import synth
    from paper_2001_06113_gb300 import Problem
    d = tuple([1.0] + [0.0] * (len(shape) - 1))
    inst = synth.random_periodic(shape, 5, 1e-3, 12, pulse=synth.Pulse(2.0, 10.0, 0.05, d))
    got = []
    for on in (True, False):
        with Problem(shape, inst.dt, inst.nsteps, precision=precision, **kw) as p:
            p.set_overlap(on)
            p.set_potential(inst.V0, inst.vfac_table())
            q = inst.pulse
            p.set_pulse(q.A0, q.omega, q.T_pulse, q.direction)
            p.set_initial(inst.u0)
            p.step(12)
            got.append(p.read_u(0))
    assert np.array_equal(*got)
