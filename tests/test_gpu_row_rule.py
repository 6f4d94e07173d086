"""2D mixed batches whose intermediates exceed the L2 take the shared-memory row pass
for 512-point lines, smaller ones the register pass (csrc/periodic2d.cuh): the same
bits, in an uneven split of the instances into step groups too."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n0,batch", [(64, 230), (512, 29), (8, 1832)])
def test_batches_beyond_the_l2_keep_their_bits(n0, batch):
    import torch
    import synth
    from paper_2001_06113_gb300 import Problem
    shape, n = (n0, 512), 12
    assert n0 * 512 * batch * 16 > 120e6
    inst = synth.random_periodic(shape, 3, 1e-3, n, pulse=synth.Pulse(2.0, 10.0, 0.05, (1.0, 0.5)))
    out = []
    for b in (1, batch):
        with Problem(shape, inst.dt, n, precision="mixed", batch=b) as p:
            p.set_potential(inst.V0, inst.vfac_table())
            q = inst.pulse
            p.set_pulse(q.A0, q.omega, q.T_pulse, q.direction)
            p.set_initial(inst.u0)
            p.step(n)
            out.append([p.read_u(i) for i in {0, b // 2, b - 1}])
        torch.cuda.empty_cache()
    for u in out[1]:
        assert np.array_equal(u, out[0][0])
