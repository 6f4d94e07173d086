"""Free-space line transforms (csrc/freespace.cuh) at the edges of their range:
every grid length and nu / n built (the folded 512-point lines, the lines whose
two sides have different widths), with a potential and a field, against the
oracle; a strong field, whose phase factors need a larger scale, alone and in
a batch; a checkpoint without the scale in its flags."""
import struct

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _problem(M, R, H, precision, n, batch=1):
    from paper_2001_06113_gb300 import Problem
    return Problem((M,), 1e-3, n, order=4, batch=batch, bc="free", nu=(M * R,), H=H, precision=precision)


def _setup(p, inst, i=-1):
    q = inst.pulse
    p.set_potential(inst.V0, instance=i)
    p.set_pulse(q.A0, q.omega, q.T_pulse, q.direction, instance=i)
    p.set_initial(inst.u0, instance=i)


@pytest.mark.parametrize("M,R", [(32, 4), (32, 16), (64, 8), (128, 4), (128, 16), (256, 4), (256, 16), (512, 4), (512, 8)])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 2e-6)])
def test_lines_match_oracle(M, R, precision, tol):
    import synth
    from oracle import fields, gamma
    from oracle.freespace import FreeSpaceOracle
    H, n = 1.0, 6
    inst = synth.free_bump_gaussians((M,), seed=M + R, dt=1e-3, nsteps=n, A0=5.0)
    o = FreeSpaceOracle([gamma.GammaRule.for_nu(M, M * R, H)], inst.dt, inst.V0, inst.vfac, fields.phi_callable(inst.pulse, 1),
                        order=4)
    ref = o.solve(inst.u0, n)
    with _problem(M, R, H, precision, n) as p:
        _setup(p, inst)
        p.step(n)
        u, m = p.read_u(0), p.read_modes(0)
    assert np.linalg.norm(u - ref) <= tol * np.linalg.norm(ref)
    assert np.linalg.norm(m - o.last_uhat) <= tol * np.linalg.norm(o.last_uhat)


def test_strong_field_alone_in_a_batch_and_resumed():
    import synth
    H, n = 2.0, 6
    weak = synth.free_bump_gaussians((64,), seed=1, dt=1e-3, nsteps=n, A0=1.0)
    strong = synth.free_bump_gaussians((64,), seed=2, dt=1e-3, nsteps=n, A0=150.0)
    with _problem(64, 8, H, "fp64", n, batch=2) as pb:
        _setup(pb, weak, 0)
        _setup(pb, strong, 1)
        pb.step(n)
        both = pb.read_u()
    for i, inst in enumerate((weak, strong)):
        with _problem(64, 8, H, "fp64", n) as p:
            _setup(p, inst)
            p.step(4)
            blob = p.save()
            p.step(2)
            assert np.array_equal(p.read_u(0), both[i])
        with _problem(64, 8, H, "fp64", n) as q:
            q.load(blob)
            q.step(2)
            assert np.array_equal(q.read_u(0), both[i])
        flags = len(blob) - struct.unpack_from("<Q", blob, 88)[0] - 2      # ws_bytes of the header
        old = blob[:flags] + bytes([blob[flags] & 1]) + blob[flags + 1:]
        assert blob[flags] > 1
        with _problem(64, 8, H, "fp64", n) as q:
            q.load(old)
            q.step(2)
            u = q.read_u(0)
        assert np.linalg.norm(u - both[i]) <= 1e-12 * np.linalg.norm(both[i])

