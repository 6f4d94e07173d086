"""Fields in free space: a field set inside a captured graph (its phase tables and
their scale belong together, whatever is set between capture and replay)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("A0", [150.0, 400.0])       # scale 3; FP64 phases
def test_pulse_set_in_a_captured_graph(A0):
    import torch
    import synth
    from paper_2001_06113_gb300 import Problem
    n, H = 6, 2.0
    strong = synth.free_bump_gaussians((64,), seed=2, dt=1e-3, nsteps=n, A0=A0)
    q = strong.pulse

    def solve(p):
        p.set_initial(strong.u0)
        p.step(n)
        return p.read_u(0)

    stream = torch.cuda.Stream()
    with Problem((64,), 1e-3, n, order=4, bc="free", nu=(512,), H=H, stream=stream) as p:
        p.set_potential(strong.V0)
        p.set_pulse(q.A0, q.omega, q.T_pulse, q.direction)
        ref = solve(p)
        p.set_pulse(1.0, q.omega, q.T_pulse, q.direction)
        weak = solve(p)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            p.set_pulse(q.A0, q.omega, q.T_pulse, q.direction)
        p.set_pulse(1.0, q.omega, q.T_pulse, q.direction)
        assert np.array_equal(solve(p), weak)
        with torch.cuda.stream(stream):
            graph.replay()
        assert np.array_equal(solve(p), ref)


def _oracle(inst, M, R, H, r, d, relative=0.0):
    """u, u^ and phi(t) = r/2 (1 - cos(2 pi t / 4 dt)) per axis; `relative`:
    random relative errors of the transforms' entries, which show how far
    rounding errors of that size carry."""
    import math
    from oracle import gamma
    from oracle.freespace import FreeSpaceOracle
    w = 2.0 * math.pi / (4.0 * inst.dt)
    o = FreeSpaceOracle([gamma.GammaRule.for_nu(M, M * R, H)] * d, inst.dt, inst.V0, inst.vfac,
                        lambda t: np.full(d, 0.5 * r * (1.0 - math.cos(w * t))), order=4)
    rng = np.random.default_rng(0)
    o.F = [f * (1.0 + relative * rng.uniform(-1, 1, f.shape)) for f in o.F]
    o.G = [g * (1.0 + relative * rng.uniform(-1, 1, g.shape)) for g in o.G]
    u = o.solve(inst.u0, inst.nsteps)
    return u, o.last_uhat, lambda t: [0.5 * r * w * math.sin(w * t)] * d


# Scales 2 and 4 (fixed-point factors), then FP64 phases: just past the line, 2^30
# over the history, and one-step phases of 2^26.
@pytest.mark.parametrize("d,M,H,r,g", [(1, 64, 2.0, 0.25, 2), (1, 64, 2.0, 0.49, 4), (1, 64, 2.0, 0.6, 5), (1, 64, 2.0, 3.0, 5),
                                       (1, 128, 4.5, 8.0, 5), (2, 32, 2.0, 0.12, 2), (2, 32, 2.0, 0.6, 5), (2, 32, 2.178, 4.0, 5)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_strong_field_matches_oracle(d, M, H, r, g, precision):
    import struct
    import synth
    from paper_2001_06113_gb300 import Problem
    R, n = 8, 6
    inst = synth.free_bump_gaussians((M,) * d, seed=2, dt=1e-3, nsteps=n, A0=1.0)
    u, m, A = _oracle(inst, M, R, H, r, d)
    v, k, _ = _oracle(inst, M, R, H, r, d, 2.0 ** -50)

    def rel(a, b):
        return float(np.linalg.norm(a - b) / np.linalg.norm(b))

    # rounding errors of 2^-50 (2^-21) per entry, a hundred of them, and the phases' own
    scale, floor = (1.0, 1e-12) if precision == "fp64" else (2.0 ** 29, 2e-6)
    tol_u, tol_m = (100.0 * rel(x, y) * scale + floor for x, y in ((v, u), (k, m)))
    with Problem((M,) * d, inst.dt, n, order=4, bc="free", nu=(M * R,) * d, H=H, precision=precision, batch=2) as p:
        p.set_potential(inst.V0)
        p.set_vector_potential(A, instance=1)
        p.set_initial(inst.u0)
        p.step(n)
        got_u, got_m, blob = p.read_u(1), p.read_modes(1), p.save()
    if tol_m < 0.1:
        assert rel(got_m, m) <= tol_m
    if tol_u < 0.1:
        assert rel(got_u, u) <= tol_u
    flags = len(blob) - struct.unpack_from("<Q", blob, 88)[0] - 4      # two instances, two bytes each
    assert (blob[flags] >> 1) - 1 == 0 and (blob[flags + 2] >> 1) - 1 == g


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_fp64_phases_alone_in_a_batch_and_resumed(precision):
    import synth
    from paper_2001_06113_gb300 import Problem
    n = 8
    weak, strong = (synth.free_bump_gaussians((64,), seed=s, dt=1e-3, nsteps=n, A0=a) for s, a in ((1, 1.0), (2, 400.0)))

    def problem(batch=1):
        return Problem((64,), 1e-3, n, order=4, batch=batch, bc="free", nu=(512,), H=2.0, precision=precision)

    def setup(p, inst, i=-1):
        q = inst.pulse
        p.set_potential(inst.V0, instance=i)
        p.set_pulse(q.A0, q.omega, q.T_pulse, q.direction, instance=i)
        p.set_initial(inst.u0, instance=i)

    with problem(2) as p:
        setup(p, weak, 0)
        setup(p, strong, 1)
        p.step(n)
        both = p.read_u()
    for i, inst in enumerate((weak, strong)):
        with problem() as p:
            setup(p, inst)
            p.step(5)
            blob = p.save()
            p.step(3)
            assert np.array_equal(p.read_u(0), both[i])
        with problem() as p:
            p.load(blob)
            p.step(3)
            assert np.array_equal(p.read_u(0), both[i])
