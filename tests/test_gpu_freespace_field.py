"""Fields in free space: a field set inside a captured graph (its phase tables and
their scale belong together, whatever is set between capture and replay)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_pulse_set_in_a_captured_graph():
    import torch
    import synth
    from paper_2001_06113_gb300 import Problem
    n, H = 6, 2.0
    strong = synth.free_bump_gaussians((64,), seed=2, dt=1e-3, nsteps=n, A0=150.0)
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
