"""1D FP64 runs of 8 and 16 points (csrc/run1d64.cu), where threads without a mode
of their own stand by: they have no part in the result, so that a run's bits do
not depend on how its steps are split into calls.  All of u0 sits in mode -1 (the
last of the array), from where a potential spreads it: the other modes' scale
falls below what an idle thread's copy of that mode would keep."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 16])
@pytest.mark.parametrize("seed", range(4))
def test_idle_threads_leave_no_trace(n, seed):
    from paper_2001_06113_gb300 import Problem
    rng = np.random.default_rng(seed)
    x = -np.pi + 2.0 * np.pi * np.arange(n) / n
    V = 12.0 * np.cos(x + rng.uniform(0, 6)) + 5.0 * np.cos(2 * x + rng.uniform(0, 6))
    u0 = np.exp(-1j * x)
    got = []
    for calls in ([60], [12] + [1] * 48, [7, 13, 20, 20]):
        with Problem((n,), 4e-3, 60, order=8) as p:
            p.set_potential(V)
            p.set_initial(u0)
            for k in calls:
                p.step(k)
            got.append((p.read_u(0), p.read_modes(0)))
    for u, m in got[1:]:
        assert np.array_equal(u, got[0][0]) and np.array_equal(m, got[0][1])
