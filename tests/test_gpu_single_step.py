"""Problems that can run many steps per launch do so where it is the shorter way: not in calls of one step, and
beside problems that go step by step only where they would lengthen the step graph.  The chains are the same
whatever the calls' lengths."""
import numpy as np
import pytest

from paper_2501_17334_gb300 import workload as W

pytestmark = pytest.mark.gpu

LENGTHS = (1, 5, 1, 1, 2, 1, 17, 1)


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("sizes", [[(1, 64)], [(2, 300)], [(1, 100), (3, 300), (2, 257), (4, 33)], [(1, 5), (2, 9)]])
def test_calls_of_any_length(qst, cuda_ok, graph, sizes):
    probs = [W.config_problem(q, num_chains=R) for q, R in sizes]
    kw = dict(precision=qst.PREC_PAULI, use_graph=graph, thin=2, burn_in=3, diag_chains=4, traj_capacity=20, acf_lmax=3,
              adapt_interval=6, trace_steps=29)
    with qst.Sampler(probs, **kw) as a, qst.Sampler(probs, **kw) as b:
        for n in LENGTHS:
            a.run_chains(n)
        b.run_chains(sum(LENGTHS))
        for i in range(len(probs)):
            x, y = a.get_state(i), b.get_state(i)
            assert all(np.array_equal(x[k], y[k]) for k in x)
            assert np.array_equal(a.posterior_sum(i)[0], b.posterior_sum(i)[0])
            assert np.array_equal(a.diagnostics(i)["tau"], b.diagnostics(i)["tau"])
            for u, v in zip(a.get_trace(i), b.get_trace(i)):
                assert np.array_equal(u, v)


@pytest.mark.parametrize("sizes, steps, multi", [
    ([(1, 64)], 1, False), ([(1, 64)], 2, True), ([(2, 65536)], 2, False), ([(2, 65536)], 3, True),
    ([(1, 64), (2, 64)], 2, False), ([(1, 64), (2, 64)], 3, True), ([(1, 64), (2, 64)], 40, True),
    ([(1, 500), (2, 500), (3, 500), (4, 500)], 10, False), ([(1, 17)] * 20 + [(3, 40)], 3, False),
    ([(1, 17)] * 20 + [(3, 40)], 12, True), ([(1, 65536), (3, 40)], 8, True)])
def test_which_launches(qst, cuda_ok, sizes, steps, multi):
    """Three kernels a problem and step, or two a problem (steps, pooling) and one for the counters; the
    same chains as with kernel timing, which takes the per-step kernels."""
    probs = [W.config_problem(q, num_chains=R) for q, R in sizes]
    kw = dict(precision=qst.PREC_PAULI, diag_chains=0, thin=2)
    with qst.Sampler(probs, **kw) as s, qst.Sampler(probs, **kw) as plain:
        plain.set_profiling(True)
        before = s.launch_count()
        s.run_chains(steps)
        small = sum(q <= 2 for q, _ in sizes)
        want = small * 2 + 1 + 3 * steps * (len(sizes) - small) if multi else 3 * steps * len(sizes)
        assert s.launch_count() - before == want
        s.run_chains(3)
        plain.run_chains(steps + 3)
        for i in (0, len(sizes) - 1):
            x, y = s.get_state(i), plain.get_state(i)
            assert all(np.array_equal(x[k], y[k]) for k in x)
            assert np.array_equal(s.posterior_sum(i)[0], plain.posterior_sum(i)[0])
