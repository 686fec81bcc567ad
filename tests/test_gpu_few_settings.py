"""Many-step launches with fewer settings than lanes per chain: every lane of a chain takes the same
decision.  Random bases of one to three settings (and more than a chain's lanes), below and just past each
line between 4 D, 2 D and D lanes per chain, against the per-step kernels: same bits."""
import numpy as np
import pytest

from paper_2501_17334_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q, chains", [(1, 40), (1, 2561), (1, 20481), (2, 40), (2, 4097), (2, 7169)])
@pytest.mark.parametrize("settings", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("poisson", [False, True])
def test_few_settings(qst, cuda_ok, q, chains, settings, poisson):
    prob = W.random_basis_problem(q, settings, num_chains=chains)
    if poisson:   # the same counts as Poisson ones
        prob.likelihood = qst.LIKELIHOOD_POISSON
        prob.trials = np.full(settings, 1000.0)
    many, plain = (qst.Sampler(prob, diag_chains=0, adapt_interval=5) for _ in range(2))
    plain.set_profiling(True)   # per-step kernels
    for s in (many, plain):
        s.run_chains(12)
    a, b = many.get_state(), plain.get_state()
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    assert np.array_equal(many.posterior_sum()[0], plain.posterior_sum()[0])
    many.close()
    plain.close()
