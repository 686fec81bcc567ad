"""One- and two-qubit problems run many steps per launch; kernel timing takes the per-step kernels.
Both give the same bits: chains, decisions, log L, pooled sums, trajectories, at the edges of a
CTA (16 or 8 chains), of a pool slot (128 chains) and of a launch (512 kept steps)."""
import numpy as np
import pytest

from paper_2501_17334_gb300 import workload as W

pytestmark = pytest.mark.gpu


def _pair(probs, **kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2501_17334_gb300 import qst
    many, plain = (qst.Sampler(probs, **kw) for _ in range(2))
    plain.set_profiling(True)
    return many, plain


def _same(many, plain, n):
    for i in range(n):
        a, b = many.get_state(i), plain.get_state(i)
        for k in a:
            assert np.array_equal(a[k], b[k]), (i, k)
        assert np.array_equal(many.posterior_sum(i)[0], plain.posterior_sum(i)[0])
        da, db = many.diagnostics(i), plain.diagnostics(i)
        assert np.array_equal(da["tau"], db["tau"]) and da["num_kept"] == db["num_kept"]
        if many.cfg.trace_steps:
            for x, y in zip(many.get_trace(i), plain.get_trace(i)):
                assert np.array_equal(x, y)


@pytest.mark.parametrize("form", ["FP32", "PAULI"])
@pytest.mark.parametrize("q, chains, prior", [(1, 1, 0), (1, 17, 0), (1, 128, 1), (1, 300, 0), (2, 7, 0), (2, 129, 0),
                                              (2, 64, 1), (2, 1000, 0)])
def test_many_steps_match_single_steps(form, q, chains, prior):
    from paper_2501_17334_gb300 import qst
    many, plain = _pair(W.config_problem(q, num_chains=chains), precision=getattr(qst, "PREC_" + form), prior=prior,
                        thin=3, burn_in=5, adapt_interval=7, diag_chains=4, traj_capacity=16, acf_lmax=4, trace_steps=30)
    for n in (20, 1, 2, 38):
        many.run_chains(n)
        plain.run_chains(n)
    _same(many, plain, 1)
    buf = many.checkpoint()          # a restored handle goes on from there in either way
    plain.restore(buf)
    many.run_chains(9)
    plain.run_chains(9)
    _same(many, plain, 1)


@pytest.mark.parametrize("form", ["FP32", "PAULI"])
@pytest.mark.parametrize("q, chains", [(1, 2561), (1, 8193), (1, 20481), (2, 2049), (2, 4097), (2, 7169)])
def test_every_number_of_lanes_per_chain(form, q, chains):
    """Just past each line between 4 D, 2 D and D lanes per chain."""
    from paper_2501_17334_gb300 import qst
    many, plain = _pair(W.config_problem(q, num_chains=chains), precision=getattr(qst, "PREC_" + form), diag_chains=0)
    for s in (many, plain):
        s.run_chains(12)
    _same(many, plain, 1)


@pytest.mark.parametrize("poisson", [False, True])
def test_runs_longer_than_a_launch(poisson):
    """600 kept steps (512 fit one launch), multinomial and Poisson counts."""
    prob = W.lossy_pauli_problem(1, 40) if poisson else W.config_problem(1, num_chains=40)
    many, plain = _pair(prob, diag_chains=2, traj_capacity=700, acf_lmax=20)
    many.run_chains(600)
    plain.run_chains(600)
    _same(many, plain, 1)


def test_beside_problems_that_go_step_by_step():
    """Small problems of a handle run on their own branches beside the others, in graph and plain steps."""
    from paper_2501_17334_gb300 import qst
    probs = [W.config_problem(q, num_chains=R) for q, R in [(1, 100), (3, 300), (2, 257), (1, 33)]]
    for graph in (0, 1):
        many, plain = _pair(probs, precision=qst.PREC_PAULI, use_graph=graph, thin=2, diag_chains=4, traj_capacity=30,
                            acf_lmax=3)
        for n in (25, 4):
            many.run_chains(n)
            plain.run_chains(n)
        _same(many, plain, len(probs))


def test_an_odd_povm_and_an_invalid_state():
    """Eleven Haar-random settings; a chain whose latent state turns NaN rejects everything."""
    many, plain = _pair(W.random_basis_problem(2, 11, num_chains=50), diag_chains=0)
    for s in (many, plain):
        s.run_chains(10)
        s.inject_nan(13)
        s.run_chains(10)
    a, b = many.get_state(), plain.get_state()
    assert np.array_equal(a["y"], b["y"], equal_nan=True) and np.array_equal(a["accepts"], b["accepts"])
    assert np.array_equal(many.posterior_sum()[0], plain.posterior_sum()[0])
