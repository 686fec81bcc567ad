"""Where two or four groups of lanes share a chain (few chains of three and four qubits; the many-step
launches of one and two), the lanes that hold one row of the refinement's triangular system read it before
any of them replaces it: the same bits as with one lane per row, ill-conditioned H (several passes of the
refinement) among the rows."""
import numpy as np
import pytest

from paper_2501_17334_gb300 import workload as W

from tests.test_gpu_refinement import _rows

pytestmark = pytest.mark.gpu


def _latent(q, rows, seed):
    """Prior draws, every third row with cond(H) from 1e2 to 3e5."""
    x = W.latent_batch(rows, q, seed).astype(np.float32)
    bad = _rows(q, [1e2, 3e4, 1e5, 3e5], (rows + 11) // 12, seed + 1)
    x[::3] = bad[np.random.default_rng(seed).permutation(len(bad))[: len(x[::3])]]
    return x


@pytest.mark.parametrize("q", [3, 4])
@pytest.mark.parametrize("rows", [1, 3, 65, 1001, 1215, 1216])
def test_two_groups_match_one(qst, cuda_ok, q, rows):
    import torch
    prob = W.config_problem(q, num_chains=rows)
    x = torch.from_numpy(_latent(q, rows, 900 + q)).cuda()
    two = qst.Sampler(prob, precision=qst.PREC_PAULI, diag_chains=0)   # up to 1216 rows: 32 / D chains a CTA
    got = two.evaluate(x)
    assert two.diagnostics()["propose_chains_per_cta"] == 32 >> q
    for threads in (32, 64, 128):                                      # a CTA size asked for: one group
        one = qst.Sampler(prob, precision=qst.PREC_PAULI, diag_chains=0, propose_threads=threads)
        assert one.diagnostics()["propose_chains_per_cta"] == threads >> q
        for a, b in zip(got, one.evaluate(x)):
            assert torch.equal(a, b)
        one.close()
    two.close()


@pytest.mark.parametrize("form", ["FP32", "PAULI"])
@pytest.mark.parametrize("q, chains", [(1, 33), (1, 2561), (2, 17), (2, 2049), (2, 4097)])   # 4 D and 2 D lanes a chain
def test_many_step_launches_on_ill_conditioned_states(qst, cuda_ok, form, q, chains):
    kw = dict(precision=getattr(qst, "PREC_" + form), diag_chains=0, beta0=1e-5, adapt_interval=1000)
    prob = W.config_problem(q, num_chains=chains)
    prob.beta0 = 0.0   # (the configuration's: 1e-5, so that proposals keep the rows' conditioning)
    many, plain = (qst.Sampler(prob, **kw) for _ in range(2))
    plain.set_profiling(True)   # per-step kernels, one lane per row
    buf = np.array(many.checkpoint())
    x = _latent(q, chains, 910 + q)
    at = 2 * 8                  # after (steps, kept): both copies of the latent states
    for half in range(2):
        buf[at + half * x.nbytes: at + (half + 1) * x.nbytes] = x.reshape(-1).view(np.uint8)
    for s in (many, plain):
        s.restore(buf)
        s.run_chains(12)
    a, b = many.get_state(), plain.get_state()
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    assert np.array_equal(many.posterior_sum()[0], plain.posterior_sum()[0])
    assert not np.array_equal(a["y"], x)   # some proposals were accepted
    many.close()
    plain.close()


def test_groups_by_the_handles_problems(qst, cuda_ok):
    """Two groups while all of a handle's larger problems together are few; the same chains in either handle."""
    few, more = W.config_problem(4, num_chains=500), W.config_problem(4, num_chains=800)
    small = W.config_problem(2, num_chains=3000)
    kw = dict(precision=qst.PREC_PAULI, diag_chains=0)
    with qst.Sampler([few, small], **kw) as a, qst.Sampler([few, more], **kw) as b:
        assert a.diagnostics()["propose_chains_per_cta"] == 2
        assert b.diagnostics()["propose_chains_per_cta"] in (2, 4, 8)   # (32 threads, 64 or 128: timed)
        for s in (a, b):
            s.run_chains(6)
        x, y = a.get_state(0), b.get_state(0)
        assert all(np.array_equal(x[k], y[k]) for k in x)
