"""What the FP32 form's lists of used rows leave as it was: the checkpoint's size, and evaluation in the
other forms."""
import numpy as np
import pytest

from paper_2501_17334_gb300 import workload as W

pytestmark = pytest.mark.gpu


def _checkpoint_size(qst, prob, **cfg):
    with qst.Sampler(prob, diag_chains=0, **cfg) as s:
        return len(s.checkpoint())


@pytest.mark.parametrize("q, chains", [(3, 64), (3, 2048), (4, 32), (4, 64), (4, 1024), (4, 20000)])
def test_checkpoint_size_is_the_column_tiles(qst, cuda_ok, q, chains):
    """A checkpoint holds a partial sum per 128-column tile of P and chain in the FP32 form, one in the
    structured Pauli form, whatever number the projection uses at this size: saved files stay readable."""
    prob = W.config_problem(q, num_chains=chains)
    tiles = (prob.num_povms * prob.dim + 127) // 128
    extra = _checkpoint_size(qst, prob) - _checkpoint_size(qst, prob, precision=qst.PREC_PAULI)
    assert extra == 8 * chains * (tiles - 1)


@pytest.mark.parametrize("q, chains", [(3, 300), (4, 64)])
def test_restored_runs_go_on_the_same(qst, cuda_ok, q, chains):
    prob = W.config_problem(q, num_chains=chains)
    with qst.Sampler(prob, diag_chains=0) as a, qst.Sampler(prob, diag_chains=0) as b:
        a.run_chains(7)
        b.restore(a.checkpoint())
        for s in (a, b):
            s.run_chains(5)
        x, y = a.get_state(), b.get_state()
        assert all(np.array_equal(x[k], y[k]) for k in x)
        assert np.array_equal(a.posterior_sum()[0], b.posterior_sum()[0])


@pytest.mark.parametrize("q", [3, 4])
def test_automatic_form_evaluates_part_of_its_chains(qst, cuda_ok, q):
    """Pauli arrays with rounding noise in their zeros: not exact in bf16, so QST_PREC_AUTO takes the
    structured form, and a batch smaller than the chains gives the rows' own log L."""
    import torch
    prob = W.config_problem(q, num_chains=600)
    prob.povm_re = prob.povm_re.copy()
    prob.povm_re[prob.povm_re == 0.0] = 1e-14
    x = torch.from_numpy(W.latent_batch(600, q, 5).astype(np.float32)).cuda()
    with qst.Sampler(prob, precision=qst.PREC_AUTO, diag_chains=0) as s:
        assert s.diagnostics()["projection_form"] == qst.PREC_PAULI
        s.run_chains(3)
        full = s.evaluate(x)[2].clone()
        for n in (1, 37, 300):
            assert torch.equal(s.evaluate(x[:n])[2], full[:n]), n
