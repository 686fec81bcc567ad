"""What the FP32 form's lists of used rows leave as it was: evaluation in the other forms."""
import numpy as np
import pytest

from paper_2501_17334_gb300 import workload as W

pytestmark = pytest.mark.gpu


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
