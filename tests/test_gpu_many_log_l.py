"""Millions of proposals' log L of the many-step launches have the per-step kernels' bits: log t of the trace,
whose second-order term lies near log L's last bit, is formed by the same FP64 operations in both."""
import numpy as np
import pytest

from paper_2501_17334_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["FP32", "PAULI"])
@pytest.mark.parametrize("q, chains", [(1, 32768), (2, 16384), (1, 1000), (2, 1000)])
def test_traces_have_the_same_bits(qst, cuda_ok, form, q, chains):
    steps = 10_000_000 // (4 * chains) if chains > 1000 else 1000
    kw = dict(precision=getattr(qst, "PREC_" + form), diag_chains=0, trace_steps=steps)
    prob = W.config_problem(q, num_chains=chains)
    with qst.Sampler(prob, **kw) as many, qst.Sampler(prob, **kw) as plain:
        plain.set_profiling(True)
        for s in (many, plain):
            s.run_chains(steps)
        for a, b in zip(many.get_trace(), plain.get_trace()):
            assert np.array_equal(a, b), np.count_nonzero(a != b)
