"""A call that fails part way leaves nothing running behind the handle's stream."""
import ctypes

import pytest

from paper_2501_17334_gb300 import workload as W

pytestmark = pytest.mark.gpu


def test_branches_join_when_a_launch_fails(qst, cuda_ok):
    """Two many-step problems run on branches beside the handle's stream.  The failure is made on the host: an
    allocation of more than the card's memory leaves its error code in the CUDA runtime, where the check
    after the first launch finds it, with that launch's kernel (1000 steps, several milliseconds) under way."""
    import torch
    probs = [W.config_problem(1, num_chains=65536) for _ in range(2)]
    s = qst.Sampler(probs, diag_chains=0, thin=1000)   # one launch per problem and call
    s.run_chains(5)
    s.synchronize()
    cfg = qst.default_config(diag_chains=0, trace_steps=2_000_000)   # 1.2 TB of decisions
    descs = qst._Descs(probs[:1])
    handle = ctypes.c_void_p()
    status = s.lib.qst_create(descs.descs, 1, ctypes.byref(cfg), None, 0, None, ctypes.byref(handle))
    assert status == 3 and not handle
    with pytest.raises(qst.QstError):
        s.run_chains(1000)
    first = s.workspace.clone()   # (on the handle's stream)
    torch.cuda.synchronize()
    assert torch.equal(first, s.workspace)
    s.close()
