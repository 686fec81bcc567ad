"""The FP32 projection over the rows of P a setting uses (three and four qubits): ragged tiles, few
and many settings, full lists (random bases), empty and short ones, unaligned output, and more CTAs
per tile than one, against numpy in FP64 on the kernel's own rho."""
import ctypes

import numpy as np
import pytest

from paper_2501_17334_gb300 import workload as W

pytestmark = pytest.mark.gpu


def _problem(kind, q, rows):
    if kind == "pauli":
        return W.config_problem(q, num_chains=rows)
    if kind == "bases":
        return W.random_basis_problem(q, 5, num_chains=rows)
    if kind == "one":
        return W.random_basis_problem(q, 1, num_chains=rows)
    prob = W.lossy_pauli_problem(q, rows)   # Poisson; the first setting's detectors see nothing at all
    D = 1 << q
    prob.povm_re, prob.povm_im, prob.counts = prob.povm_re.copy(), prob.povm_im.copy(), prob.counts.copy()
    prob.povm_re[:D] = 0.0
    prob.povm_im[:D] = 0.0
    prob.counts[:D] = 0
    return prob


@pytest.mark.parametrize("kind", ["pauli", "bases", "one", "dark"])
@pytest.mark.parametrize("q, rows, chains", [(3, 1, 1), (3, 255, 255), (3, 257, 300), (4, 127, 127), (4, 129, 129),
                                             (4, 1000, 1000), (4, 3, 20000), (3, 40001, 40001)])
def test_q_and_log_l(kind, q, rows, chains):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2501_17334_gb300 import qst
    prob = _problem(kind, q, chains)
    s = qst.Sampler(prob, diag_chains=0)
    x = torch.from_numpy(W.latent_batch(rows, q, 77).astype(np.float32)).cuda()
    rho, p, ll = s.evaluate(x)
    # the same with p one float past an aligned address
    off = torch.zeros(p.numel() + 1, device="cuda")
    ll2 = torch.empty_like(ll)
    assert s.lib.qst_evaluate(s.handle, 0, ctypes.c_void_p(x.data_ptr()), rows, None,
                              ctypes.c_void_p(off.data_ptr() + 4), ctypes.c_void_p(ll2.data_ptr())) == 0
    torch.cuda.synchronize()
    assert torch.equal(off[1:].reshape(p.shape), p) and torch.equal(ll, ll2)
    s.close()
    pick = np.unique(np.linspace(0, rows - 1, 300).astype(int))
    r = rho.double().cpu().numpy()[pick]
    P = qst.pack_projectors(q, prob.povm_re, prob.povm_im).astype(np.float64)
    D = 1 << q
    t = r[:, :: D + 1].sum(1)[:, None]
    ref = r @ P / t
    # chunks of 32 products and their sum: at most 40 roundings of partial sums below sum |rho P|
    bound = 40 * 2.0 ** -24 * (np.abs(r) @ np.abs(P)) + 2.0 ** -22 * np.abs(ref)
    got = p.double().cpu().numpy()[pick]
    assert (np.abs(got - ref) <= bound).all()
    # log L on the kernel's own p (FP32 logs <= 2 ulp, products and the settings' terms): 8 2^-24 a count
    # of the terms' sizes, c (1 + |log|), and for the Poisson terms of mu
    c = prob.counts.astype(np.float64)
    on = c > 0
    S = got.reshape(len(pick), -1, D).sum(2)
    if kind == "dark":
        mu = np.repeat(prob.trials, D)
        want = np.log(mu[on] * got[:, on]) @ c[on] - (got @ mu)
        extra = prob.trials.sum()
    else:
        q_n = (got.reshape(len(pick), -1, D) / S[:, :, None]).reshape(got.shape)
        want = np.log(q_n[:, on]) @ c[on]
        extra = 0.0
    f = np.maximum(c, 1.0) / np.repeat(np.maximum(c.reshape(-1, D).sum(1), 1.0), D)
    size = (c[on] * (2.0 + np.abs(np.log(got[:, on] / f[on])))).sum(1)
    assert (np.abs(ll.cpu().numpy()[pick] - want) <= 8 * 2.0 ** -24 * (size + extra)).all()
