"""The ACF kernel (Eq. ACFrho) against numpy in FP64 on the same kept states, at the edges of its
tiles: slabs of 4, 16, 32 and several times 32 entries, segments of 256 samples, chunks of 32,
lag tiles of 16 and more than one group of 208 lags."""
import numpy as np
import pytest

from paper_2501_17334_gb300 import workload as W

pytestmark = pytest.mark.gpu


def _acf(x, lmax):
    """c[0..lmax] of one chain's packed states x [N, d] (off-diagonal entries count twice)."""
    N, d = x.shape
    D = int(round(d ** 0.5))
    w = np.where(np.eye(D).reshape(-1) > 0, 1.0, 2.0)
    z = x - x.mean(0)
    m = N - lmax
    c = np.array([np.sum(w * z[:m] * z[l:l + m]) for l in range(lmax + 1)])
    return c / c[0]


@pytest.mark.parametrize("q, kept, lmax, chains", [(1, 9, 8, 3), (1, 70, 15, 130), (2, 300, 20, 5), (2, 64, 32, 2),
                                                   (3, 129, 16, 4), (4, 290, 210, 3), (4, 33, 1, 2), (5, 40, 7, 2),
                                                   (3, 620, 417, 2)])
def test_acf_matches_numpy(q, kept, lmax, chains):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2501_17334_gb300 import qst
    prob = (W.five_qubit_problem(num_chains=chains) if q == 5 else W.config_problem(q, num_chains=chains))
    s = qst.Sampler(prob, precision=qst.PREC_PAULI, diag_chains=chains, traj_capacity=kept, acf_lmax=lmax)
    traj = []
    for _ in range(kept):
        s.run_chains(1)
        y = torch.from_numpy(s.get_state()["y"]).cuda()
        traj.append(s.evaluate(y, want_p=False)[0].double().cpu().numpy())
    x = np.stack(traj, 1)   # [chain, sample, d]
    dg = s.diagnostics()
    s.close()
    ref = np.stack([_acf(x[c], lmax) for c in range(chains)])
    tau = 1.0 + 2.0 * ref[:, 1:].sum(1)
    # a kept state is the evaluated one up to its FP32 rescaling by 1 / t (2^-23 of an entry <= 1); the FP32
    # chunks of 32 products round by at most 32 2^-24 of the sum of |z z'| <= c~[0] (N / (N - lmax) at most)
    rms = min(np.sqrt(np.mean((x[c] - x[c].mean(0))[: kept - lmax] ** 2)) for c in range(chains))
    full = max(np.mean((x[c] - x[c].mean(0)) ** 2) ** 0.5 for c in range(chains))
    tol = (32 * 2.0 ** -24 + 2 * 2.0 ** -23 / rms) * 2 * (1 + full / rms) * kept / (kept - lmax)
    assert np.abs(dg["acf"] - ref.mean(0)).max() < tol
    assert np.abs(dg["tau"] - tau).max() < 2 * lmax * tol
