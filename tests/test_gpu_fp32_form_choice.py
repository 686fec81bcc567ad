"""The FP32 projection at three and four qubits takes the tiled kernel where lists without zeros save nothing
(around whole waves of tiles, and for many settings and few rows), the list kernel elsewhere; a handle changes
between them with the rows of a call.  Both against numpy in FP64 on the kernel's own rho."""
import numpy as np
import pytest

from paper_2501_17334_gb300 import workload as W

pytestmark = pytest.mark.gpu


def _list_groups(chains):
    """Partial sums per chain the list kernel has, with one and with four chains a lane: one per CTA of a
    tile, 152 CTAs in all (none of the tiled kernel's powers of two or column tiles at the tiled sizes below)."""
    return {(152 + t - 1) // t + 1 for t in ((chains + 31) // 32, (chains + 127) // 128)}


def _check(qst, prob, q, s, rows):
    import torch
    x = torch.from_numpy(W.latent_batch(rows, q, rows).astype(np.float32)).cuda()
    rho, p, ll = s.evaluate(x)
    pick = np.unique(np.linspace(0, rows - 1, 100).astype(int))
    r, got = rho.double().cpu().numpy()[pick], p.double().cpu().numpy()[pick]
    P = qst.pack_projectors(q, prob.povm_re, prob.povm_im).astype(np.float64)
    D = 1 << q
    t = r[:, :: D + 1].sum(1)[:, None]
    # chunks of 32 products and their sum: at most 40 roundings of partial sums below sum |rho P|
    bound = 40 * 2.0 ** -24 * (np.abs(r) @ np.abs(P)) + 2.0 ** -22 * np.abs(r @ P / t)
    assert (np.abs(got - r @ P / t) <= bound).all()
    # log L on the kernel's own p: 8 2^-24 a count of its term's size (FP32 logs, products and settings' sums)
    c = prob.counts.astype(np.float64)
    on = c > 0
    q_n = (got.reshape(len(pick), -1, D) / got.reshape(len(pick), -1, D).sum(2)[:, :, None]).reshape(got.shape)
    want = np.log(q_n[:, on]) @ c[on]
    f = np.maximum(c, 1.0) / np.repeat(np.maximum(c.reshape(-1, D).sum(1), 1.0), D)
    size = (c[on] * (2.0 + np.abs(np.log(got[:, on] / f[on])))).sum(1)
    assert (np.abs(ll.cpu().numpy()[pick] - want) <= 8 * 2.0 ** -24 * size).all()


@pytest.mark.parametrize("q, K, chains, tiled", [(4, 81, 1400, True), (4, 81, 1500, True), (4, 150, 1000, True),
                                                 (4, 300, 300, True), (4, 1000, 65, True), (3, 300, 1000, True),
                                                 (3, 1000, 64, True), (4, 81, 700, False), (4, 81, 2000, False),
                                                 (4, 1000, 1000, False), (3, 27, 1500, False), (4, 5, 20000, False)])
def test_choice_by_rows_and_settings(qst, cuda_ok, q, K, chains, tiled):
    prob = W.random_basis_problem(q, K, num_chains=chains)
    with qst.Sampler(prob, diag_chains=0) as s:
        assert (s.diagnostics()["column_groups"] not in _list_groups(chains)) == tiled
        _check(qst, prob, q, s, chains)


def test_pauli_settings_take_their_lists(qst, cuda_ok):
    for q, chains in ((4, 1500), (4, 1664), (3, 9728)):
        with qst.Sampler(W.config_problem(q, num_chains=chains), diag_chains=0) as s:
            assert s.diagnostics()["column_groups"] in _list_groups(chains)


def test_a_handle_changes_with_the_rows(qst, cuda_ok):
    """1500 chains run tiled, 64 and 300 rows of them take the lists; 10007 chains the other way round."""
    for chains, rows in ((1500, (64, 1500, 300)), (10007, (1400, 10007, 64))):
        prob = W.random_basis_problem(4, 81, num_chains=chains)
        with qst.Sampler(prob, diag_chains=0) as s:
            for n in rows:
                _check(qst, prob, 4, s, n)
            s.run_chains(3)
            _check(qst, prob, 4, s, rows[0])


def test_rows_close_to_the_chains(qst, cuda_ok):
    """16384 chains run tiled in one column group, 12000 rows of them take the lists, over all SMs: the
    projection of fewer rows is no slower than twice that of all."""
    import torch
    prob = W.random_basis_problem(4, 5, num_chains=16384)
    with qst.Sampler(prob, diag_chains=0) as s:
        assert s.diagnostics()["column_groups"] not in _list_groups(16384)
        _check(qst, prob, 4, s, 12000)
        s.set_profiling(True)
        us = []
        for n in (16384, 12000):
            x = torch.from_numpy(W.latent_batch(n, 4, 3).astype(np.float32)).cuda()
            s.evaluate(x)
            s.kernel_time(qst.KERNEL_PROJECT, reset=True)
            for _ in range(5):
                s.evaluate(x)
            ms, k = s.kernel_time(qst.KERNEL_PROJECT, reset=True)
            us.append(ms / k * 1e3)
        assert us[1] < 2 * us[0], us
