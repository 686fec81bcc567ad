"""The list projection's sums of log L at four qubits: nothing but the logarithms is rounded to FP32.

The maximally mixed state makes every q = 1/16 exact, so each term is an integer count times the FP32
logarithm of a known argument (csrc/log_poly.h gives the same bits on the host) and log L is known to FP64.
The counts are uneven, so that terms are far larger than the sums they join.
"""
import os
import subprocess

import numpy as np
import pytest

from paper_2501_17334_gb300 import workload as W

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_17334_gb300", "csrc")
HARNESS = """
#include <stdio.h>
#include "log_poly.h"
int main(void) {
    float x;
    while (fread(&x, sizeof x, 1, stdin) == 1) { x = qst_log_poly(x); fwrite(&x, sizeof x, 1, stdout); }
    return 0;
}
"""


@pytest.fixture(scope="module")
def log_poly(tmp_path_factory):
    d = tmp_path_factory.mktemp("log")
    (d / "h.c").write_text(HARNESS)
    subprocess.run(["gcc", "-std=c99", "-O2", "-I", CSRC, str(d / "h.c"), "-o", str(d / "h"), "-lm"], check=True)

    def f(x):
        r = subprocess.run([str(d / "h")], input=np.float32(x).tobytes(), capture_output=True, check=True)
        return np.frombuffer(r.stdout, np.float32).astype(np.float64)
    return f


@pytest.mark.parametrize("rows", [1, 130, 5200])       # 32- and 128-chain tiles
@pytest.mark.parametrize("poisson", [0.0, 1000.0, 100.0])   # multinomial; mu near the counts' sum and far below it
def test_sums_of_known_terms(qst, cuda_ok, log_poly, rows, poisson):
    import torch
    D, K = 16, 81
    x = np.zeros((rows, 4, D, D), np.float32)
    x[:, 0] = x[:, 2] = np.eye(D)   # G = H = I: U = I, W = 2 I, rho = I / 16
    for seed in range(8):
        rng = np.random.default_rng(seed)
        prob = W.config_problem(4, num_chains=rows)
        c = rng.integers(0, 8, (K, D))
        c[np.arange(K), rng.integers(0, D, K)] = rng.integers(700, 950, K)
        prob.counts = c.reshape(-1).astype(np.int32)
        wk = c.sum(1).astype(np.float64)
        if poisson:
            prob.likelihood = qst.LIKELIHOOD_POISSON
            prob.trials = wk = np.full(K, poisson)
        with qst.Sampler(prob, diag_chains=0) as s:
            rho, p, ll = s.evaluate(torch.from_numpy(x.reshape(rows, -1)).cuda())
            ll = ll.cpu().numpy()
        assert torch.equal(rho[0], torch.eye(D).reshape(-1).cuda() / D) and (p == 1 / D).all()
        on = c > 0
        invf = np.float32((wk[:, None] / np.maximum(c, 1))[on]).astype(np.float64)
        log = log_poly(invf / D)
        ref = np.sum(c[on] * (log - np.log(invf)))
        if poisson:
            ref += np.sum(c * np.log(wk)[:, None]) - wk.sum()
        # a setting's sum rests on a grid of g (14 bits below its shots); what lies off the grid is added in
        # FP32: 16 adds of at most 4 g a setting; a warp's settings (an eighth of them or fewer) and the 16
        # warps are joined as pairs, with three and two roundings of the low part
        g = 2.0 ** (np.floor(np.log2(c.sum(1).max())) - 14)
        w = (K + 7) // 8
        h = w * (np.abs(np.where(on, c, 0)[on] * log).sum() / K) * 2
        low = 8 * g + 2.0 ** -23 * h
        bound = 2.0 ** -24 * (K * 16 * 4 * g + K * 3 * w * low + 16 * 2 * K * low) + 1e-7
        assert np.abs(ll - ref).max() <= bound, (seed, np.abs(ll - ref).max(), bound)
