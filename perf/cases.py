"""The work a user of the sampler has it do, as timed cases.

A case is one call, or one short sequence of calls, of the public entry points
(``paper_2501_17334_gb300.qst``) on a seeded synthetic tomography problem:

* ``run``       chains of one problem (or a batch of problems) advance by a number of steps and
                the pooled posterior mean is read back -- what every program built on the
                sampler repeats;
* ``evaluate``  rho, the outcome probabilities and log L of a batch of latent vectors the caller
                holds on the device;
* ``diagnose``  the autocorrelation function and the integrated autocorrelation times of the
                stored trajectories, once a run is over;
* ``noalloc``   log L of a batch of latent vectors by the entry point that allocates nothing.

Problem sizes, shots and step sizes are those of ``workload.config_problem``, of its five- and
six-qubit problems and of its heterogeneous batch, and of the tests (odd chain counts, lossy
Poisson counts, bases that are not Pauli bases).  Truth, counts, chain seed and latent vectors all
follow from ``seed``.
"""
import math
import random

import numpy as np
import torch

from paper_2501_17334_gb300 import qst, workload

FORMS = {"fp32": qst.PREC_FP32, "bf16x3": qst.PREC_BF16X3, "tf32x2": qst.PREC_TF32X2, "pauli": qst.PREC_PAULI}
PRIORS = {"bures": qst.PRIOR_BURES, "hs": qst.PRIOR_HS}
# shots per setting and initial step of the configurations, by qubit count
SHOTS = {1: 1000, 2: 1000, 3: 2000, 4: 1000, 5: 1000, 6: 1000}
BETA0 = {1: 0.1, 2: 0.05, 3: 0.1, 4: 0.02, 5: 0.05, 6: 0.02}


def _run(name, qubits, chains, steps, form, **more):
    return dict({"name": name, "kind": "run", "qubits": qubits, "chains": chains, "steps": steps, "form": form,
                 "prior": "bures", "thin": 1, "poisson": False}, **more)


def listed():
    return [
        # the smallest call: one qubit, 64 chains, the default (FP32) form; a short run between two
        # looks at the posterior mean, where a step is all latency and launches
        _run("run-1q", 1, 64, 100, "fp32"),
        # two qubits, 4096 chains, the default form: the paper's smaller experiments
        _run("run-2q", 2, 4096, 50, "fp32"),
        # three qubits, 16384 chains on the tensor cores: an ordinary problem
        _run("run-3q", 3, 16384, 20, "bf16x3"),
        # four qubits, 65536 chains on the tensor cores: the headline workload
        _run("run-4q", 4, 65536, 10, "bf16x3"),
        # an odd, small number of four-qubit chains, thinned, in the structured form
        _run("run-4q-few", 4, 1001, 20, "pauli", thin=2),
        # five qubits in the structured form (the one that is chosen for them)
        _run("run-5q", 5, 8192, 5, "pauli"),
        # six qubits, the largest state there is
        _run("run-6q", 6, 1024, 4, "pauli"),
        # a batch of uneven problems of one to five qubits in one handle
        {"name": "run-batch", "kind": "batch", "problems": 12, "max_qubits": 5, "max_chains": 8192, "steps": 5,
         "form": "pauli"},
        # rho, p and log L of latent vectors, four qubits, the default form, a ragged last tile
        {"name": "evaluate-4q", "kind": "evaluate", "qubits": 4, "rows": 10007, "form": "fp32", "povm": "pauli"},
        # the same on counts from lossy detectors (Poisson likelihood), three qubits, TF32x2
        {"name": "evaluate-3q-lossy", "kind": "evaluate", "qubits": 3, "rows": 5001, "form": "tf32x2", "povm": "lossy"},
        # the end of a run: ACF and IACT of 256 four-qubit chains
        {"name": "diagnose-4q", "kind": "diagnose", "qubits": 4, "chains": 256, "kept": 600, "lmax": 200},
        # log L without device allocation, as a plugin's likelihood callback
        {"name": "noalloc-4q", "kind": "noalloc", "qubits": 4, "rows": 1000, "povm": "pauli"},
    ]


# ---- drawn cases ----------------------------------------------------------------------------

def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


_MAX_CHAINS = {1: 65536, 2: 65536, 3: 65536, 4: 65536, 5: 16384, 6: 2048}
_RUN_FORMS = {1: ("fp32", "bf16x3", "pauli"), 2: ("fp32", "bf16x3", "pauli"), 3: ("bf16x3", "tf32x2", "pauli"),
              4: ("bf16x3", "pauli"), 5: ("bf16x3", "pauli"), 6: ("pauli",)}


def draw(rng: random.Random):
    """A case of the same ranges; none costs more than the four-qubit run of ``listed``."""
    kind = rng.choice(["run", "run", "run", "run", "batch", "evaluate", "evaluate", "diagnose", "noalloc"])
    if kind == "run":
        q = rng.randint(1, 6)
        limit = _flops_step(4, True) * 65536 * 10
        form = rng.choice(_RUN_FORMS[q])
        chains = _log_uniform(rng, 64, _MAX_CHAINS[q])
        most = max(1, min(100, int(limit / (_flops_step(q, True) * chains))))
        case = {"kind": "run", "qubits": q, "chains": chains, "steps": _log_uniform(rng, 1, most), "form": form,
                "prior": rng.choice(["bures", "bures", "bures", "hs"]), "thin": rng.choice([1, 1, 2, 5]),
                "poisson": q <= 4 and rng.random() < 0.2}
        case["steps"] = max(case["steps"], case["thin"])
        return case
    if kind == "batch":
        return {"kind": "batch", "problems": rng.randint(2, 16), "max_qubits": rng.randint(2, 5),
                "max_chains": _log_uniform(rng, 512, 4096), "steps": rng.randint(2, 10), "form": "pauli"}
    if kind == "evaluate":
        q = rng.randint(1, 5)
        povm = rng.choice(["pauli", "pauli", "bases", "lossy"]) if q <= 4 else "pauli"
        form = "fp32" if povm == "bases" else rng.choice(["fp32", "bf16x3"] + (["tf32x2"] if q <= 3 else []) +
                                                         (["pauli"] if povm == "pauli" else []))
        return {"kind": "evaluate", "qubits": q, "rows": _log_uniform(rng, 1, 20000 if q <= 4 else 2000), "form": form,
                "povm": povm}
    if kind == "diagnose":
        return {"kind": "diagnose", "qubits": rng.randint(1, 4), "chains": rng.choice([16, 64, 100, 256, 512]),
                "kept": rng.randint(210, 1024), "lmax": rng.choice([50, 100, 200])}
    return {"kind": "noalloc", "qubits": rng.randint(1, 4), "rows": _log_uniform(rng, 1, 4096),
            "povm": rng.choice(["pauli", "pauli", "bases"])}


# ---- problems -------------------------------------------------------------------------------

def _settings(q):
    """Settings of the measurement in bases that are not Pauli bases: as many as the Pauli ones."""
    return 3 ** q


def _run_problem(q, chains, seed, shots, beta0, rank, weight):
    """A Pauli problem (the built-in POVMs: no arrays) with a Ginibre truth of the given rank
    depolarised by `weight`."""
    rng = np.random.default_rng(seed)
    truth = workload.depolarise(workload.ginibre_state(1 << q, rank, rng), weight)
    counts = workload.sample_counts(truth, q, shots, rng)
    return workload.Problem(q, None, None, counts, truth, int(chains), 0, beta0, int(rng.integers(1 << 31)), "case")


def _problem(case, seed, chains):
    q = case["qubits"]
    povm = case.get("povm", "lossy" if case.get("poisson") and case["form"] != "pauli" else "pauli")
    if povm == "lossy":
        return workload.lossy_pauli_problem(q, chains, trials=float(SHOTS[q]), seed=seed, beta0=BETA0[q])
    if povm == "bases":
        return workload.random_basis_problem(q, _settings(q), seed=seed, num_chains=chains, beta0=BETA0[q])
    p = _run_problem(q, chains, seed, SHOTS[q], BETA0[q], {1: 2, 2: 4, 3: 2, 4: 1, 5: 3, 6: 3}[q],
                     {1: 0.0, 2: 0.1, 3: 0.05, 4: 0.02, 5: 0.05, 6: 0.05}[q])
    if case.get("poisson"):   # the Pauli settings through perfect detectors
        p.likelihood = qst.LIKELIHOOD_POISSON
        p.trials = np.full(3 ** q, float(SHOTS[q]))
    return p


def _latent(case, seed):
    """Standard-normal latent vectors, as the prior draws them."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(case["rows"], 4 << (2 * case["qubits"]), generator=g, device="cuda", dtype=torch.float32)


# ---- prepare and run ------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "run":
        prob = _problem(case, seed, case["chains"])
        return case, qst.Sampler(prob, precision=FORMS[case["form"]], prior=PRIORS[case["prior"]], thin=case["thin"])
    if kind == "batch":
        rng = np.random.default_rng(seed)
        shape = np.random.default_rng(case["problems"] * 8 + case["max_qubits"])   # the sizes are the case's
        probs = []
        for _ in range(case["problems"]):
            q = int(shape.integers(1, case["max_qubits"] + 1))
            chains = int(round(math.exp(shape.uniform(math.log(256), math.log(case["max_chains"])))))
            probs.append(_run_problem(q, chains, int(rng.integers(1 << 31)), int(shape.integers(500, 4001)), 0.05,
                                      int(shape.integers(1, (1 << q) + 1)), 0.0))
        return case, qst.Sampler(probs, precision=FORMS[case["form"]], diag_chains=0)
    if kind == "evaluate":
        prob = _problem(case, seed, case["rows"])
        return case, qst.Sampler(prob, precision=FORMS[case["form"]], diag_chains=0), _latent(case, seed)
    if kind == "diagnose":
        prob = _run_problem(case["qubits"], case["chains"], seed, SHOTS[case["qubits"]], BETA0[case["qubits"]], 1, 0.05)
        s = qst.Sampler(prob, precision=qst.PREC_PAULI, diag_chains=case["chains"], traj_capacity=1024,
                        acf_lmax=case["lmax"])
        s.run_chains(case["kept"])
        return case, s
    prob = _problem(dict(case, form="fp32"), seed, case["rows"])
    q = case["qubits"]
    if prob.povm_re is None:
        P = qst.pack_projectors(q, *qst.pauli_povms(q))
    else:
        P = qst.pack_projectors(q, prob.povm_re, prob.povm_im)
    logl = torch.empty(case["rows"], dtype=torch.float64, device="cuda")
    return case, q, prob.num_povms, torch.from_numpy(P).cuda(), prob.counts, _latent(case, seed), logl


_DIAG_FIELDS = ("acf", "tau", "accept_rate", "beta_min", "beta_mean", "beta_max", "tau_mean", "tau_max", "n_eff",
                "steps_done", "num_kept", "num_pooled", "num_nonfinite")


def run(state):
    kind = state[0]["kind"]
    if kind == "run":
        state[1].run_chains(state[0]["steps"])
        return state[1].posterior_mean()
    if kind == "batch":
        state[1].run_chains(state[0]["steps"])
        return [state[1].posterior_mean(i) for i in range(state[0]["problems"])]
    if kind == "evaluate":
        return state[1].evaluate(state[2])
    if kind == "diagnose":
        d = state[1].diagnostics()
        return {k: d[k] for k in _DIAG_FIELDS}
    _, q, settings, P, counts, x, logl = state
    qst.loglik_noalloc(q, settings, P, counts, x, logl)
    return logl


# ---- what a pass cannot do without ----------------------------------------------------------

def _flops_rho(q, bures=True):
    """Algorithm 1 per chain: one QR of H, W = (U + I) G, the Hermitian half of W W^dag."""
    D = 1 << q
    return (8 * D * D * (D - 1) + 8 * D ** 3 if bures else 0) + 4 * D * D * (D + 1) + D * D


def _flops_logl(q, pauli, settings=None):
    """The probabilities and their logarithms: for the Pauli settings 3.5 adds per outcome by
    splitting rho one qubit at a time, else the dense contraction; a logarithm is about 20."""
    D = 1 << q
    K = 3 ** q if settings is None else settings
    return K * D * (20 + (3.5 if pauli else 2 * D * D))


def _flops_step(q, bures=True, pauli=True):
    """A chain's step: 4 D^2 normals (a quarter of a Philox block and half a Box-Muller each,
    about 30 operations) and their pCN update, rho, log L."""
    return 32 * 4 * (1 << (2 * q)) + _flops_rho(q, bures) + _flops_logl(q, pauli)


def _bytes_run(q, chains, steps):
    """The latent state (4 D^2 floats a chain) is read and written once in a pass where the chip
    can hold it (129 MB of L2), and at every step where it cannot."""
    state = 16 * (1 << (2 * q)) * chains
    return 2 * state * (steps if state > 129e6 else 1)


def work(case):
    kind = case["kind"]
    if kind == "run":
        q = case["qubits"]
        lossy = case["poisson"] and case["form"] != "pauli"   # elements that are no Pauli projectors
        return {"bytes": _bytes_run(q, case["chains"], case["steps"]),
                "flops": case["chains"] * case["steps"] * _flops_step(q, case["prior"] == "bures", not lossy)}
    if kind == "batch":
        shape = np.random.default_rng(case["problems"] * 8 + case["max_qubits"])
        b = f = 0
        for _ in range(case["problems"]):
            q = int(shape.integers(1, case["max_qubits"] + 1))
            chains = int(round(math.exp(shape.uniform(math.log(256), math.log(case["max_chains"])))))
            shape.integers(500, 4001), shape.integers(1, (1 << q) + 1)
            b += _bytes_run(q, chains, case["steps"])
            f += chains * case["steps"] * _flops_step(q)
        return {"bytes": b, "flops": f}
    if kind == "diagnose":
        d = 1 << (2 * case["qubits"])
        kept, lmax = case["kept"], case["lmax"]
        return {"bytes": case["chains"] * (4 * d * kept + 8 * (lmax + 1)),
                "flops": case["chains"] * 2.0 * d * (kept - lmax) * (lmax + 1)}
    q, n = case["qubits"], case["rows"]
    d, KD = 1 << (2 * q), (3 ** q) << q
    pauli = case["povm"] == "pauli"
    out = 4 * d + 4 * KD + 8 if kind == "evaluate" else 8
    return {"bytes": n * (16 * d + out) + (0 if pauli else 4 * d * KD),
            "flops": n * (_flops_rho(q) + _flops_logl(q, pauli))}


# ---- the same in 64 bits --------------------------------------------------------------------

def _pauli_vectors(q):
    s = 1 / math.sqrt(2)
    single = np.array([[[s, s], [s, -s]], [[s, 1j * s], [s, -1j * s]], [[1, 0], [0, 1]]])   # [setting][outcome]
    t = np.ones((1, 1, 1), complex)
    for _ in range(q):   # qubit 0 most significant, in the setting, the outcome and the component
        k, l, c = t.shape
        t = np.einsum("klc,sbm->kslbcm", t, single).reshape(3 * k, 2 * l, 2 * c)
    return t.reshape(-1, 1 << q)


def exact(case, seed):
    """rho, p and log L of the latent vectors by numpy in 64 bits; the runs (a chain's decisions)
    and the diagnostics (of a run's states) have no such value."""
    if case["kind"] not in ("evaluate", "noalloc"):
        return None
    q, n = case["qubits"], case["rows"]
    D = 1 << q
    prob = _problem(case if "form" in case else dict(case, form="fp32"), seed, n)
    x = _latent(case, seed).cpu().numpy().astype(np.float64).reshape(n, 4, D, D).transpose(0, 1, 3, 2)
    G, H = x[:, 0] + 1j * x[:, 1], x[:, 2] + 1j * x[:, 3]
    Q, R = np.linalg.qr(H)
    r = np.diagonal(R, axis1=1, axis2=2)
    W = G + (Q * (r / np.abs(r))[:, None, :]) @ G
    rho = W @ W.conj().transpose(0, 2, 1)
    rho /= np.trace(rho, axis1=1, axis2=2).real[:, None, None]
    if prob.povm_re is None:
        povm = np.einsum("ma,mb->mab", (v := _pauli_vectors(q)), v.conj())
    else:
        povm = prob.povm_re + 1j * prob.povm_im
    # Tr(Lambda rho) = sum_ab Lambda_ab rho_ba, as a real product
    flat, lam = rho.transpose(0, 2, 1).reshape(n, -1), povm.reshape(povm.shape[0], -1)
    p = flat.real @ lam.real.T - flat.imag @ lam.imag.T
    c = prob.counts.astype(np.float64)
    on = c > 0
    if prob.likelihood == qst.LIKELIHOOD_POISSON:
        mu = np.repeat(np.asarray(prob.trials, np.float64), D)
        logl = np.log(mu[on] * p[:, on]) @ c[on] - p @ mu
    else:
        logl = np.log(p[:, on]) @ c[on]
    if case["kind"] == "noalloc":
        return torch.from_numpy(logl)
    upper = np.triu(np.ones((D, D), bool))
    packed = np.where(upper, rho.real, rho.imag).reshape(n, D * D)
    return torch.from_numpy(packed), torch.from_numpy(p), torch.from_numpy(logl)
