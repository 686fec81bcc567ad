"""The probabilities every form writes, at aligned and unaligned addresses and at row lengths that are
no multiple of 8: the same bits wherever they go, and p = rho . P / t of the rho written beside."""
import ctypes

import numpy as np
import pytest

from paper_2501_17334_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form, q, rows", [("BF16X3", 1, 300), ("BF16X3", 2, 129), ("BF16X3", 3, 257), ("TF32X2", 3, 65),
                                           ("BF16X3", 4, 130), ("BF16X3", 5, 129), ("PAULI", 1, 129), ("PAULI", 2, 3),
                                           ("PAULI", 3, 49), ("PAULI", 4, 17), ("PAULI", 5, 3), ("FP32", 2, 77)])
def test_p_is_the_same_wherever_it_is_written(form, q, rows):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2501_17334_gb300 import qst
    prob = W.five_qubit_problem(num_chains=rows) if q == 5 else W.config_problem(q, num_chains=rows)
    s = qst.Sampler(prob, precision=getattr(qst, "PREC_" + form), diag_chains=0, autotune=0)
    x = torch.from_numpy(W.latent_batch(rows, q, 5).astype(np.float32)).cuda()
    rho, p, _ = s.evaluate(x)
    n = p.numel()
    for shift in (1, 3, 4):   # floats past a 512-byte boundary
        buf = torch.full((n + 64,), -7.0, device="cuda")
        assert s.lib.qst_evaluate(s.handle, 0, ctypes.c_void_p(x.data_ptr()), rows, None,
                                  ctypes.c_void_p(buf.data_ptr() + 4 * shift), None) == 0
        torch.cuda.synchronize()
        assert torch.equal(buf[shift:shift + n].reshape(p.shape), p)
        assert bool((buf[:shift] == -7.0).all()) and bool((buf[shift + n:] == -7.0).all())
    s.close()
    P = qst.pack_projectors(q, prob.povm_re, prob.povm_im).astype(np.float64)
    r = rho.double().cpu().numpy()
    ref = r @ P / r[:, :: (1 << q) + 1].sum(1)[:, None]
    # FP32 or split operands: 2^-22 of sum |rho P| bounds every form's rounding (23 bits, at most 10 sums of it)
    assert (np.abs(p.double().cpu().numpy() - ref) <= 10 * 2.0 ** -22 * (np.abs(r) @ np.abs(P))).all()
