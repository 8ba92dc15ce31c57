"""prism_grad_noalloc on signals so small that the reciprocal of their b0 mean overflows (and around that line): the same
objective and gradient as for the signals times a power of two, which leaves every quotient the same."""
import ctypes

import numpy as np
import pytest
import torch

import phantoms as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_shells", [2, 20])   # the shell form and the per-measurement form
@pytest.mark.parametrize("exponent", [-149, -147, -143, -140])
def test_tiny_signals(n_shells, exponent):
    import paper_2604_00250_gb300 as prism
    from paper_2604_00250_gb300 import _lib
    from phantoms import schemes
    lib, K, V = _lib.load(), 2, 70
    bvals, bvecs = schemes.make_scheme(5, [(200 + 150 * i, 60 // n_shells) for i in range(n_shells)], 3)
    vol = P.random_volume((7, 5, 2), scheme=(bvals, bvecs), seed=1, mask_density=1.0)
    units = np.rint(np.asarray(vol.signal, np.float64) * 2e5).clip(1, 2 ** 20)   # whole numbers: exact at every scale
    th = torch.as_tensor(P.default_init(V, K, 4).astype(np.float32)).cuda()
    o, out = prism.options(K=K), []
    for e in (0, exponent):
        s = torch.as_tensor(np.ldexp(units, e).astype(np.float32)).cuda()
        grad = torch.full((V, 4 * K + 5), float("nan"), device="cuda")
        loss = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
        _lib.check(lib.prism_grad_noalloc(ctypes.c_void_p(s.data_ptr()), bvals.ctypes.data, bvecs.ctypes.data,
                                          ctypes.c_void_p(th.data_ptr()), V, len(bvals), K, o.lam_rep, o.lam_sparse, o.tau,
                                          ctypes.c_void_p(grad.data_ptr()), ctypes.c_void_p(loss.data_ptr()),
                                          ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
        torch.cuda.synchronize()
        out.append((float(loss[0]), grad.cpu().numpy()))
    (J0, g0), (J1, g1) = out
    # the b0 means of the two scales may round differently (a subnormal mean has fewer bits: at 2^-149 times about 2e5,
    # 18 of them), 4e-6 of every quotient; the objective and the gradient of a model far from its data follow in proportion
    assert abs(J1 - J0) <= 1e-4 * abs(J0)
    assert np.linalg.norm(g1 - g0) <= 1e-4 * np.linalg.norm(g0)
