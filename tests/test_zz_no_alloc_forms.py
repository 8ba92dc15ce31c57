"""prism_grad_noalloc over the forms its kernel tells apart: whole and odd shells, more b-values than
the shell loop takes, b <= 50 measurements past one chunk, voxel counts around a warp and a block;
against the plain handle path (separate kernels, tests/helpers.py tolerances). Collected late."""
import ctypes
import types

import numpy as np
import pytest
import torch

import phantoms as P
from tests.helpers import TOL_GRAD, TOL_LOSS, block_slices, normwise

pytestmark = pytest.mark.gpu


def _scheme(kind):
    from phantoms import schemes
    if kind == "even":
        return schemes.make_scheme(6, [(1000, 30), (2500, 28)], 1)
    if kind == "odd":
        return schemes.make_scheme(3, [(45, 5), (1000, 31), (2500, 27)], 2)
    if kind == "many":
        return schemes.make_scheme(2, [(300 + 137 * i, 1 + i % 2) for i in range(23)], 3)
    if kind == "many_b0":
        return schemes.make_scheme(37, [(20, 30), (1000, 33)], 4)
    return schemes.make_scheme(1, [(700, 1)], 5)


@pytest.mark.parametrize("kind", ["even", "odd", "many", "many_b0", "two"])
@pytest.mark.parametrize("V,K", [(1, 3), (31, 1), (33, 2), (127, 4), (129, 5), (700, 3)])
def test_forms_match_the_handle_path(kind, V, K):
    import paper_2604_00250_gb300 as prism
    from paper_2604_00250_gb300 import _lib
    lib = _lib.load()
    bvals, bvecs = _scheme(kind)
    order = np.random.default_rng(V).permutation(len(bvals))
    bvals, bvecs = np.ascontiguousarray(bvals[order]), np.ascontiguousarray(bvecs[order])
    vol = P.random_volume((10, 10, 7), scheme=(bvals, bvecs), seed=V)
    mask = np.zeros((10, 10, 7), np.uint8)
    mask.flat[:V] = 1
    sig = np.ascontiguousarray(vol.signal[:V]) * 743.0
    th = (P.default_init(V, K, 4) + np.random.default_rng(K).normal(0, 0.3, (V, 4 * K + 5))).astype(np.float32)
    v = types.SimpleNamespace(mask=mask, signal=sig, bvals=bvals, bvecs=bvecs, init=th)
    with prism.Fitter([v], prism.options(K=K, fused=0)) as f:
        J = float(f.forward()[0][0])
        g = f.backward()[0].cpu().numpy()
    s, t = torch.as_tensor(sig).cuda(), torch.as_tensor(th).cuda()
    grad = torch.full((V, 4 * K + 5), float("nan"), device="cuda")
    loss = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
    o = prism.options(K=K)
    rc = lib.prism_grad_noalloc(ctypes.c_void_p(s.data_ptr()), bvals.ctypes.data, bvecs.ctypes.data,
                                ctypes.c_void_p(t.data_ptr()), V, len(bvals), K, o.lam_rep, o.lam_sparse, o.tau,
                                ctypes.c_void_p(grad.data_ptr()), ctypes.c_void_p(loss.data_ptr()),
                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, lib.prism_last_error()
    torch.cuda.synchronize()
    assert abs(float(loss[0]) - J) <= TOL_LOSS * abs(J)
    for name, sl in block_slices(K).items():
        assert normwise(grad.cpu().numpy()[:, sl], g[:, sl]) <= TOL_GRAD, name
