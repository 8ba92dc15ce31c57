"""prism_forward / prism_backward on a fused handle (the fused kernel's gradient form) against the
same calls on a plain handle (separate synthesis, data term and adjoint kernels), and that an
evaluation leaves the running fit as it was."""
import numpy as np
import pytest
import torch

import phantoms as P
from tests.helpers import TOL_GRAD, TOL_LOSS, TOL_SIGNAL, normwise, signal_rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lanes", [1, 4, 16])
@pytest.mark.parametrize("loss,cal", [("mse", False), ("mse", True), ("nll", False), ("nll", True)])
@pytest.mark.parametrize("K,spatial,n_b0", [(3, True, 6), (5, False, 7), (2, True, 1)])
def test_matches_the_plain_kernels(lanes, loss, cal, K, spatial, n_b0):
    import paper_2604_00250_gb300 as prism
    from phantoms import schemes
    sch = [schemes.make_scheme(n_b0, [(1000, 30), (2500, 20)], 3), schemes.make_scheme(2, [(700, 11)], 4)]
    vols = [P.random_volume((9, 6, 5), scheme=sch[0], seed=3, mask_density=0.8, calibration=cal),
            P.random_volume((4, 3, 3), scheme=sch[1], seed=4, calibration=cal)]
    for i, v in enumerate(vols):
        rng = np.random.default_rng(i)
        v.init = (P.default_init(v.n_vox, K, i) + rng.normal(0, 0.2, (v.n_vox, 4 * K + 5))).astype(np.float32)
    kw = dict(K=K, loss=loss, calibration=cal, patch_dim=4, threads_per_voxel=lanes)
    if spatial:
        kw.update(lam_sp=0.01, lam_dir=0.005)
    with prism.Fitter(vols, prism.options(**kw)) as f, prism.Fitter(vols, prism.options(**kw, fused=0)) as ref:
        before = f.state()
        J, y = f.forward(want_yhat=True)
        g, gg = f.backward()
        Jr, yr = ref.forward(want_yhat=True)
        gr, ggr = ref.backward()
        torch.cuda.synchronize()
        assert np.allclose(J.cpu().numpy(), Jr.cpu().numpy(), rtol=TOL_LOSS, atol=0)
        assert signal_rel(y.cpu().numpy(), yr.cpu().numpy()) <= TOL_SIGNAL
        assert normwise(g.cpu().numpy(), gr.cpu().numpy()) <= TOL_GRAD
        if float(ggr.norm()) > 0:
            assert normwise(gg.cpu().numpy(), ggr.cpu().numpy()) <= TOL_GRAD
        assert f.state() == before
        f.step(2)
        ref.step(2)
        assert np.allclose(f.loss(), ref.loss(), rtol=TOL_LOSS, atol=0)
