"""Group finalisation by the fused kernel's last CTA (objective, its history, Adam on sigma): a batch of
volumes against each volume's own fit, on both sides of the line where a warp takes each group, in fits that do
take this kernel (one lane per voxel, or neighbour priors), not the many-iteration one."""
import numpy as np
import pytest

import phantoms as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("loss", ["mse", "nll"])
@pytest.mark.parametrize("G", [3, 4, 9])
@pytest.mark.parametrize("opts", [dict(threads_per_voxel=1), dict(threads_per_voxel=4, lam_sp=0.01, lam_dir=0.005)])
def test_batch_of_groups_matches_single_fits(G, loss, opts):
    import paper_2604_00250_gb300 as prism
    vols = [P.random_volume((3 + g % 4, 5, 2 + g), seed=40 + g, mask_density=0.9) for g in range(G)]
    kw = dict(K=2, loss=loss, patch_dim=4, **opts)
    for g, v in enumerate(vols):
        v.init = P.default_init(v.n_vox, 2, g)
    with prism.Fitter(vols, prism.options(**kw)) as f:
        assert f.shape()["iterations_per_launch"] == 1
        f.step(5)
        hist, theta, groups = f.loss_history(), f.params_host(), f.group_view()
    at = 0
    for g, v in enumerate(vols):
        with prism.Fitter([v], prism.options(**kw)) as one:
            one.step(5)
            # the same tile partials in another order of FP64 sums: 1e-12 relative (a few hundred
            # terms at 1.1e-16); sigma follows from them through a rounding to FP32
            assert np.allclose(hist[:, g], one.loss_history()[:, 0], rtol=1e-12 if loss == "mse" else 1e-6, atol=0)
            t = one.params_host()
            assert np.allclose(theta[at:at + v.n_vox], t, rtol=0, atol=0 if loss == "mse" else 3e-4)
            assert abs(groups[g]["sigma_log"] - one.group_view()[0]["sigma_log"]) <= 1e-6
            at += v.n_vox
