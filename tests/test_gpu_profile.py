"""prism_profile runs and times what prism_step runs, also where one launch holds many iterations."""
import numpy as np
import pytest
import torch

import phantoms as P

pytestmark = pytest.mark.gpu


def _step_ms(f, n):
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    f.step(n)
    e1.record()
    e1.synchronize()
    return e0.elapsed_time(e1) / n


@pytest.mark.parametrize("loss", ["mse", "nll"])
@pytest.mark.parametrize("lanes", [4, 16])
def test_small_fit(loss, lanes):
    import paper_2604_00250_gb300 as prism
    vol = P.random_volume((8, 8, 8), seed=2, mask_density=1.0)
    vol.init = P.default_init(vol.n_vox, 3, 2).astype(np.float32)
    kw = dict(K=3, loss=loss, patch_dim=8, threads_per_voxel=lanes)
    with prism.Fitter([vol], prism.options(**kw)) as f, prism.Fitter([vol], prism.options(**kw)) as ref:
        s = f.shape()
        assert s["iterations_per_launch"] == 32
        assert s["fused_grid"] == -(-f.n_vox // s["tile_voxels"])   # a CTA per tile
        ms = f.profile(45)
        ref.step(45)
        assert f.iterations == 45 and f.state() == ref.state()
        assert ms["fused_ms"] == ms["iter_ms"] > 0 and ms["prep_ms"] == ms["group_ms"] == 0
        # the same launches: within a factor of two (another kernel took six times as long)
        assert min(f.profile(64)["iter_ms"] for _ in range(5)) <= 2 * min(_step_ms(ref, 64) for _ in range(5))


@pytest.mark.parametrize("kw", [dict(threads_per_voxel=1), dict(threads_per_voxel=4, lam_sp=0.01), dict(calibration=True),
                                dict(fused=0)])
def test_one_iteration_per_launch(kw):
    import paper_2604_00250_gb300 as prism
    vol = P.random_volume((6, 5, 4), seed=2, mask_density=1.0)
    with prism.Fitter([vol], prism.options(K=2, **kw)) as f:
        assert f.shape()["iterations_per_launch"] == 1
        assert (f.shape()["fused_grid"] > 0) == (kw.get("fused", 1) == 1)
