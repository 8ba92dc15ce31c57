"""The calibrated shell loop's per-measurement sums (dJ/dalpha_n, dJ/dbeta_n) go through shared memory four pairs
of a lane at a time: pair counts around the multiples of four (one lane per voxel) and sixteen (four lanes),
of a chunk's sixteen pairs, and voxel counts that leave lanes and whole warps of a tile idle, each block of the
gradient against the plain kernels' (tolerance of the gradient tests). 600 measurements with one lane leave no
room for the staging rows: there the sums go by shuffles."""
import numpy as np
import pytest
import torch

import phantoms as P
from tests.helpers import TOL_GRAD, normwise

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lanes", [1, 4])
@pytest.mark.parametrize("loss", ["mse", "nll"])
@pytest.mark.parametrize("n_meas", [8, 10, 30, 32, 33, 34, 39, 95, 131, 600])
@pytest.mark.parametrize("shape", [(5, 1, 1), (11, 4, 3)])
def test_alpha_beta_gradients(lanes, loss, n_meas, shape):
    import paper_2604_00250_gb300 as prism
    from phantoms import schemes
    K, h = 2, (n_meas - 2) // 2
    sch = schemes.make_scheme(2, [(900, h), (2600, n_meas - 2 - h)], 6)
    vol = P.random_volume(shape, scheme=sch, seed=n_meas, mask_density=1.0, calibration=True)
    rng = np.random.default_rng(5)
    vol.init = (P.default_init(vol.n_vox, K, 1) + rng.normal(0, 0.2, (vol.n_vox, 4 * K + 5))).astype(np.float32)
    kw = dict(K=K, loss=loss, calibration=True, threads_per_voxel=lanes)
    with prism.Fitter([vol], prism.options(**kw)) as f, prism.Fitter([vol], prism.options(**kw, fused=0)) as ref:
        f.forward()
        ref.forward()
        gg, rr = f.backward()[1], ref.backward()[1]
        torch.cuda.synchronize()
        a, b = f.group_view(gg.cpu().numpy())[0], ref.group_view(rr.cpu().numpy())[0]
    for name in ("alpha", "beta"):
        assert np.any(b[name] != 0) and normwise(a[name], b[name]) <= TOL_GRAD, name
