"""An alpha gradient that overflows stays infinite through the sums over tiles (it does not become a NaN)."""
import numpy as np
import pytest
import torch

import phantoms as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lanes", [1, 4, 16])
def test_overflowing_alpha_gradient(lanes):
    import paper_2604_00250_gb300 as prism
    vol = P.random_volume((6, 6, 9), seed=3, mask_density=1.0)
    th = P.default_init(vol.n_vox, 2, 1).astype(np.float32)
    th[7, 0] = 1e25   # S0 = 1e25: r S overflows, r and S do not
    vol.init = th
    with prism.Fitter([vol], prism.options(K=2, calibration=True, threads_per_voxel=lanes)) as f:
        f.forward()
        _, g = f.backward()
        off = f.group_layout()
        alpha = g[int(off[1]):int(off[1]) + f.n_meas[0]]
        b0 = torch.as_tensor(np.asarray(vol.bvals) == 0).cuda()
        assert bool(torch.isposinf(alpha[b0]).all())
        assert not bool(torch.isnan(alpha).any())
