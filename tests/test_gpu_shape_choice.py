"""The automatic lanes per voxel of Rician fits without neighbour priors and calibration: sixteen only where all tiles
of eight voxels are resident at once (the many-iteration kernel's condition), else four."""
import numpy as np
import pytest

import phantoms as P

pytestmark = pytest.mark.gpu


def _cube(K, n):
    from phantoms import schemes
    v = P.random_volume((16, 16, 16), scheme=schemes.make_scheme(3, [(900, n - 3)], 5), seed=1, mask_density=1.0)
    return [v], dict(K=K, patch_dim=16)


def _many(n_vols):
    """More volumes than resident CTAs, each with one tile whatever the lanes."""
    from phantoms import schemes
    sch = schemes.make_scheme(2, [(900, 10)], 5)
    return [P.random_volume((5, 1, 1), scheme=sch, seed=i, mask_density=1.0) for i in range(n_vols)], dict(K=2, patch_dim=8)


# 4,096 voxels are 512 tiles of 8 or 128 of 32, on 152 SMs: K <= 3 takes four CTAs an SM at small N, K = 5 at most
# three, N = 1,000 (52 KB of table and signal, and state, a tile) three; 900 volumes exceed 608 CTAs
@pytest.mark.parametrize("make,lanes", [(lambda: _cube(3, 40), 16), (lambda: _cube(5, 40), 4), (lambda: _cube(3, 1000), 4),
                                        (lambda: _many(900), 4)])
def test_lanes_of_small_rician_fits(make, lanes):
    import paper_2604_00250_gb300 as prism
    vols, kw = make()
    for i, v in enumerate(vols):
        v.init = P.default_init(v.n_vox, kw["K"], i).astype(np.float32)
    with prism.Fitter(vols, prism.options(loss="nll", **kw)) as f:
        assert 2048 <= f.n_vox < 4200 or len(vols) > 1
        assert f.shape()["threads_per_voxel"] == lanes
        f.step(3)
        f.sync()
        assert np.all(np.isfinite(f.params_host())) and np.all(np.diff(f.loss_history().sum(1)) < 0)
