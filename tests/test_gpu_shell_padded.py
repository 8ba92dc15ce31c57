"""The shell loop with padded odd shells (32,768 voxels and more) against the plain kernels and the
per-measurement loop: gradient per block, objective, a short trajectory, and y_hat in the caller's order."""
import numpy as np
import pytest
import torch

import phantoms as P
from tests.helpers import TOL_GRAD, TOL_LOSS, TOL_SIGNAL, block_slices, normwise, signal_rel

pytestmark = pytest.mark.gpu

SCHEMES = {
    "odd": (3, [(1000, 7), (2500, 5)]),            # every shell odd
    "one_odd": (2, [(45, 3), (1000, 6), (2500, 6)]),
    "single": (1, [(700, 1), (1400, 1), (2100, 1)]),   # shells of one measurement
    "chunk": (1, [(800, 31), (1600, 33)]),         # a shell's end on either side of a 32-measurement chunk
    "even_k5": (2, [(1000, 6), (2500, 8)]),
}


@pytest.mark.parametrize("name", sorted(SCHEMES))
@pytest.mark.parametrize("K", [1, 3, 4, 5])
def test_padded_shells(name, K):
    import paper_2604_00250_gb300 as prism
    from phantoms import schemes
    sch = schemes.make_scheme(*SCHEMES[name], 7)
    order = np.random.default_rng(1).permutation(len(sch[0]))
    vol = P.random_volume((33, 33, 31), scheme=(sch[0][order], sch[1][order]), seed=3, mask_density=0.98)
    assert vol.n_vox >= 32768
    rng = np.random.default_rng(K)
    vol.init = (P.default_init(vol.n_vox, K, 2) + rng.normal(0, 0.2, (vol.n_vox, 4 * K + 5))).astype(np.float32)
    kw = dict(K=K, threads_per_voxel=1, lam_sp=0.01, lam_dir=0.005)
    out = {}
    for form, extra in (("pad", {}), ("loop", dict(shells=-1)), ("plain", dict(fused=0))):
        with prism.Fitter([vol], prism.options(**kw, **extra)) as f:
            if form != "plain":
                assert f.shape()["shell_loop"] == (1 if form == "pad" else 0)
            J, y = f.forward(want_yhat=True)
            g, _ = f.backward()
            torch.cuda.synchronize()
            f.step(3)
            out[form] = (float(J[0]), y.cpu().numpy(), g.cpu().numpy(), f.loss()[0])
    for form in ("pad", "loop"):
        assert abs(out[form][0] - out["plain"][0]) <= TOL_LOSS * abs(out["plain"][0])
        assert signal_rel(out[form][1], out["plain"][1]) <= TOL_SIGNAL
        for block, sl in block_slices(K).items():
            assert normwise(out[form][2][:, sl], out["plain"][2][:, sl]) <= TOL_GRAD, (form, block)
        assert abs(out[form][3] - out["plain"][3]) <= TOL_LOSS * abs(out["plain"][3])
