"""The objective of prism_forward on a fused handle: sums of many like terms within one voxel keep their accuracy.

Volumes of one voxel whose N = 1,024 measurements all have b = 0 and the same signal: every term of a voxel's data
term is the same, so a sum in FP32 drifts by up to 1e-5 of its value (each addition rounds the same way until the
sum doubles), while FP64 sums, or FP32 sums of one ring stage added up exactly, do not."""
import types

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

N, K, G = 1024, 2, 64
# Roundings of 2^-24: a term (2), its stage's sum (up to 32 additions and the fold of two halves): 35 units, 2.1e-6
# of the sum of magnitudes. The prediction handed out may differ from the one in the sum by two units: of a
# residual of at least 0.3 at a prediction of at most 0.7, 6e-7 of r^2.
TOL = 2.7e-6


@pytest.mark.parametrize("lanes,shells", [(1, 0), (1, -1), (4, 0), (4, -1), (16, 0)])
@pytest.mark.parametrize("loss", ["mse", "nll"])
@pytest.mark.parametrize("cal", [False, True])
def test_like_terms(lanes, shells, loss, cal):
    import paper_2604_00250_gb300 as prism
    sp = pytest.importorskip("scipy.special")
    rng = np.random.default_rng(0)
    vols = []
    for _ in range(G):
        th = rng.normal(0, 0.3, (1, 4 * K + 5)).astype(np.float32)
        th[0, 0] = np.log(np.expm1(rng.uniform(0.2, 0.7)))
        vols.append(types.SimpleNamespace(mask=np.ones((1, 1, 1), np.uint8), signal=np.full((1, N), 1024.0, np.float32),
                                          bvals=np.zeros(N, np.float32), bvecs=np.zeros((N, 3), np.float32), init=th))
    o = prism.options(K=K, loss=loss, calibration=cal, threads_per_voxel=lanes, shells=shells, lam_rep=0.0, lam_sparse=0.0)
    with prism.Fitter(vols, o) as f:
        off, g = f.group_layout(), f.groups()
        g[off[:-1:4]] = -1.2
        J, y = f.forward(groups=torch.as_tensor(g).cuda(), want_yhat=True)
        J, y = J.cpu().numpy(), y.cpu().numpy().astype(np.float64).reshape(G, N)
    if loss == "mse":
        terms = [(1.0 - y) ** 2]
    else:
        s = float(np.float32(-1.2))
        terms = [np.full_like(y, 2 * s), (1.0 - y) ** 2 / (2 * np.exp(2 * s)), -np.log(sp.i0e(y * np.exp(-2 * s)))]
    want, size = sum(t.sum(1) for t in terms), sum(np.abs(t).sum(1) for t in terms)
    assert np.max(np.abs(J - want) / size) <= TOL
