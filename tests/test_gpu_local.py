"""Fits without neighbour priors and calibration run many iterations per launch (several lanes per voxel):
the same parameters, moments and history as one iteration per call, bit for bit (each voxel's
arithmetic is the same, and the objective's sums take the same order for the same tiles)."""
import numpy as np
import pytest

import phantoms as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lanes", [4, 16])
@pytest.mark.parametrize("optimizer,loss", [("adam", "mse"), ("rprop", "mse"), ("adam", "nll"), ("rprop", "nll")])
@pytest.mark.parametrize("N", [96, 193])
def test_many_iterations_per_launch(lanes, optimizer, loss, N):
    import paper_2604_00250_gb300 as prism
    from phantoms import schemes
    sch = schemes.scheme_96(3) if N == 96 else schemes.scheme_193(3)
    vols = [P.random_volume(s, scheme=sch, seed=60 + i, mask_density=0.8)
            for i, s in enumerate([(11, 7, 5), (3, 3, 1), (2, 1, 1), (6, 9, 4)])]
    kw = dict(K=2, loss=loss, patch_dim=5, threads_per_voxel=lanes, optimizer=optimizer)
    with prism.Fitter(vols, prism.options(**kw)) as one, prism.Fitter(vols, prism.options(**kw)) as many:
        for n in (1, 5, 33, 64):
            for _ in range(n):
                one.step(1)
            many.step(n)
            assert many.iterations == one.iterations
            assert np.array_equal(one.params_host(), many.params_host())
        a = one.state()
        assert a == many.state()
        assert np.array_equal(one.loss_history(), many.loss_history())
        many.load_state(a)
        many.step(40)
        for _ in range(40):
            one.step(1)
        assert np.array_equal(one.params_host(), many.params_host())
        many.sync()


@pytest.mark.parametrize("lanes", [4, 16])
@pytest.mark.parametrize("K,N", [(1, 21), (3, 96), (5, 97), (4, 8)])
@pytest.mark.parametrize("loss", ["mse", "nll"])
def test_gradient_against_the_oracle(lanes, K, N, loss):
    """One iteration from zero moments leaves m = (1 - beta1) g in the checkpoint: g per block against
    the FP64 oracle's gradient (tolerances of tests/helpers.py), and the objective."""
    import paper_2604_00250_gb300 as prism
    import torch
    from oracle import prism_oracle as O
    from phantoms import schemes
    from tests.helpers import TOL_GRAD, TOL_LOSS, block_slices, normwise
    sch = schemes.make_scheme(2, [(900, (N - 2) // 2), (2600, N - 2 - (N - 2) // 2)], 5)
    vol = P.random_volume((7, 5, 3), scheme=sch, seed=K, mask_density=0.9)
    rng = np.random.default_rng(7)
    th = (P.default_init(vol.n_vox, K, 2) + rng.normal(0, 0.2, (vol.n_vox, 4 * K + 5))).astype(np.float32)
    vol.init = th
    with prism.Fitter([vol], prism.options(K=K, loss=loss, threads_per_voxel=lanes)) as f:
        groups = f.group_view()[0]
        f.step(1)
        blob = f.state()
        J = f.loss()[0]
        n = vol.n_vox * f.Q
        at = len(blob) - 12 * (n + f.n_group_params) + 4 * n
        g = np.frombuffer(blob, np.float32, n, at).reshape(-1, f.Q) / np.float32(0.1)
    o = O.Options(K=K, loss=loss, patch_dim=16)
    ov = O.OracleVolume(vol.mask, vol.signal, vol.bvals, vol.bvecs, o)
    gp = O.group_init(ov)
    gp["sigma_log"] = torch.tensor(groups["sigma_log"], dtype=torch.float64)
    Jr, _, gr, _ = O.value_and_grad(ov, torch.as_tensor(th).double(), gp, n_norm=ov.n_mask)
    assert abs(J - float(Jr)) <= TOL_LOSS * abs(float(Jr))
    for name, sl in block_slices(K).items():
        assert normwise(g[:, sl], gr.numpy()[:, sl]) <= TOL_GRAD, name



@pytest.mark.parametrize("n_vols", [3, 700])
def test_objectives_of_many_volumes(n_vols):
    """Each volume's objectives are summed by the CTA that finishes its last tile; 700 one-tile volumes are
    more tiles than CTAs. A volume's history is that of its lone fit, bit for bit (same tiles, same sums)."""
    import paper_2604_00250_gb300 as prism
    from phantoms import schemes
    sch = schemes.scheme_96(3)
    vols = [P.random_volume((2, 2, 1 + i % 2), scheme=sch, seed=900 + i, mask_density=1.0) for i in range(n_vols)]
    for i, v in enumerate(vols):
        v.init = P.default_init(v.n_vox, 2, i).astype(np.float32)
    kw = dict(K=2, loss="mse", patch_dim=4, threads_per_voxel=16)
    at = np.cumsum([0] + [v.n_vox for v in vols])
    with prism.Fitter(vols, prism.options(**kw)) as f:
        f.step(37)
        f.step(2)
        h, J, th = f.loss_history(), f.loss(), f.params_host()
    assert h.shape == (39, n_vols)
    for i in (0, 1, n_vols // 2, n_vols - 1):
        with prism.Fitter([vols[i]], prism.options(**kw)) as f:
            f.step(39)
            assert np.array_equal(f.loss_history()[:, 0], h[:, i])
            assert f.loss()[0] == J[i]
            assert np.array_equal(f.params_host(), th[at[i]:at[i + 1]])
