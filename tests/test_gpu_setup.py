"""Set-up kernels at the edges of their blocks: refused signals (and how many voxels are named), and
parameters through the [V][Q] <-> slot layout."""
import numpy as np
import pytest

import phantoms as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slabs", [None, (4, 1)])
@pytest.mark.parametrize("lanes", [1, 4, 16])
def test_refused_signals_are_counted_once(lanes, slabs):
    import paper_2604_00250_gb300 as prism
    from phantoms import schemes
    sch = schemes.make_scheme(9, [(1000, 70), (2500, 71)], 1)
    order = np.random.default_rng(0).permutation(150)
    vol = P.random_volume((7, 6, 4), scheme=(sch[0][order], sch[1][order]), seed=1, mask_density=0.9)
    b0 = np.flatnonzero(vol.bvals == 0)
    dw = np.flatnonzero(vol.bvals > 0)
    clean = vol.signal.copy()
    V = vol.n_vox

    def refused(edit):
        vol.signal = clean.copy()
        edit(vol.signal)
        with pytest.raises(prism.PrismError) as e:
            prism.Fitter([vol], prism.options(K=2, threads_per_voxel=lanes), slabs=slabs)
        assert e.value.code == 5
        return int(str(e.value).split("E_NONFINITE: ")[1].split()[0])

    def put(*cells):
        def edit(s):
            for v, n, x in cells:
                s[v, n] = x
        return edit

    assert refused(put((0, dw[0], np.nan))) == 1
    assert refused(put((V - 1, dw[-1], np.inf), (V - 1, dw[3], -np.inf))) == 1
    assert refused(put((5, b0[2], np.nan), (5, dw[9], np.nan))) == 1      # mean and row: one voxel
    assert refused(put((31, b0[-1], -np.inf), (32, b0[0], np.inf), (33, dw[1], np.nan))) == 3

    def zero_mean(s):
        s[7, b0] = 0.0
    assert refused(zero_mean) == 1
    vol.signal = clean
    with prism.Fitter([vol], prism.options(K=2, threads_per_voxel=lanes), slabs=slabs) as f:
        f.step(2)
        f.sync()


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("V", [1, 127, 128, 129, 300])
def test_parameters_round_trip(K, V):
    import paper_2604_00250_gb300 as prism
    mask = np.zeros((10, 10, 5), np.uint8)
    mask.flat[np.random.default_rng(V).permutation(500)[:V]] = 1
    base = P.random_volume((10, 10, 5), seed=2)
    base.mask, base.signal = mask, base.signal[mask.ravel().astype(bool)]
    with prism.Fitter([base], prism.options(K=K, patch_dim=3)) as f:
        th = np.random.default_rng(K).normal(size=(V, 4 * K + 5)).astype(np.float32)
        f.set_params(th)
        assert np.array_equal(f.params_host(), th)
        assert np.array_equal(f.params().cpu().numpy(), th)
