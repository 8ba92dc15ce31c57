"""The many-iteration kernel called for few iterations at a time: the objective's history bit for bit that of long
calls, also where a volume has more tiles than a CTA has threads, and no cost beyond a call's own."""
import numpy as np
import pytest
import torch

import phantoms as P

pytestmark = pytest.mark.gpu


def _fitter(shape, lanes, **kw):
    import paper_2604_00250_gb300 as prism
    vol = P.random_volume(shape, seed=8, mask_density=1.0)
    vol.init = P.default_init(vol.n_vox, 2, 8).astype(np.float32)
    f = prism.Fitter([vol], prism.options(K=2, patch_dim=16, threads_per_voxel=lanes, **kw))
    assert f.shape()["iterations_per_launch"] == 32
    return f


@pytest.mark.parametrize("loss", ["mse", "nll"])
@pytest.mark.parametrize("shape,lanes", [((14, 14, 14), 16), ((2, 2, 2), 16), ((9, 8, 14), 16), ((14, 14, 14), 4)])
def test_history_does_not_depend_on_the_calls(shape, lanes, loss):
    with _fitter(shape, lanes, loss=loss) as a, _fitter(shape, lanes, loss=loss) as b:
        for n in (1, 2, 3, 4, 1, 5, 33):
            a.step(n)
        b.step(49)
        assert np.array_equal(a.loss_history(), b.loss_history()) and np.array_equal(a.loss(), b.loss())
        assert a.state() == b.state()


def test_single_iteration_calls():
    """32,768 voxels in 4,096 tiles, MSE: 32 calls of one iteration against one of 32. A call's own cost (launch,
    tiles in and out) is below an iteration's here; one warp summing every tile's objective took four iterations'."""
    with _fitter((32, 32, 32), 16, loss="mse") as f:
        def ms(calls, n):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(calls):
                f.step(n)
            e1.record()
            e1.synchronize()
            return e0.elapsed_time(e1)
        f.step(32)
        assert min(ms(32, 1) for _ in range(5)) <= 2.5 * min(ms(1, 32) for _ in range(5))
