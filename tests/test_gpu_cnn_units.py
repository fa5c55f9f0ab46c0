"""The depth of the network's units follows the number of units of all boxes
(2, 4 or 8 depths): the same image alone (shallow units) and among copies of
itself (deep ones) gives the same prediction bit for bit."""
import numpy as np
import pytest

from paper_2505_03067_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,copies", [((32, 32, 32), 6), ((48, 48, 40), 2), ((33, 17, 31), 7), ((24, 40, 5), 16)])
def test_prediction_does_not_depend_on_the_units_depth(dims, copies):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2505_03067_gb300 import build, mpm as M
    build.build()
    wl = W.random_case(sum(dims), dims, nspecies=3, p_mask=0.7)
    ctx = M.Context()
    lat, prm = M.DeviceLattice(wl.lattice), M.DeviceParams(wl.params)
    cnn = M.CNN(ctx, dims, copies, M.cnn_init_params(3, last_scale=0.3), s_out=0.3)
    box = ((0, 0, 0), dims)
    for b in range(copies):
        cnn.load_image(b, lat, prm, box, M.CNN_INPUT)
    one = cnn.forward(1).cpu().numpy()
    many = cnn.forward(copies).cpu().numpy().reshape(copies, -1, 3)
    on = wl.lattice.mask.reshape(-1) > 0
    assert np.isfinite(one[:on.size][on]).all()
    for b in range(copies):
        assert np.array_equal(many[b][on], one[:on.size][on]), b
