"""FP32 fields whose activations overflow: an infinity goes through the layers
as FP32 FMAs carry it (times a positive weight an infinity, times a negative one
cut by the ReLU), and the other rays of the batch are left alone."""
import numpy as np
import pytest

from oracle import ddf_oracle as O
from paper_2606_00817_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _blob(net):
    """Layer 1's output 0 is 3e38 relu(ox), layer 2's output 0 four times that,
    an infinity from ox = 0.29 on; every output of layer 3 has it with a weight of
    its own (some exact in bf16, some not, of both signs), and the head takes all
    of layer 3 with positive weights into z0 and negative ones into z1."""
    octaves, W, H = net
    assert H == 3
    blob = I.xavier_blob(I.NetShape(*net))
    d = 6 + 12 * octaves
    w1, b1 = blob[:W * d].reshape(W, d), blob[W * d:W * d + W]
    o2 = W * d + W
    w2, b2 = blob[o2:o2 + W * W].reshape(W, W), blob[o2 + W * W:o2 + W * W + W]
    o3 = o2 + W * W + W
    w3 = blob[o3:o3 + W * W].reshape(W, W)
    wo = blob[o3 + W * W + W:-2].reshape(2, W)
    w1[0], b1[0] = 0.0, 0.0
    w1[0, 0] = 3e38
    w2[0], w2[:, 0], b2[0] = 0.0, 0.0, 0.0
    w2[0, 0] = 4.0
    w3[:, 0] = np.resize(np.float32([2.0, 1.2345e-3, -0.777, 0.1, -4.0, 3.0000002]), W)
    wo[0], wo[1] = np.abs(wo[0]) + 1e-3, -np.abs(wo[1]) - 1e-3
    return blob


@pytest.mark.parametrize("width", [256, 768])
@pytest.mark.parametrize("n", [1, 300])
def test_an_infinite_activation_stays_one(cuda_lib, width, n):
    import torch
    from paper_2606_00817_gb300 import ddf
    net = (4, width, 3)
    blob = _blob(net)
    m = ddf.DDF(*net, precision="fp32")
    m.load(blob)
    rays = I.uniform_rays(n, seed=n)
    rays.ox[:] = np.where(np.arange(n) % 3 == 0, 0.5, -np.abs(rays.ox) - 0.01)
    big = rays.ox > 0
    t, v = m.query([torch.from_numpy(a).cuda() for a in rays.soa()])
    t, v = t.cpu().numpy(), v.cpu().numpy()
    assert np.all(t[big] == np.inf) and np.all(v[big] == 0.0)
    if n > 1:
        ex = O.ddf_forward(rays.origins()[~big], rays.dirs()[~big], blob, *net)
        assert np.abs(t[~big] - ex["t"]).max() <= 1e-4 * max(1.0, np.abs(ex["t"]).max())
        assert np.abs(v[~big] - ex["vis"]).max() <= 1e-4
    assert ddf.ddf_check_status(m.h) == 0
