"""The FP32 layers on the tensor cores (widths that are multiples of 256),
every operand split into three bf16 values.

Tolerances: every ray within the FP32 bound 1e-4 of the exact oracle, and
normwise 1e-6: a pre-activation is a sum of K / 32 blocks and some 12
roundings inside one, each of 2^-24 of the running sum, so a random walk of
about 52 steps a layer (at K = 1280) over at most 8 layers gives
2^-24 sqrt(8 x 52) = 1.2e-6 of sums of order one, and the widths here are
smaller (K <= 512, 3 layers: 5e-7)."""
import numpy as np
import pytest

from oracle import ddf_oracle as O
from paper_2606_00817_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _field(net, scale=1.0):
    from paper_2606_00817_gb300 import ddf
    blob = I.xavier_blob(I.NetShape(*net)) * np.float32(scale)
    m = ddf.DDF(*net, precision="fp32")
    m.load(blob)
    return ddf, m, blob


def _dev(torch, rays):
    return [torch.from_numpy(a).cuda() for a in rays.soa()]


# one row, the edges of the 128-row halves and the 256-row tile; K of layer 1
# below, at and above one 64-wide block; one layer, which is first and last
@pytest.mark.parametrize("net", [(0, 256, 1), (4, 256, 2), (10, 512, 3), (16, 768, 2)])
@pytest.mark.parametrize("n", [1, 127, 129, 255, 256, 257, 700])
def test_split_layers_match_exact_oracle(cuda_lib, net, n):
    import torch
    ddf, m, blob = _field(net)
    rays = I.uniform_rays(n, seed=n)
    t, v = m.query(_dev(torch, rays))
    ex = O.ddf_forward(rays.origins(), rays.dirs(), blob, *net)
    for g, r in ((t, ex["t"]), (v, ex["vis"])):
        e = np.abs(g.cpu().numpy().astype(np.float64) - r)
        assert (e / np.maximum(1.0, np.abs(r))).max() <= 1e-4
        assert np.sqrt(np.mean(e ** 2)) <= 1e-6 * max(1.0, np.sqrt(np.mean(r ** 2)))
    assert ddf.ddf_check_status(m.h) == 0


def test_passes_of_the_rows_and_the_static_scratch_agree(cuda_lib):
    """More rows than one pass takes, and the allocation-free query, which
    takes fewer at a time: the same bits."""
    import torch
    ddf, m, _ = _field((6, 256, 2))
    n = 131072 + 129
    rays = _dev(torch, I.uniform_rays(n, seed=3))
    t, v = m.query(rays)
    for lo, k in ((0, 300), (131072 - 200, 329), (1000, 11000)):
        part = [r[lo:lo + k].clone() for r in rays]
        a, b = torch.empty(k, device="cuda"), torch.empty(k, device="cuda")
        ddf.ddf_query_rays_noalloc(m.h, part, k, a, b, torch.cuda.current_stream())
        assert torch.equal(a, t[lo:lo + k]) and torch.equal(b, v[lo:lo + k])


def test_rows_that_are_not_finite_leave_the_others_alone(cuda_lib):
    import torch
    net = (6, 256, 3)
    ddf, m, blob = _field(net)
    rays = I.uniform_rays(300, seed=4)
    clean = m.query(_dev(torch, rays))
    for k, (i, x) in enumerate(((7, np.nan), (130, np.inf), (299, -np.inf), (40, 1e30))):
        rays.soa()[k][i] = x
    t, v = m.query(_dev(torch, rays))
    keep = np.ones(300, bool)
    keep[[7, 130, 299, 40]] = False
    keep = torch.from_numpy(keep).cuda()
    assert torch.equal(t[keep], clean[0][keep]) and torch.equal(v[keep], clean[1][keep])
    # a NaN coordinate makes every pre-activation NaN, which the ReLU takes to
    # 0, so the row's outputs are those of zero activations in layer 2
    assert torch.isfinite(t[~keep][:1]).all()


@pytest.mark.parametrize("n", [1, 256, 769, 1025, 2048, 3841, 4097, 5000])
def test_whole_and_split_tiles_agree(cuda_lib, n):
    """At width 1280 five tiles per 256 rows: batches of less than a wave of
    them in four or two parts, a wave and a rest, and the last rows of a batch
    of several waves: the same bits."""
    import torch
    ddf, m, _ = _field((4, 1280, 2))
    rays = _dev(torch, I.uniform_rays(16387, seed=6))
    t, v = m.query(rays)
    a, b = m.query([r[-n:].clone() for r in rays])
    assert torch.equal(a, t[-n:]) and torch.equal(b, v[-n:])
    assert ddf.ddf_check_status(m.h) == 0
