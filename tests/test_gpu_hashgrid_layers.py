"""The hash grid's FP32 query and training kernels at the edges of their
tiles (128 rays a query block, 32 a training block) and the Adam pass over
the tables.

Tolerances. The query sums 59 and 64 products in FP32 in order: the FP32 bound
of test_gpu_hashgrid.py (1e-4, 1e-5 on average). The gradient: 1e-3 of the
block's largest value against the oracle with float32 positions, the bound of
test_gpu_hashgrid.py. Adam: equal bits, since the tables' division by a bias
correction is correctly rounded like the general one."""
import numpy as np
import pytest

from oracle import ddf_oracle as O
from paper_2606_00817_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _field(hidden, precision="fp32", table_scale=1.0):
    from paper_2606_00817_gb300 import ddf
    m = ddf.DDF(4, 64, hidden, precision=precision, kind="hashgrid")
    dims = [(64, 59)] + [(64, 64)] * (hidden - 1) + [(2, 64)]
    blob = I.hashgrid_blob(m.n_params, dims, seed=hidden, table_scale=table_scale)
    m.load(blob)
    return ddf, m, blob


def _dev(torch, rays):
    return [torch.from_numpy(a).cuda() for a in rays.soa()]


@pytest.mark.parametrize("hidden", [1, 2, 4])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 1000])
def test_fp32_query_tile_edges(cuda_lib, hidden, n):
    import torch
    _, m, blob = _field(hidden)
    rays = I.uniform_rays(n, seed=n)
    rays.ox[0] = 1.0      # the box's upper face, where the cell index is clamped
    t, v = m.query(_dev(torch, rays))
    r = O.hashgrid_forward(rays.origins(), rays.dirs(), blob, hidden=hidden)
    for g, x in ((t, r["t"]), (v, r["vis"])):
        e = np.abs(g.cpu().numpy() - x) / np.maximum(1.0, np.abs(x))
        assert e.max() <= 1e-3 and e.mean() <= 1e-4


def test_persistent_blocks_cover_every_ray(cuda_lib):
    """More tiles than resident blocks: a ray's result does not depend on
    where in the batch it stands."""
    import torch
    _, m, _ = _field(2)
    n = 152 * 3 * 128 + 77
    rays = _dev(torch, I.uniform_rays(n, seed=1))
    t, v = m.query(rays)
    for lo in (0, 58000, n - 77):
        a, b = m.query([r[lo:lo + 77].clone() for r in rays])
        assert torch.equal(a, t[lo:lo + 77]) and torch.equal(b, v[lo:lo + 77])


@pytest.mark.parametrize("hidden", [1, 3])
@pytest.mark.parametrize("batch", [8, 32, 40, 264])
def test_gradient_tile_edges(cuda_lib, hidden, batch):
    import torch
    ddf, m, blob = _field(hidden, "bf16")
    rays = I.uniform_rays(batch, seed=batch)
    rng = np.random.default_rng(batch)
    tt = rng.uniform(0.1, 3.0, batch).astype(np.float32)
    y = (rng.random(batch) < 0.6).astype(np.uint8)
    loss = torch.zeros(1, device="cuda")
    ddf.ddf_compute_grad(m.h, _dev(torch, rays), torch.from_numpy(tt).cuda(),
                         torch.from_numpy(y).cuda(), batch, loss)
    g = ddf.ddf_get_grad(m.h, m.n_params).astype(np.float64)
    L, ref = O.hashgrid_loss_grad(rays.origins(), rays.dirs(), blob, tt, y, hidden=hidden,
                                  positions="fp32")
    assert abs(float(loss[0]) - L) <= 1e-4 * max(1.0, abs(L))
    table = m.n_params - sum(a * b + a for a, b in [(64, 59)] + [(64, 64)] * (hidden - 1) + [(2, 64)])
    for a, b in ((0, table), (table, m.n_params)):
        assert np.abs(g[a:b] - ref[a:b]).max() <= 1e-3 * np.abs(ref[a:b]).max()


def test_adam_of_the_tables_equals_the_general_one(cuda_lib):
    """An FP32 field's tables go through the general Adam kernel, a bf16
    field's through the pass that divides by the bias corrections with
    Markstein's method: the same bits. Eight rays far apart, so that no table
    entry receives two contributions whose order could differ."""
    import torch
    ddf, a, blob = _field(2, "bf16")
    _, b, _ = _field(2, "fp32")
    sign = np.array([[x, y, z] for x in (-1, 1) for y in (-1, 1) for z in (-1, 1)], np.float64)
    rays = I.Rays.from_arrays(0.83 * sign + 0.01 * np.arange(8)[:, None],
                              sign / np.sqrt(3.0))
    dev = _dev(torch, rays)
    tt = torch.full((8,), 0.7, device="cuda")
    y = torch.tensor([1, 0, 1, 1, 0, 1, 1, 1], dtype=torch.uint8, device="cuda")
    for k in range(5):
        got = []
        for m in (a, b):
            ddf.ddf_train_step(m.h, dev, tt, y, 8, 3e-3)
            got.append((ddf.ddf_get_grad(m.h, m.n_params), ddf.ddf_get_weights(m.h, m.n_params)))
        assert np.array_equal(got[0][0], got[1][0]), k
        assert np.array_equal(got[0][1], got[1][1]), k
    assert not np.array_equal(got[0][1], blob)
