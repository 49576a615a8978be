"""The tables' Adam pass of a bf16 hash grid against the general Adam kernel (an
FP32 field's), where the moments or their quotients by the bias corrections
leave the normal range: the same bits. Eight rays far apart, so that no table
entry receives two contributions whose order could differ."""
import numpy as np
import pytest

from paper_2606_00817_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DIMS = [(64, 59), (64, 64), (2, 64)]


def _steps(blob_of, steps):
    import torch
    from paper_2606_00817_gb300 import ddf
    sign = np.array([[x, y, z] for x in (-1, 1) for y in (-1, 1) for z in (-1, 1)], np.float64)
    rays = I.Rays.from_arrays(0.83 * sign + 0.01 * np.arange(8)[:, None], sign / np.sqrt(3.0))
    dev = [torch.from_numpy(a).cuda() for a in rays.soa()]
    tt = torch.full((8,), 0.7, device="cuda")
    y = torch.tensor([1, 0, 1, 1, 0, 1, 0, 1], dtype=torch.uint8, device="cuda")
    fields = [ddf.DDF(4, 64, 2, precision=p, kind="hashgrid") for p in ("bf16", "fp32")]
    table = fields[0].n_params - sum(a * b + a for a, b in DIMS)
    blob = blob_of(fields[0].n_params)
    for m in fields:
        m.load(blob)
    for k in range(steps):
        got = []
        for m in fields:
            ddf.ddf_train_step(m.h, dev, tt, y, 8, 3e-3)
            got.append((ddf.ddf_get_grad(m.h, m.n_params), ddf.ddf_get_weights(m.h, m.n_params)))
        yield k, table, got, blob


@pytest.mark.parametrize("scale", [1e22, 1e23, 1e24])
def test_second_moments_that_overflow(cuda_lib, scale):
    """A head of weights around `scale` makes table gradients whose second
    moment, or its quotient by 1 - 0.999^t, is an infinity: such an entry moves
    by nothing and stays a number."""
    def blob_of(n):
        b = I.hashgrid_blob(n, DIMS, seed=3, table_scale=1.0)
        b[-2 - 64:-2] *= np.float32(scale)     # the visibility row
        return b
    for k, table, got, _ in _steps(blob_of, 3):
        assert np.array_equal(got[0][0], got[1][0]), k
        assert np.isfinite(got[1][1][:table]).all()
        assert np.array_equal(got[0][1], got[1][1]), k
        if k == 0:
            g = np.abs(got[0][0][:table])
            assert (g > 2e19).any()


@pytest.mark.parametrize("scale", [1e-26, 1e-32, 1e-38, 1e-42])
def test_first_moments_near_and_below_the_normal_range(cuda_lib, scale):
    """Tables of zeros and a head of weights around `scale`: the first step's
    weights are the first moment's quotient by 1 - 0.9^t over the epsilon."""
    def blob_of(n):
        b = I.hashgrid_blob(n, DIMS, seed=4, table_scale=0.0)
        b[-2 - 128:-2] *= np.float32(scale)
        return b
    for k, table, got, _ in _steps(blob_of, 3):
        assert np.array_equal(got[0][0], got[1][0]), k
        assert np.array_equal(got[0][1], got[1][1]), k
        if scale >= 1e-32:       # below, the gradient's sums are subnormal or 0
            assert got[0][1][:table].any()
