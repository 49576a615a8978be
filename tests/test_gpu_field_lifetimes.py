"""Fields that are made, loaded, queried and destroyed in a row: a later field's
weights and the maps of them may lie where an earlier one's did, and its
queries must still read its own."""
import numpy as np
import pytest

from paper_2606_00817_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nets", [[(6, 128, 4)], [(8, 256, 3)], [(6, 128, 4), (10, 128, 6), (4, 256, 1)]])
def test_each_narrow_field_reads_its_own_weights(cuda_lib, nets):
    """The one-kernel query against the layer kernels (default tiles set
    explicitly), the same bits, for 24 short-lived fields one after another."""
    import torch
    from paper_2606_00817_gb300 import ddf
    rays = [torch.from_numpy(x).cuda() for x in I.uniform_rays(300, seed=1).soa()]
    seen = []
    for k in range(24):
        net = nets[k % len(nets)]
        blob = I.xavier_blob(I.NetShape(*net), seed=k)
        a, b = ddf.DDF(*net), ddf.DDF(*net)
        for m in (a, b):
            m.load(blob)
        for which in (0, 1):
            ddf.ddf_set_tile(b.h, ddf.ddf_get_tile(b.h, which), which)
        got, want = a.query(rays), b.query(rays)
        for x, y in zip(got, want):
            assert torch.equal(x, y), k
        assert ddf.ddf_check_status(a.h) == 0
        seen.append(got[0].cpu().numpy())
        a.close()
        b.close()
    assert not np.array_equal(seen[0], seen[len(nets)])
