"""CTA-pair kernels launched many times over while other kernels come and go
on the same SMs (so that a pair's two CTAs need not start together): every
launch ends, and the results are the same bits each time. A training step's
gradients are summed in a fixed order, so two runs from the same weights agree."""
import numpy as np
import pytest

from paper_2606_00817_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_wide_sdf_training_steps_beside_their_reductions(cuda_lib):
    import torch
    from paper_2606_00817_gb300 import ddf
    net, B, steps = (10, 1280, 8), 65536, 150
    blob = I.xavier_blob_dims(I.sdf_layer_dims(*net))
    pts = torch.from_numpy(np.ascontiguousarray(I.uniform_points(B, seed=7).T)).cuda().float()
    pts = [c.contiguous() for c in pts]
    target = torch.linalg.norm(torch.stack(pts), dim=0) - 0.5
    out = []
    for _ in range(2):
        m = ddf.DDF(*net, kind="sdf")
        m.load(blob)
        loss = torch.zeros(1, device="cuda")
        first = None
        for k in range(steps):
            ddf.ddf_sdf_train_step(m.h, pts, target, B, 1e-4, loss, torch.cuda.current_stream())
            if k == 0:
                first = float(loss.item())
        assert ddf.ddf_check_status(m.h) == 0
        assert 0.0 < float(loss.item()) < first
        out.append(ddf.ddf_get_weights(m.h, m.n_params))
        m.close()
    assert np.array_equal(*out)


@pytest.mark.parametrize("precision,n", [("fp32", 700), ("bf16", 30000)])
def test_queries_beside_another_stream(cuda_lib, precision, n):
    import torch
    from paper_2606_00817_gb300 import ddf
    net = (8, 512, 3)
    m = ddf.DDF(*net, precision=precision)
    m.load(I.xavier_blob(I.NetShape(*net)))
    rays = [torch.from_numpy(x).cuda() for x in I.uniform_rays(n, seed=2).soa()]
    want = [x.clone() for x in m.query(rays)]
    side, x = torch.cuda.Stream(), torch.rand(1 << 22, device="cuda")
    torch.cuda.synchronize()
    for _ in range(100):
        with torch.cuda.stream(side):
            for _ in range(3):
                x = x.sin()
        for g, w in zip(m.query(rays), want):
            assert torch.equal(g, w)
    torch.cuda.synchronize()
    assert ddf.ddf_check_status(m.h) == 0
