"""Waits that run out, in every pipelined kernel of a query or a trace. With a
limit of 0 ns a wait gives up once it has outlasted 16 polls, each of which the
hardware may suspend for a while, so the shapes are those with waits of many
microseconds: most have more than one tile a CTA, or K blocks enough. The status
bit must then be set, the kernel ends by itself, and the next call with the
normal limit gives the right bits."""
import numpy as np
import pytest

from paper_2606_00817_gb300 import inputs as I

pytestmark = pytest.mark.gpu

WIDE = (10, 1280, 4)
NORMAL = 2_000_000_000


def _field(net, precision, kind="ray", tiles=False):
    from paper_2606_00817_gb300 import ddf
    m = ddf.DDF(*net, precision=precision, kind=kind)
    if kind == "ray":
        m.load(I.xavier_blob(I.NetShape(*net)),
               np.full(net[2] - 1, 2.0 ** -6, np.float32) if precision == "fp8" else None)
    else:
        m.load(I.xavier_blob_dims(I.sdf_layer_dims(*net), seed=1))
    if tiles:
        for which in (0, 1):
            ddf.ddf_set_tile(m.h, ddf.ddf_get_tile(m.h, which), which)
    return ddf, m


def _gives_up_and_recovers(torch, ddf, m, call):
    want = [x.clone() for x in call()]
    assert ddf.ddf_check_status(m.h) == 0
    ddf.ddf_set_timeout_ns(m.h, 0)
    seen = 0
    for _ in range(5):
        call()
        seen |= ddf.ddf_check_status(m.h)
    ddf.ddf_set_timeout_ns(m.h, NORMAL)
    got = call()
    assert ddf.ddf_check_status(m.h) == 0
    for x, y in zip(got, want):
        assert torch.equal(x, y)
    assert seen & 1


# a few hundred rays (128 x 64 tiles), some thousand (whole and split tiles), the
# default tiles set explicitly, the pair tile and the fused layer 1, FP32 layers,
# one kernel for the whole query
@pytest.mark.parametrize("net,precision,n,tiles", [
    (WIDE, "bf16", 300, False), (WIDE, "fp8", 300, False), (WIDE, "bf16", 4099, False),
    (WIDE, "fp8", 20000, False), (WIDE, "bf16", 65536, True), (WIDE, "fp8", 65536, True),
    (WIDE, "bf16", 65536, False), (WIDE, "fp8", 65536, False), (WIDE, "fp32", 5000, False),
    ((16, 256, 5), "bf16", 60000, False)])
def test_query(cuda_lib, net, precision, n, tiles):
    import torch
    ddf, m = _field(net, precision, tiles=tiles)
    rays = [torch.from_numpy(x).cuda() for x in I.uniform_rays(n, seed=n).soa()]
    _gives_up_and_recovers(torch, ddf, m, lambda: m.query(rays))


# one persistent kernel on clusters of four CTAs and of two; the step kernels
@pytest.mark.parametrize("net,n", [((8, 512, 6), 300), ((8, 256, 4), 3000), ((8, 512, 6), 30000),
                                   ((4, 1280, 3), 5000)])
def test_trace(cuda_lib, net, n):
    import torch
    ddf, m = _field(net, "bf16", kind="sdf")
    rays = [torch.from_numpy(x).cuda() for x in I.uniform_rays(n, seed=n).soa()]

    def call():
        t = torch.zeros(n, device="cuda")
        hit = torch.zeros(n, dtype=torch.uint8, device="cuda")
        steps = torch.zeros(n, dtype=torch.int32, device="cuda")
        ddf.ddf_sphere_trace(m.h, rays, n, 12, 1e-3, 4.0, t, hit, steps,
                             torch.cuda.current_stream())
        torch.cuda.synchronize()
        return t, hit, steps

    _gives_up_and_recovers(torch, ddf, m, call)
