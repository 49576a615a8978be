"""The one-kernel query of narrow bf16 fields (width 128 or 256) against the
layer kernels with the default tiles: the same bits, for resident and
streamed weights, one and two tiles a CTA, ragged batches, every kind of
query."""
import numpy as np
import pytest

from paper_2606_00817_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LIGHT = (3.0, 3.0, 3.0)
# resident with two groups; resident with one; streamed at width 128 (6 layers);
# no encoding bands; 16 bands (4 K blocks of layer 1); width 256 streamed; one layer
NETS = [(6, 128, 4), (6, 128, 5), (10, 128, 6), (0, 128, 2), (16, 128, 3), (8, 256, 3),
        (16, 256, 5), (4, 256, 1), (4, 128, 1)]


def _pair(net):
    """The same field twice: on its own, and with the default tiles set, which
    sends it through the layer kernels."""
    from paper_2606_00817_gb300 import ddf
    blob = I.xavier_blob(I.NetShape(*net))
    a, b = ddf.DDF(*net), ddf.DDF(*net)
    for m in (a, b):
        m.load(blob)
    for which in (0, 1):
        ddf.ddf_set_tile(b.h, ddf.ddf_get_tile(b.h, which), which)
    return ddf, a, b


def _dev(torch, rays):
    return [torch.from_numpy(x).cuda() for x in rays.soa()]


@pytest.mark.parametrize("net", NETS)
@pytest.mark.parametrize("n", [1, 127, 128, 129, 257, 152 * 128 + 1, 2 * 152 * 128 + 300])
def test_narrow_query_equals_the_layers(cuda_lib, net, n):
    import torch
    ddf, a, b = _pair(net)
    rays = _dev(torch, I.uniform_rays(n, seed=n))
    for x, y in zip(a.shadow(rays, LIGHT), b.shadow(rays, LIGHT)):
        assert torch.equal(x, y)
    for x, y in zip(a.query(rays), b.query(rays)):
        assert torch.equal(x, y)
    assert ddf.ddf_check_status(a.h) == 0 and ddf.ddf_check_status(b.h) == 0


def test_mixed_graph_noalloc_and_chunks(cuda_lib):
    import torch
    ddf, a, b = _pair((6, 128, 4))
    scene = I.random_scene(16, 0, seed=2)
    sh = _dev(torch, I.shadow_rays(scene, 777, LIGHT, seed=1))
    ao, off = I.ao_rays(scene, 50, seed=3)
    aod, offd = _dev(torch, ao), torch.from_numpy(off).cuda()
    got = []
    for m in (a, b):
        ddf.ddf_set_chunk_rays(m.h, 640)     # joins inside a chunk
        ddf.ddf_set_graph_mode(m.h, True)
        o = [torch.empty(777, device="cuda"), torch.empty(777, device="cuda"),
             torch.empty(777, dtype=torch.uint8, device="cuda"), torch.empty(50, device="cuda"),
             torch.empty(50, device="cuda")]
        for _ in range(2):
            ddf.ddf_query_mixed(m.h, sh, 777, LIGHT, o[0], o[1], o[2], aod, ao.n, offd, 50, o[3],
                                o[4], torch.cuda.current_stream())
        torch.cuda.synchronize()
        got.append(o)
    for x, y in zip(*got):
        assert torch.equal(x, y)
    t, v = torch.empty(777, device="cuda"), torch.empty(777, device="cuda")
    ddf.ddf_query_rays_noalloc(a.h, sh, 777, t, v, torch.cuda.current_stream())
    assert torch.equal(t, got[1][0]) and torch.equal(v, got[1][1])


@pytest.mark.parametrize("net", [(6, 128, 4), (8, 256, 3)])
def test_waits_that_run_out_leave_the_handle_usable(cuda_lib, net):
    """With a limit of 0 ns a wait may give up (a short one may also succeed
    within its first tries): whichever happened, the next query is whole."""
    import torch
    ddf, a, b = _pair(net)
    rays = _dev(torch, I.uniform_rays(5000, seed=5))
    ddf.ddf_set_timeout_ns(a.h, 0)
    a.query(rays)
    ddf.ddf_check_status(a.h)
    ddf.ddf_set_timeout_ns(a.h, 2000000000)
    for x, y in zip(a.query(rays), b.query(rays)):
        assert torch.equal(x, y)
    assert ddf.ddf_check_status(a.h) == 0


def test_autotune_keeps_a_working_choice(cuda_lib):
    import torch
    ddf, a, b = _pair((6, 128, 4))
    rays = _dev(torch, I.uniform_rays(4096, seed=6))
    ddf.ddf_autotune(a.h, rays, 4096)
    t, v = a.query(rays)
    rt, rv = b.query(rays)
    # tiles agree up to the FP32 rounding of the head sums
    assert float((t - rt).abs().max()) <= 1e-5 and float((v - rv).abs().max()) <= 1e-5
