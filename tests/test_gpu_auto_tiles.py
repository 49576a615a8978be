"""The tiles a field takes by itself, by the size of the batch, where nobody
set any: the same bits as the default tiles set explicitly, on both sides of
each line, for bf16, e4m3 and SDF fields, with and without the fused layer 1."""
import numpy as np
import pytest

from paper_2606_00817_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LIGHT = (3.0, 3.0, 3.0)
# rows: one, small batches (narrow column tiles up to two waves of them), the line of the
# pair tiles and past it, a chunk's remainder
ROWS = [1, 100, 129, 700, 2000, 10239, 10240, 10369]


def _pair(net, precision="bf16", kind="ray"):
    """The same field twice; the second with the default tiles set."""
    from paper_2606_00817_gb300 import ddf
    a, b = (ddf.DDF(*net, precision=precision, kind=kind) for _ in range(2))
    blob = I.xavier_blob(I.NetShape(*net)) if kind == "ray" else \
        I.xavier_blob_dims(I.sdf_layer_dims(*net))
    for m in (a, b):
        m.load(blob, np.full(net[2] - 1, 2.0 ** -6, np.float32) if precision == "fp8" else None)
    for which in (0, 1):
        ddf.ddf_set_tile(b.h, ddf.ddf_get_tile(b.h, which), which)
    return ddf, a, b


def _dev(torch, rays):
    return [torch.from_numpy(x).cuda() for x in rays.soa()]


@pytest.mark.parametrize("net,precision", [((10, 512, 4), "bf16"), ((10, 512, 4), "fp8"),
                                           ((12, 768, 3), "bf16"), ((4, 512, 1), "bf16"),
                                           ((4, 512, 2), "fp8"), ((10, 1280, 2), "bf16"),
                                           ((10, 384, 3), "bf16")])
def test_sizes_choose_tiles_with_the_same_results(cuda_lib, net, precision):
    import torch
    ddf, a, b = _pair(net, precision)
    rays = _dev(torch, I.uniform_rays(max(ROWS), seed=3))
    for n in ROWS:
        part = [r[:n].contiguous() for r in rays]
        for x, y in zip(a.shadow(part, LIGHT), b.shadow(part, LIGHT)):
            assert torch.equal(x, y), n
    ddf.ddf_set_chunk_rays(a.h, 10300)   # a large chunk, then a small one
    for x, y in zip(a.query(rays), b.query(rays)):
        assert torch.equal(x, y)
    for m in (a, b):                     # the same through a graph
        ddf.ddf_set_graph_mode(m.h, True)
    for n in (700, 10369):
        part = [r[:n].contiguous() for r in rays]
        for x, y in zip(a.shadow(part, LIGHT), b.shadow(part, LIGHT)):
            assert torch.equal(x, y), n
    assert ddf.ddf_check_status(a.h) == 0 and ddf.ddf_check_status(b.h) == 0


def test_sdf_values_do_not_depend_on_the_choice(cuda_lib):
    import torch
    ddf, a, b = _pair((8, 512, 4), kind="sdf")
    pts = torch.from_numpy(I.uniform_points(12000, seed=4)).cuda().T.float().contiguous()
    for n in (1, 129, 2000, 10240, 12000):
        out = []
        for m in (a, b):
            s = torch.empty(n, device="cuda")
            ddf.ddf_sdf_eval(m.h, [c[:n].contiguous() for c in pts], n, s, torch.cuda.current_stream())
            out.append(s)
        torch.cuda.synchronize()
        assert torch.equal(*out), n


def test_noalloc_follows_the_same_rule(cuda_lib):
    import torch
    ddf, a, b = _pair((10, 1280, 3))
    for n in (1, 193, 1500, 4099):
        rays = _dev(torch, I.uniform_rays(n, seed=n))
        t, v = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
        ddf.ddf_query_rays_noalloc(a.h, rays, n, t, v, torch.cuda.current_stream())
        rt, rv = b.query(rays)
        assert torch.equal(t, rt) and torch.equal(v, rv), n


@pytest.mark.parametrize("net,precision", [((10, 1280, 3), "bf16"), ((10, 1280, 3), "fp8"),
                                           ((8, 512, 2), "bf16"), ((10, 384, 3), "fp8")])
@pytest.mark.parametrize("n", [2001, 3963, 4099, 4864, 4865, 5760, 5761, 7801, 9729])
def test_layers_cut_into_whole_and_split_tiles(cuda_lib, net, precision, n):
    """Between the small batches and the pair tiles: whole waves of wide tiles
    and what is left of them split in two or four, with and without room for the
    last layer's activations, the same bits as the default tiles."""
    import torch
    ddf, a, b = _pair(net, precision)
    rays = _dev(torch, I.uniform_rays(n, seed=n))
    want = b.query(rays)
    for x, y in zip(a.query(rays), want):
        assert torch.equal(x, y)
    if n <= 5761:                        # the static scratch holds 6,061 rays of the widest
        t, v = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
        ddf.ddf_query_rays_noalloc(a.h, rays, n, t, v, torch.cuda.current_stream())
        assert torch.equal(t, want[0]) and torch.equal(v, want[1])
    assert ddf.ddf_check_status(a.h) == 0


@pytest.mark.parametrize("net,precision,n", [((4, 768, 2), "bf16", 38911), ((4, 768, 2), "bf16", 38912),
                                             ((4, 768, 2), "fp8", 64853), ((4, 768, 2), "fp8", 64854),
                                             ((4, 384, 2), "bf16", 70001), ((4, 768, 1), "bf16", 896)])
def test_the_line_of_the_pair_tiles(cuda_lib, net, precision, n):
    """Six waves of wide tiles on 152 SMs (e4m3 ten); fields without pair tiles
    have no such line; a single layer."""
    import torch
    ddf, a, b = _pair(net, precision)
    rays = _dev(torch, I.uniform_rays(n, seed=5))
    for x, y in zip(a.shadow(rays, LIGHT), b.shadow(rays, LIGHT)):
        assert torch.equal(x, y)
    assert ddf.ddf_check_status(a.h) == 0
