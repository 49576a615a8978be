"""The one-kernel sphere trace (SDF fields of width 128 to 512) against the
step-by-step kernels, which a field with explicitly set tiles takes: t, hit and
steps bit for bit, for every cluster size, fewer rays than lanes and many more,
step limits and rays that never end by themselves."""
import numpy as np
import pytest

from paper_2606_00817_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _sphere_blob(net, seed, radius=0.6):
    """Weights close to |p| - radius: layer 1 holds unit directions (|p| is 4
    times the mean of relu(n . p) over them) and a little of every band, the
    layers between pass it on, the head sums it up."""
    octaves, W, H = net
    rng = np.random.default_rng(seed)
    d_in = 3 + 6 * octaves
    w1 = rng.uniform(-0.01, 0.01, (W, d_in))
    v = rng.normal(size=(W, 3))
    w1[:, :3] = v / np.linalg.norm(v, axis=1, keepdims=True)
    parts = [w1.ravel(), np.zeros(W)]
    for _ in range(H - 1):
        parts += [(np.eye(W) + rng.uniform(-1e-3, 1e-3, (W, W))).ravel(), np.zeros(W)]
    parts += [np.full(W, 4.0 / W), [-radius]]
    return np.concatenate(parts).astype(np.float32)


def _pair(net, blob):
    from paper_2606_00817_gb300 import ddf
    a, b = (ddf.DDF(*net, kind="sdf") for _ in range(2))
    for m in (a, b):
        m.load(blob)
    for which in (0, 1):
        ddf.ddf_set_tile(b.h, ddf.ddf_get_tile(b.h, which), which)
    return ddf, a, b


def _trace(ddf, m, rays, n, max_steps=128, eps=1e-3, t_max=4.0, want_steps=True):
    import torch
    t = torch.full((n,), -7.0, device="cuda")
    hit = torch.full((n,), 9, dtype=torch.uint8, device="cuda")
    steps = torch.full((n,), -7, dtype=torch.int32, device="cuda") if want_steps else None
    ddf.ddf_sphere_trace(m.h, rays, n, max_steps, eps, t_max, t, hit, steps,
                         torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert ddf.ddf_check_status(m.h) == 0
    return t, hit, steps


def _rays(torch, n, seed):
    return [torch.from_numpy(x).cuda() for x in I.uniform_rays(n, seed=seed).soa()]


@pytest.mark.parametrize("net", [(8, 128, 2), (0, 128, 4), (10, 256, 3), (16, 256, 2),
                                 (6, 384, 3), (8, 512, 6), (10, 512, 2)])
@pytest.mark.parametrize("n", [1, 127, 129, 1000, 25000])
def test_one_kernel_trace_equals_the_steps(cuda_lib, net, n):
    import torch
    ddf, a, b = _pair(net, _sphere_blob(net, seed=n))
    rays = _rays(torch, n, seed=n)
    x, y = _trace(ddf, a, rays, n), _trace(ddf, b, rays, n)
    for u, v in zip(x, y):
        assert torch.equal(u, v)
    if n >= 1000:
        assert 0.02 < float(x[1].float().mean()) < 0.98 and int(x[2].max()) > 5


@pytest.mark.parametrize("max_steps,eps,t_max", [(1, 1e-3, 4.0), (7, 1e-3, 4.0), (128, 0.3, 4.0),
                                                 (128, 1e-3, 0.0), (20, 1e-9, 1e6)])
def test_limits(cuda_lib, max_steps, eps, t_max):
    import torch
    net = (8, 256, 3)
    ddf, a, b = _pair(net, _sphere_blob(net, seed=2))
    n = 20000
    rays = _rays(torch, n, seed=9)
    x = _trace(ddf, a, rays, n, max_steps, eps, t_max)
    y = _trace(ddf, b, rays, n, max_steps, eps, t_max)
    for u, v in zip(x, y):
        assert torch.equal(u, v)
    z = _trace(ddf, a, rays, n, max_steps, eps, t_max, want_steps=False)
    assert torch.equal(x[0], z[0]) and torch.equal(x[1], z[1])


def test_rays_that_are_not_finite(cuda_lib):
    import torch
    net = (4, 512, 2)
    ddf, a, b = _pair(net, _sphere_blob(net, seed=3))
    n = 3000
    rays = _rays(torch, n, seed=10)
    rays[0][17], rays[4][999], rays[2][2999] = float("nan"), float("inf"), -float("inf")
    x, y = _trace(ddf, a, rays, n, 16), _trace(ddf, b, rays, n, 16)
    assert torch.equal(x[1], y[1]) and torch.equal(x[2], y[2])
    assert torch.equal(torch.nan_to_num(x[0], 123.0), torch.nan_to_num(y[0], 123.0))


def test_random_field_and_weights_loaded_again(cuda_lib):
    import torch
    net = (8, 512, 4)
    first, second = (I.xavier_blob_dims(I.sdf_layer_dims(*net), seed=s) for s in (1, 2))
    ddf, a, b = _pair(net, first)
    rays = _rays(torch, 5000, seed=11)
    for blob in (first, second):
        a.load(blob)
        b.load(blob)
        for u, v in zip(_trace(ddf, a, rays, 5000, 40), _trace(ddf, b, rays, 5000, 40)):
            assert torch.equal(u, v)


@pytest.mark.parametrize("net", [(4, 640, 2), (10, 1280, 3), (4, 2048, 2)])
@pytest.mark.parametrize("n", [1, 129, 2304, 2305, 3840, 3841, 9000])
def test_step_kernels_where_their_tiles_change(cuda_lib, net, n):
    """Wide fields: a trace of one step moves each ray by the field's value at
    its origin, as ddf_sdf_eval has it, or reports a hit (an output bias of 0: a
    trace adds it before the head's blocks, ddf_sdf_eval after them); with more
    steps a ray's trace does not depend on the batch, so on the tiles its steps
    take."""
    import torch
    rays = _rays(torch, n, seed=n)
    ddf, a, _ = _pair(net, _sphere_blob(net, seed=n, radius=0.0))
    s = torch.empty(n, device="cuda")
    ddf.ddf_sdf_eval(a.h, rays[:3], n, s, torch.cuda.current_stream())
    t, hit, steps = _trace(ddf, a, rays, n, 1, 0.5, 1e6)
    assert torch.equal(hit.bool(), s < 0.5) and bool((steps == 1).all())
    assert torch.equal(t, torch.where(s < 0.5, torch.zeros_like(s), s))
    ddf, a, _ = _pair(net, _sphere_blob(net, seed=n))
    x = _trace(ddf, a, rays, n)
    k = max(1, n // 3)
    y = _trace(ddf, a, [r[n - k:].clone() for r in rays], k)
    for u, v in zip(x, y):
        assert torch.equal(u[n - k:], v)
