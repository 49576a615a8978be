"""Two fields of the same kernels and different sizes, each used by a host thread
of its own on a stream of its own: no call fails, and the results are those of
one thread alone."""
import threading

import numpy as np
import pytest

from paper_2606_00817_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LIGHT = (3.0, 3.0, 3.0)


def _field(net, precision, kind="ray"):
    from paper_2606_00817_gb300 import ddf
    m = ddf.DDF(*net, precision=precision, kind=kind)
    if kind == "hashgrid":
        dims = [(64, ddf.HASHGRID_CODE)] + [(64, 64)] * (net[2] - 1) + [(2, 64)]
        m.load(I.hashgrid_blob(m.n_params, dims, seed=1))
    elif kind == "sdf":
        m.load(I.xavier_blob_dims(I.sdf_layer_dims(*net)))
    else:
        m.load(I.xavier_blob(I.NetShape(*net)))
    return ddf, m


# one-kernel queries with small and large shared memory; heads of small batches of
# narrow and wide fields; FP32 encodings; hash grids of one and four layers; traces
@pytest.mark.parametrize("a,b,n", [
    (((0, 128, 2), "bf16"), ((10, 128, 6), "bf16"), 2000),
    (((4, 512, 2), "bf16"), ((10, 1280, 2), "bf16"), 100),
    (((0, 512, 2), "fp32"), ((16, 512, 2), "fp32"), 100),
    (((4, 64, 1), "bf16", "hashgrid"), ((4, 64, 4), "bf16", "hashgrid"), 5000),
    (((4, 64, 1), "fp32", "hashgrid"), ((4, 64, 4), "fp32", "hashgrid"), 5000),
    (((0, 256, 2), "bf16", "sdf"), ((8, 256, 6), "bf16", "sdf"), 300)])
def test_two_threads(cuda_lib, a, b, n):
    import torch
    rays = [torch.from_numpy(x).cuda() for x in I.uniform_rays(n, seed=3).soa()]
    torch.cuda.synchronize()

    def call(ddf, m, sdf, stream):
        if not sdf:
            return m.shadow(rays, LIGHT, stream)
        t = torch.empty(n, device="cuda")
        hit = torch.empty(n, dtype=torch.uint8, device="cuda")
        ddf.ddf_sphere_trace(m.h, rays, n, 4, 1e-3, 4.0, t, hit, None, stream)
        return t, hit

    fields = [(*_field(*x), len(x) > 2 and x[2] == "sdf") for x in (a, b)]
    streams = [torch.cuda.Stream() for _ in fields]
    want = []
    for f, s in zip(fields, streams):
        with torch.cuda.stream(s):
            want.append([x.cpu().numpy() for x in call(*f, s)])
    errors, start = [], threading.Barrier(2)

    def run(k):
        try:
            start.wait()
            with torch.cuda.stream(streams[k]):
                for _ in range(300):
                    got = call(*fields[k], streams[k])
                streams[k].synchronize()
                for x, y in zip(got, want[k]):
                    assert np.array_equal(x.cpu().numpy(), y)
        except Exception as e:      # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=run, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for ddf, m, _ in fields:
        assert ddf.ddf_check_status(m.h) == 0
