"""Autotuning a field at a size for which it has kernels of its own as long as no
tile is set: the tuned handle is not slower than the untouched one, and where those
kernels win it is left as it was, for batches of every size."""
import numpy as np
import pytest

from paper_2606_00817_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _us(torch, call):
    """Device time of a call among others, the median of 9 rounds of 8."""
    for _ in range(5):
        call()
    times = []
    for _ in range(9):
        a, b = torch.cuda.Event(True), torch.cuda.Event(True)
        call()
        a.record()
        for _ in range(8):
            call()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) / 8e-3)
    return sorted(times)[4]


# 1280 wide, a few hundred rays take about half of what any tile does
@pytest.mark.parametrize("precision", ["bf16", "fp8"])
def test_small_batches_keep_their_kernels(cuda_lib, precision):
    import torch
    from paper_2606_00817_gb300 import ddf
    net, n = (10, 1280, 8), 193
    a, b = (ddf.DDF(*net, precision=precision) for _ in range(2))
    for m in (a, b):
        m.load(I.xavier_blob(I.NetShape(*net)),
               np.full(7, 2.0 ** -6, np.float32) if precision == "fp8" else None)
    rays = [torch.from_numpy(x).cuda() for x in I.uniform_rays(30000, seed=4).soa()]
    few = [r[:n].contiguous() for r in rays]
    ddf.ddf_autotune(a.h, few, n)
    assert _us(torch, lambda: a.query(few)) <= 1.3 * _us(torch, lambda: b.query(few))
    assert ddf.ddf_get_tile(a.h, 0) == ddf.ddf_get_tile(b.h, 0)
    for k in (1, n, 4099, 30000):
        part = [r[:k].contiguous() for r in rays]
        for x, y in zip(a.query(part), b.query(part)):
            assert torch.equal(x, y), k
    assert ddf.ddf_check_status(a.h) == 0


@pytest.mark.parametrize("net,n", [((8, 384, 3), 5000), ((6, 128, 4), 3000), ((8, 512, 3), 70000)])
def test_any_choice_gives_the_results(cuda_lib, net, n):
    """Fields without a pair tile, narrow ones, and a batch beyond the sizes that
    have kernels of their own: the results are those of the untouched field up to
    the FP32 rounding of the head sums, at the tuned size and at others."""
    import torch
    from paper_2606_00817_gb300 import ddf
    a, b = ddf.DDF(*net), ddf.DDF(*net)
    for m in (a, b):
        m.load(I.xavier_blob(I.NetShape(*net)))
    rays = [torch.from_numpy(x).cuda() for x in I.uniform_rays(n, seed=5).soa()]
    for _ in range(2):                   # tuned twice: from either state
        ddf.ddf_autotune(a.h, rays, n)
        for k in (1, 300, n):
            part = [r[:k].contiguous() for r in rays]
            for x, y in zip(a.query(part), b.query(part)):
                assert float((x - y).abs().max()) <= 1e-5
    assert ddf.ddf_check_status(a.h) == 0
