"""The tile lists of the Gaussian-depth renderer where their sorting takes
another way: more equal depths in one tile than a window holds, buckets too
crowded for one thread, a list of a single key, and an image of more tiles
than a binning block counts in shared memory. Compared with the oracle's
composite of every Gaussian at every pixel, with the bounds of
test_gpu_gs.py: 1e-4 relative, at most 0.5 % of the pixels beyond it (float32
decisions at a threshold)."""
import numpy as np
import pytest

from oracle import ddf_oracle as O

pytestmark = pytest.mark.gpu

CAM = np.array([0, 0, -3, 0, 0, 0, 0, 1, 0, np.radians(40.0)], np.float32)


def _gaussians(n, seed, depth, spread):
    """n faint round Gaussians at given depths, within `spread` of the axis."""
    rng = np.random.default_rng(seed)
    means = np.zeros((n, 3), np.float32)
    means[:, :2] = rng.uniform(-spread, spread, (n, 2))
    means[:, 2] = depth(rng, n)
    covs = np.zeros((n, 6), np.float32)
    covs[:, [0, 3, 5]] = rng.uniform(0.02, 0.05, (n, 1)) ** 2
    return means, covs, rng.uniform(0.01, 0.03, n).astype(np.float32)


@pytest.mark.parametrize("name,n,depth,spread,size", [
    ("one key", 1, lambda r, n: 0.0, 0.1, 16),
    ("a full window", 2048, lambda r, n: r.uniform(-0.5, 0.5, n), 0.1, 48),
    ("one more than a window", 2049, lambda r, n: r.uniform(-0.5, 0.5, n), 0.1, 48),
    ("equal depths", 3000, lambda r, n: 0.25, 0.1, 48),
    ("two equal depths", 3000, lambda r, n: np.where(np.arange(n) % 2, 0.25, 0.5), 0.1, 48),
    ("a crowd and a straggler", 3000, lambda r, n: np.where(
        np.arange(n) == 7, 1.9, 0.25 + r.uniform(0, 1e-4, n)), 0.1, 48),
    ("many tiles", 60, lambda r, n: r.uniform(-0.5, 0.5, n), 1.0, 1030),
])
def test_lists_match_the_oracle(cuda_lib, name, n, depth, spread, size):
    import torch
    from paper_2606_00817_gb300 import ddf
    m, c, o = _gaussians(n, 11, depth, spread)
    dev = [torch.from_numpy(a).cuda() for a in (m, c, o)]
    t = torch.empty(size * size, device="cuda")
    hit = torch.empty(size * size, dtype=torch.uint8, device="cuda")
    ddf.ddf_render_gs_depth(*dev, n, CAM, size, size, t, hit)
    torch.cuda.synchronize()
    pix = np.arange(size * size) if size < 100 else \
        np.random.default_rng(1).integers(0, size * size, 3000)
    rt, rh = O.gs_depth(m.astype(np.float64), O.gs_cov_matrices(c), o.astype(np.float64),
                        CAM[0:3], CAM[3:6], CAM[6:9], float(CAM[9]), size, size, pixels=pix)
    gt = t.cpu().numpy().astype(np.float64)[pix]
    bad = np.isfinite(gt) != np.isfinite(rt)
    both = np.isfinite(gt) & np.isfinite(rt)
    bad[both] |= np.abs(gt[both] - rt[both]) > 1e-4 * rt[both]
    assert bad.mean() <= 0.005, (name, bad.mean())
    assert (hit.cpu().numpy()[pix].astype(bool) != rh).mean() <= 0.005
