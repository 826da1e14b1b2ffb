"""Device memory of an eigensolve: a level's block is taken when a cluster goes down to it."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

J = 512
MB = 1 << 20


def _grown(gpu_lib, call):
    torch.cuda.synchronize()
    gpu_lib.memory_trim()
    before = gpu_lib.memory_stats()["pool_reserved"]
    out = call()
    grown = gpu_lib.memory_stats()["pool_reserved"] - before
    print(f"pool grew by {grown / MB:.0f} MB")
    return out, grown


@pytest.mark.parametrize("kind", ["low_rank", "clusters", "graded", "flat"])
def test_eig_memory(gpu_lib, kind):
    """Five levels of 9 J^2 doubles would be 90 MB: the pool (which grows by blocks of 32 MB) stays within that where few
    levels are needed, and within eight such levels anywhere."""
    rng = np.random.default_rng(7)
    q = np.linalg.qr(rng.standard_normal((J, J)))[0]
    lam = np.sort(rng.random(J))[::-1] + 0.5
    if kind == "low_rank":
        lam[100:] *= 1e-9
    elif kind == "clusters":  # levels below levels, of different widths at different depths
        lam = np.concatenate([4 + 1e-7 * rng.random(200), 3 + 1e-9 * rng.random(70), 2 + 1e-7 * rng.random(160),
                              1 + 1e-11 * rng.random(82)])
        lam = np.sort(lam)[::-1]
    elif kind == "graded":
        lam = 10.0 ** (-12 * np.arange(J) / J)
    a = (q * lam) @ q.T
    a = torch.from_numpy((a + a.T) / 2).cuda()
    (l, v, _), grown = _grown(gpu_lib, lambda: gpu_lib.eig(a))
    assert grown <= (96 if kind in ("graded", "flat") else 160) * MB
    l, v, an = l.cpu().numpy(), v.cpu().numpy(), a.cpu().numpy()
    assert np.abs(an @ v - v * l).max() <= 17 * J * 2.0 ** -53 * l[0]


def test_sthosvd_memory(gpu_lib):
    """A 512-long mode of low rank plus noise, the tail discarded: within five levels' worth with all else of the call."""
    from synthetic import tucker_tensor_np

    x = torch.from_numpy(tucker_tensor_np((J, 20, 20), (30, 8, 8), seed=1, noise=1e-4)).cuda()
    res, grown = _grown(gpu_lib, lambda: gpu_lib.sthosvd(x, (J, 20, 20), 1e-3))
    assert res.ranks[0] == 30 and grown <= 96 * MB
