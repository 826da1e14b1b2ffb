"""Clusters of close eigenvalues on both sides of the line between one launch for all and a level each."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _matrix(J, sizes, width=1e-8):
    rng = np.random.default_rng(J + sum(sizes))
    q = np.linalg.qr(rng.standard_normal((J, J)))[0]
    lam = list(1 + 0.05 * np.arange(J - sum(sizes)))
    for c, n in enumerate(sizes):
        lam += list(40 + 3 * c + width * rng.random(n))
    a = (q * np.sort(lam)[::-1]) @ q.T
    return (a + a.T) / 2


@pytest.mark.parametrize("sizes", [(11,), (12,), (13,), (32,), (33,), (16, 16), (24, 20), (13, 13, 13, 13, 13), (32, 5, 12, 2),
                                   (20, 33, 2, 14)])
def test_eig_clusters(gpu_lib, monkeypatch, sizes):
    """The solver's own bounds, 16 J u lambda_1 and 16 J u, without the way back to the Jacobi."""
    monkeypatch.setenv("TUCKER_EIG_MP_STRICT", "1")
    J = sum(sizes) + 9
    a = _matrix(J, sizes)
    lam, v, _ = gpu_lib.eig(torch.from_numpy(a).cuda())
    lam, v = lam.cpu().numpy(), v.cpu().numpy()
    assert np.abs(a @ v - v * lam).max() <= 17 * J * U * lam[0]
    assert np.abs(v.T @ v - np.eye(J)).max() <= 17 * J * U
    assert np.abs(lam - np.linalg.eigvalsh(a)[::-1]).max() <= 17 * J * U * lam[0]


def test_cost_of_a_cluster(gpu_lib):
    """32 eigenvalues a float32 solve cannot tell apart cost a level of their own, another solve with its refinement, so
    less than twice the solve without them, and half as much again for the launches' jitter."""
    def cost(a):
        a, best = torch.from_numpy(a).cuda(), 1e9
        for _ in range(20):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            gpu_lib.eig(a)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best
    assert cost(_matrix(40, (32,))) <= 3 * cost(_matrix(40, ()))
