"""What runs with the device memory of the faster paths also runs without it (TUCKER_FAULT=scratch refuses it on the
host), on the plain kernels; and a captured mode product holds kernels only."""
import numpy as np
import pytest
import torch

import oracle
from synthetic import tucker_tensor_np

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("precision", ["fp64", "bf16x4"])
def test_without_optional_scratch(gpu_lib, monkeypatch, precision):
    dims, ranks = (100, 64, 50), (12, 9, 8)
    xh = tucker_tensor_np(dims, ranks, seed=4, noise=1e-4)
    x = torch.from_numpy(xh).cuda()
    rng = np.random.default_rng(1)
    m = rng.standard_normal((64, 9))
    usual = gpu_lib.sthosvd(x, dims, 1e-3, precision=precision)
    monkeypatch.setenv("TUCKER_FAULT", "scratch")
    res = gpu_lib.sthosvd(x, dims, 1e-3, precision=precision)
    s = gpu_lib.gram(x, 100, 64, 50).cpu().numpy()
    z = gpu_lib.ttm(x, 100, 64, 50, torch.from_numpy(m).cuda(), transpose=True).cpu().numpy()
    back = gpu_lib.reconstruct(res).cpu().numpy()
    monkeypatch.delenv("TUCKER_FAULT")
    y = xh.reshape(50, 64, 100)
    assert res.ranks == usual.ranks == oracle.sthosvd(xh, dims, 1e-3)["ranks"]
    for n in range(3):
        a, b = np.array(res.eigvals[n]), np.array(usual.eigvals[n])
        assert np.abs(a - b).max() <= 16 * dims[n] * U * b[0]  # the solver's own bound
    assert np.linalg.norm(back - xh) <= 1.01e-3 * np.linalg.norm(xh)
    ref, mag = np.einsum("bjl,bil->ji", y, y), np.einsum("bjl,bil->ji", np.abs(y), np.abs(y))
    assert (np.abs(s - ref) <= 2 * 5000 * U * mag).all()
    ref, mag = np.einsum("jk,bjl->bkl", m, y), np.einsum("jk,bjl->bkl", np.abs(m), np.abs(y))
    assert (np.abs(z.reshape(ref.shape) - ref) <= 2 * 65 * U * mag).all()


def test_captured_mode_product(gpu_lib):
    """A graph captured before its input is known, replayed twice on different inputs."""
    J, C, K = 64, 5000, 20
    gen = torch.Generator(device="cuda").manual_seed(5)
    y, m = (torch.randn(n, generator=gen, device="cuda", dtype=torch.float64) for n in (J * C, K * J))
    m = m.view(K, J)
    gpu_lib.ttm(y, 1, J, C, m)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        z = gpu_lib.ttm(y, 1, J, C, m)
    for _ in range(2):
        y.copy_(torch.randn(J * C, generator=gen, device="cuda", dtype=torch.float64))
        graph.replay()
        ref = (y.view(C, J) @ m.t()).reshape(-1)
        assert (z - ref).abs().max() <= 2 * J * U * float((y.view(C, J).abs() @ m.abs().t()).max())
