"""Spectra without gaps, whose neighbours lie closer than the norms of the float32 stage's error."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("kind", ["equal", "pairs", "gram", "random"])
@pytest.mark.parametrize("J", [33, 48, 66, 128, 200, 300, 321, 360, 400, 450, 512])
def test_eig_dense(gpu_lib, monkeypatch, J, kind):
    """The solver's own bounds, 16 J u lambda_1 and 16 J u, without the way back to the Jacobi."""
    monkeypatch.setenv("TUCKER_EIG_MP_STRICT", "1")
    rng = np.random.default_rng(J)
    q = np.linalg.qr(rng.standard_normal((J, J)))[0]
    if kind == "gram":
        m = rng.standard_normal((J, 4 * J))
        a = m @ m.T
    else:
        lam = {"equal": 1.0 + np.arange(J), "random": rng.standard_normal(J),
               "pairs": 1 + np.repeat(np.arange((J + 1) // 2), 2)[:J] + 1e-9 * rng.random(J)}[kind]
        a = (q * lam) @ q.T
    a = (a + a.T) / 2
    lam, v, _ = gpu_lib.eig(torch.from_numpy(a).cuda())
    lam, v = lam.cpu().numpy(), v.cpu().numpy()
    top = np.abs(lam).max()
    assert np.abs(a @ v - v * lam).max() <= 17 * J * U * top
    assert np.abs(v.T @ v - np.eye(J)).max() <= 17 * J * U
    assert np.abs(lam - np.linalg.eigvalsh(a)[::-1]).max() <= 17 * J * U * top
