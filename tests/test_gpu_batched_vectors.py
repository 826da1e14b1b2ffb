"""Eigenvectors of the batched pipeline on spectra that its leading-eigenpair stage converges on slowly: geometric,
without a gap at the rank cut."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("eps", [1e-3, 5e-4, 1e-4])
@pytest.mark.parametrize("J", [20, 33, 64, 128])
def test_batched_vectors(gpu_lib, J, eps):
    """Mode-1 eigenvalues g^k, a tensor for each of 36 g, against the vectors it was made from (themselves off by a few
    u sqrt(J) in the tensor's rounding): the residual is at most 4 sqrt(J) u lambda_1 per entry, so a vector is off by at
    most 4 J u lambda_1 / gap."""
    rng = np.random.default_rng(J)
    q = np.linalg.qr(rng.standard_normal((J, J)))[0]
    w = np.linalg.qr(rng.standard_normal((320, J)))[0]
    lams = [np.maximum(g ** np.arange(J), 1e-13) for g in np.linspace(0.1, 0.45, 36)]
    xs = [torch.from_numpy(((q * np.sqrt(lam)) @ w.T).reshape(-1, order="F").copy()).cuda() for lam in lams]
    worst = 0.0
    for lam, r in zip(lams, gpu_lib.sthosvd_batched(xs, [(J, 40, 8)] * len(xs), eps)):
        u = r.factor(0).cpu().numpy()
        for c in range(min(u.shape[1], J - 1)):
            gap = min(lam[c - 1] - lam[c] if c else np.inf, lam[c] - lam[c + 1])
            err = min(np.linalg.norm(u[:, c] - q[:, c]), np.linalg.norm(u[:, c] + q[:, c]))
            worst = max(worst, err * gap / (U * lam[0]))
    print(f"J={J} eps={eps}: vector error * gap / (J u lambda_1) {worst / J:.2f}")
    assert worst <= 5 * J
