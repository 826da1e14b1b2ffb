"""The eigenvalues of a discarded tail: a cluster that the rank rule cuts off whole and that is wide enough for the
precision of its values to show."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _tail(gpu_lib, J, wide):
    """A matrix with 8 eigenvalues in [1, 2] and the others, 1e-6 lambda apart, summing to just below the threshold."""
    rng = np.random.default_rng(J)
    lam = np.concatenate([np.linspace(2, 1, 8), wide * np.linspace(2, 1, J - 8)])
    q = np.linalg.qr(rng.standard_normal((J, J)))[0]
    w = np.linalg.qr(rng.standard_normal((2 * J, J)))[0]
    m = (q * np.sqrt(lam)) @ w.T
    eps = np.sqrt(2 * 1.05 * lam[8:].sum() / lam.sum())
    res = gpu_lib.sthosvd(torch.from_numpy(m.reshape(-1, order="F").copy()).cuda(), (J, 2 * J), eps)
    assert res.ranks[0] == 8
    return lam, np.array(res.eigvals[0])


@pytest.mark.parametrize("wide", [1e-4, 1e-6])
@pytest.mark.parametrize("J", [64, 100, 200, 400])
def test_tail_sum(gpu_lib, J, wide):
    """The tail's values sum to its trace: float64 rounding of the Gram and the products, J u lambda_1 twice over."""
    lam, got = _tail(gpu_lib, J, wide)
    print(f"J={J} wide={wide}: sum off by {abs(got[8:].sum() - lam[8:].sum()) / (J * U * lam[0]):.2f} J u lambda_1")
    assert abs(got[8:].sum() - lam[8:].sum()) <= 4 * J * U * lam[0]


@pytest.mark.parametrize("wide", [1e-4, 1e-5, 1e-6, 1e-7, 1e-9])
@pytest.mark.parametrize("J", [64, 100, 200, 400])
def test_tail_values_one_by_one(gpu_lib, J, wide):
    """Every value within J u lambda_1 of its own, the rounding of a float64 solve (and as much for the tensor's), whether
    float32 stage, Rayleigh quotients or a level of its own gave it."""
    lam, got = _tail(gpu_lib, J, wide)
    print(f"J={J} wide={wide}: values off by {np.abs(got - lam).max() / (J * U * lam[0]):.2f} J u lambda_1")
    assert np.abs(got - lam).max() <= 2 * J * U * lam[0]
