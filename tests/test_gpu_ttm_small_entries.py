"""The float64 mode product where a column's small entries count: tucker_ttm with matrices that select, permute or
scale, and the products with orthonormal factors, which may take digits on the tensor cores."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("kind", ["identity", "permutation", "selection", "scaling", "sparse"])
@pytest.mark.parametrize("L,J,B,dt", [(1, 48, 5000, "f8"), (7, 48, 300, "f8"), (1, 128, 2000, "f8"), (64, 300, 9, "f8"),
                                      (1, 33, 60000, "f8"), (1, 100, 700, "f4")])
def test_ttm_small_entries(gpu_lib, L, J, B, dt, kind):
    """Columns graded over 20 orders (variables in units of their own), sizes on both sides of the digits' line: the
    error of every output is at most that of a chain of multiply-adds, (J + 1) u sum_j |m_kj y_jc|."""
    rng = np.random.default_rng([L, J, B])
    y = (rng.standard_normal((B, J, L)) * 10.0 ** rng.uniform(-15, 5, (1, J, 1))).astype(dt)
    m = np.eye(J)
    if kind == "permutation":
        m = m[rng.permutation(J)]
    elif kind == "selection":
        m = m[rng.permutation(J)[:20]]
    elif kind == "scaling":
        m = np.diag(10.0 ** rng.uniform(-8, 8, J))
    elif kind == "sparse":
        m = np.where(rng.random((24, J)) < 0.05, rng.standard_normal((24, J)), 0.0)
    z = gpu_lib.ttm(torch.from_numpy(y.reshape(-1).copy()).cuda(), L, J, B, torch.from_numpy(m.copy()).cuda())
    z = z.cpu().numpy().reshape(B, m.shape[0], L)
    ref = np.einsum("kj,bjl->bkl", m, y.astype(np.float64))
    mag = np.einsum("kj,bjl->bkl", np.abs(m), np.abs(y.astype(np.float64)))
    assert (np.abs(z - ref) <= 2 * (J + 1) * U * mag).all()  # the reference's own chains: as much again


@pytest.mark.parametrize("dims,ranks,dt", [((64, 40, 9), (20, 12, 5), "f8"), ((9, 50, 100), (4, 17, 33), "f8"),
                                           ((130, 49), (16, 16), "f8"), ((300, 70), (33, 33), "f8"), ((5, 512, 24), (3, 40, 16), "f8"),
                                           ((65, 48, 11), (31, 20, 6), "f4"), ((33, 97, 10), (12, 40, 8), "f4")])
def test_products_with_factors(gpu_lib, dims, ranks, dt):
    """Core and reconstruction against longdouble products with the factors as they came back.  Per output, with
    |m_r| = 1: roundings <= 2.2 2^-57 2 sqrt(J) |y_c|, dropped levels <= J 2^-55 4 |y_c|, together <= 1.3 J u |y_c|, and
    sqrt(K) times that over K outputs; the same for each mode, one after the other."""
    from synthetic import tucker_tensor_np

    x = tucker_tensor_np(dims, ranks, seed=3, noise=1e-5).astype(dt)
    res = gpu_lib.sthosvd(torch.from_numpy(x).cuda(), dims, 1e-3)
    assert res.ranks == tuple(ranks) or list(res.ranks) == list(ranks)
    us = [res.factor(n).cpu().numpy().astype(np.longdouble) for n in range(len(dims))]
    core = x.astype(np.longdouble).reshape(dims, order="F")
    for n, u in enumerate(us):
        core = np.moveaxis(np.tensordot(u.T, core, (1, n)), 0, n)
    got = res.core().cpu().numpy().reshape(ranks, order="F")
    bound = 1.3 * U * float(np.linalg.norm(x.astype(np.float64))) * sum(np.sqrt(r) * d for d, r in zip(dims, ranks))
    assert float(np.sqrt(((got - core) ** 2).sum())) <= bound
    back = got.astype(np.longdouble)
    for n, u in enumerate(us):
        back = np.moveaxis(np.tensordot(u, back, (1, n)), 0, n)
    y = gpu_lib.reconstruct(res).cpu().numpy().reshape(dims, order="F")
    bound = 1.3 * U * float(np.linalg.norm(got)) * sum(np.sqrt(d) * r for d, r in zip(dims, ranks))
    assert float(np.sqrt(((y - back) ** 2).sum())) <= bound


@pytest.mark.parametrize("C", [32, 127, 300])
@pytest.mark.parametrize("J,K", [(64, 33), (128, 128), (300, 200), (512, 512)])
def test_ttm_few_columns(gpu_lib, J, K, C):
    """Few columns, the rows of the small sums spread over CTAs: dense, graded and sparse rows of one matrix, each output
    within the chain's bound of test_ttm_small_entries."""
    rng = np.random.default_rng([J, K, C])
    y = rng.standard_normal((C, J)) * 10.0 ** rng.uniform(-12, 4, J)
    m = rng.standard_normal((K, J))
    m[1::3] *= 10.0 ** rng.uniform(-8, 8, J)
    m[2::3] *= rng.random((len(m[2::3]), J)) < 0.1
    z = gpu_lib.ttm(torch.from_numpy(y.reshape(-1).copy()).cuda(), 1, J, C, torch.from_numpy(m).cuda()).cpu().numpy()
    ref, mag = y @ m.T, np.abs(y) @ np.abs(m).T
    assert (np.abs(z.reshape(C, K) - ref) <= 2 * (J + 1) * U * mag).all()
