"""Batches with values outside the digits' range: what they cost and what the other tensors see of them."""
import time

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _seconds(f):
    best = 1e9
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        f()
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
    return best


@pytest.mark.parametrize("dims", [(20, 18, 16), (16, 16, 16), (70, 33, 9)])
def test_batched_tiny_values_cost(gpu_lib, dims):
    """Finite values below 2^-850 leave the digits for plain sums: at these sizes the work of an ordinary batch, so
    a few times its time and not the length of an expired wait (2^22 polls of 10 ns or more for each item)."""
    rng = np.random.default_rng(3)
    xs = [torch.from_numpy(rng.standard_normal(int(np.prod(dims)))).cuda() for _ in range(8)]
    tiny = [x * 2.0 ** -880 for x in xs]
    usual = _seconds(lambda: gpu_lib.sthosvd_batched(xs, [dims] * 8, 1e-3))
    assert _seconds(lambda: gpu_lib.sthosvd_batched(tiny, [dims] * 8, 1e-3)) <= 5 * usual + 0.01


@pytest.mark.parametrize("dims", [(40, 7, 110, 10), (100, 60, 64), (12, 128, 70)])
def test_batched_mixed_range(gpu_lib, dims):
    """A tensor whose slices span 2^-1000 .. 1: summed plainly, in whole and ragged stages, its first mode's
    eigenvalues are within 4 J u lambda_1 of LAPACK's on the same unfolding."""
    rng = np.random.default_rng(4)
    x = rng.standard_normal(dims)
    x[3] *= 2.0 ** -1000
    res = gpu_lib.sthosvd_batched([torch.from_numpy(x.reshape(-1, order="F").copy()).cuda()], [dims], 0.0)[0]
    m = x.reshape(dims[0], -1, order="F")
    lam = np.linalg.eigvalsh(m @ m.T)[::-1]
    assert np.abs(np.array(res.eigvals[0]) - lam).max() <= 4 * dims[0] * 2.0 ** -53 * lam[0]


@pytest.mark.parametrize("count", [1, 40])
def test_batched_tail_values(gpu_lib, count):
    """Past the rank cut each eigenvalue is its own: within 2^-18 of the tail's largest (float32's 2^-22, a few times)
    and the solves' 1e-12 lambda_1 of the oracle's, in order."""
    import oracle
    from synthetic import tucker_tensor_np

    shapes = [((128, 40, 9), (5, 4, 3)), ((33, 64, 65), (16, 8, 8)), ((31, 17, 100), (8, 8, 8)), ((24, 3, 70), (4, 2, 6)),
              ((70, 60, 50), (30, 30, 30))]
    xs, dims = [], []
    for i in range(count):
        d, r = shapes[i % len(shapes)]
        xs.append(tucker_tensor_np(d, r, seed=3, tensor=i, noise=3e-4, decay=0.15 * (max(r) == 30)))
        dims.append(d)
    res = gpu_lib.sthosvd_batched([torch.from_numpy(x).cuda() for x in xs], dims, 1e-2)
    for i in range(min(count, len(shapes))):
        ref = oracle.sthosvd(xs[i], dims[i], 1e-2)
        assert res[i].ranks == ref["ranks"]
        for n, J in enumerate(dims[i]):
            lam, got, k = np.array(ref["eigvals"][n]), np.array(res[i].eigvals[n]), res[i].ranks[n]
            if k < J:
                assert np.abs(got - lam).max() <= 2.0 ** -18 * lam[k] + 1e-12 * lam[0]
                assert (np.diff(got) <= 1e-12 * lam[0]).all()


@pytest.mark.parametrize("dims", [(20, 18, 16), (70, 40, 30)])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_batched_non_finite_tensor(gpu_lib, bad, dims):
    """The call succeeds; the tensor's own norm is not finite, and the others come out as without it, bit for bit."""
    rng = np.random.default_rng(2)
    xs = [rng.standard_normal(int(np.prod(dims))) for _ in range(3)]
    ok = gpu_lib.sthosvd_batched([torch.from_numpy(x).cuda() for x in xs], [dims] * 3, 1e-3)
    xs[1][777] = bad
    res = gpu_lib.sthosvd_batched([torch.from_numpy(x).cuda() for x in xs], [dims] * 3, 1e-3)
    assert not np.isfinite(res[1].norm2)
    for i in (0, 2):
        assert res[i].ranks == ok[i].ranks and torch.equal(res[i].core(), ok[i].core())
        for n in range(3):
            assert torch.equal(res[i].factor(n), ok[i].factor(n))
            assert np.array_equal(res[i].eigvals[n], ok[i].eigvals[n])
