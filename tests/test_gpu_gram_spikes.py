"""The float64 Gram from exact digits on rows of one large entry over a visible background, alone and beside
multiples of themselves, where the squares of low digits add up."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("L,J,B", [(1, 12, 152 << 14), (1, 20, 152 << 14), (1, 40, 152 << 14), (1, 100, 50 << 14),
                                   (8, 32, 19 << 14), (24, 64, (152 << 14) // 24)])
def test_gram_of_spikes(gpu_lib, L, J, B):
    """About 2^14 columns a CTA.  Per entry, over u |y_i| |y_j|: roundings, of standard deviation at most 2^-57 / sqrt(3)
    (2^E_i |y_j| + 2^E_j |y_i|) <= 0.15 as 2^E <= 2 |y|; levels 11 and above, six digit products of standard deviation
    1365 2^35 / 2^112 2^(E_i + E_j) a column, twice as correlated on the diagonal, <= 0.5 at these K; six deviations of
    both; and the CTAs' sums, 19 in a thread, three steps of the tree, one rounding each: 24."""
    gen = torch.Generator(device="cuda").manual_seed(J)
    K = L * B
    m = torch.randn(J, K, generator=gen, device="cuda", dtype=torch.float64)
    m[0] *= 1e-3
    m[0, 777] = 1.0
    m[1] = m[0]
    m[2] = 3.0 * m[0]
    m[J - 1] = -m[0]
    m[J - 2] = 1e-4 * m[J - 2]
    m[J - 2, K // 3] = -0.75
    y = m.reshape(J, B, L).permute(1, 0, 2).contiguous()
    s = gpu_lib.gram(y.reshape(-1), L, J, B).cpu().numpy()
    norms = torch.linalg.vector_norm(m, dim=1).cpu().numpy()
    worst = 0.0
    rows = {i: m[i].cpu().numpy().astype(np.longdouble) for i in (0, 1, 2, 5, J - 2, J - 1)}
    for i, j in [(0, 0), (0, 1), (1, 1), (0, 2), (2, 2), (0, 5), (5, 5), (0, J - 1), (0, J - 2), (J - 2, J - 2), (J - 1, J - 1)]:
        worst = max(worst, abs(float(s[i, j] - (rows[i] * rows[j]).sum())) / (U * norms[i] * norms[j]))
    print(f"L={L} J={J} B={B}: error / (u |y_i| |y_j|) {worst:.2f}")
    assert worst <= 24 + 6 * (0.15 + 0.5)
