"""The Grams whose MMAs are issued by two threads in turn (float64 digits, and split precision for J <= 32): every
addition to the accumulators arrives, run after run, at odd and even numbers of chunks per CTA and per drain."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("J", [8, 16, 31, 64, 120])
@pytest.mark.parametrize("K", [152 * 512 * 9 + 33, 152 * 4096 - 7])
def test_every_addition_arrives(gpu_lib, J, K, split):
    """Integers below 2^14: the sums stay below 2^28 x 700416 < 2^48, so float64 products of any order are exact and
    so are the digits' and (hi, lo) sums; twenty runs give the same bits."""
    gen = torch.Generator(device="cuda").manual_seed(J + K)
    y = torch.randint(-(1 << 14) + 1, 1 << 14, (K, J), generator=gen, device="cuda").double()
    exact = y.t() @ y
    run = gpu_lib.gram_split if split else gpu_lib.gram
    y = y.reshape(-1)
    first = run(y, 1, J, K)
    assert torch.equal(first, exact)
    for _ in range(20):
        assert torch.equal(run(y, 1, J, K), first)
