"""adapm_push_noalloc at the sizes that its 16 MiB of scratch has to hold (the header's figures for a 152-SM GPU):
the push is accepted and its sums are exact (dyadic deltas), for each width of row whose chunks differ."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,n", [(64, 870_000), (200, 880_000), (300, 802_000), (300, 860_000), (384, 791_500),
                                 (512, 850_000), (1024, 780_000)])
def test_largest_pushes_are_accepted_and_exact(gpu_lib, D, n):
    K = 4096
    pm = gpu_lib.ParameterManager(K, D, 1)
    g = torch.Generator(device="cuda").manual_seed(D + n)
    keys = torch.randint(0, K, (n,), generator=g, device="cuda")
    keys[::5] = 17                                                     # a key whose rows run over many spans
    deltas = torch.randint(-64, 65, (n, D), generator=g, device="cuda", dtype=torch.int16).float().mul_(2.0 ** -10)
    pm.push_noalloc(0, keys, deltas)
    pm.wait()
    # whole multiples of 2^-10 below 2^14 in all: every order of summation is exact in 32 bits
    want = torch.zeros(K, D, device="cuda").index_add_(0, keys, deltas)
    assert torch.equal(torch.from_numpy(pm.read_main(torch.arange(K))).cuda(), want)
    pm.close()
