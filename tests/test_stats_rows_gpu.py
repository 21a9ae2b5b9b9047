"""The statistic of unpermuted rows at the edges of its stages: rows that end inside a stage, fewer rows than stages or SMs, widths that
leave threads without a chunk, every block size that a warp sums, and blocks and permutations that the other kernel takes."""
import numpy as np
import pytest
import torch

from test_massdiff_device_gpu import B  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d,b", [(1, 32, 8), (5, 96, 32), (148, 2048, 16), (149, 4096, 32), (1187, 4096, 64), (300, 4128, 32), (1033, 8192, 128),
                                   (445, 9728, 256), (445, 9728, 512), (150, 16384, 8), (297, 20480, 16), (8, 32768, 32)])
@pytest.mark.parametrize("perm", [False, True])
def test_edges(B, T, d, b, perm):                            # noqa: F811
    gen = torch.Generator(device="cuda")
    gen.manual_seed(9300 + T + d)
    x = (torch.randn(T, d, generator=gen, device="cuda") * torch.exp2(torch.randint(-6, 7, (1, d), generator=gen, device="cuda").float())).to(torch.bfloat16)
    p = torch.randperm(d, generator=gen, device="cuda").to(torch.int32) if perm else None
    chan, block, token = B.perq_block_l1_stats(x, p, b)
    only = B.perq_block_l1_stats(x, p, b, want=("chan",))[0]
    again = B.perq_block_l1_stats(x, p, b)
    torch.cuda.synchronize()
    assert torch.equal(only, chan) and all(torch.equal(u, v) for u, v in zip(again, (chan, block, token)))
    a = x.abs().double().cpu().numpy()
    norms = (a if p is None else a[:, p.cpu().numpy()]).reshape(T, -1, b).sum(2)
    # sums of n terms in fp32, each rounding at most 2^-24 of the sum: (terms of a block or rows of a slab, slabs) * 2^-24
    eps = 2.0 ** -24
    rows = -(-T // 148)
    np.testing.assert_allclose(chan.cpu().numpy(), a.sum(0), rtol=(rows + 40) * eps)
    np.testing.assert_allclose(block.cpu().numpy(), norms.mean(0), rtol=(b + rows + 42) * eps)
    np.testing.assert_allclose(token.cpu().numpy(), norms.max(1), rtol=b * eps)
    assert B.perq_device_error() == 0


@pytest.mark.parametrize("T,d,b", [(149, 4096, 32), (300, 4128, 32), (1033, 8192, 128), (150, 16384, 8), (9, 32768, 64)])
def test_outputs_alone(B, T, d, b):                          # noqa: F811
    """An output that is asked for alone has the bits that it has among all."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(9400 + T + d)
    x = torch.randn(T, d, generator=gen, device="cuda").to(torch.bfloat16)
    for perm in (None, torch.randperm(d, generator=gen, device="cuda").to(torch.int32)):
        every = B.perq_block_l1_stats(x, perm, b)
        for i, want in enumerate(("chan", "block", "token")):
            alone = B.perq_block_l1_stats(x, perm, b, want=(want,))
            assert torch.equal(alone[i], every[i]) and all(alone[k] is None for k in range(3) if k != i)
