"""The Hessian's tiles that two launches share by their tokens: the same bits as the same columns of a smaller one, whose tiles are
whole (every entry is one chain of fused multiply-adds over the tokens in order, whatever the tile)."""

import pytest
import torch

from paper_2505_14638_b200 import binding

pytestmark = pytest.mark.gpu


# 24, 25, 32, 33 and 35 tiles a side: 300, 325, 528, 561 and 630 tiles on 296 places; tokens: too few to share, few in halves, more with a
# ragged last chunk, up to five tiles to a bundle; 4160: a last tile of 64 columns, which keeps all tiles whole
@pytest.mark.parametrize("K", [3072, 3200, 4096, 4160, 4224, 4480])
@pytest.mark.parametrize("T", [255, 300, 777, 1500])
def test_same_bits_as_whole_tiles(T, K):
    torch.manual_seed(K + T)
    batches = [torch.randn((T, K), device="cuda").bfloat16() for _ in range(2)]
    H = None
    for x in batches:
        H = binding.hessian_accumulate(x, H)
    assert torch.equal(H, H.T)
    torch.manual_seed(1)
    for _ in range(4):
        columns = torch.randperm(K, device="cuda")[:768].sort().values
        part = None
        for x in batches:
            part = binding.hessian_accumulate(x[:, columns].contiguous(), part)
        assert torch.equal(H[columns][:, columns], part)


def test_first_batch_of_rows_with_a_stride():
    torch.manual_seed(0)
    x = torch.randn((512, 4096 + 24), device="cuda").bfloat16()[:, 8:4104]
    H = binding.hessian_accumulate(x)
    assert torch.equal(H, binding.hessian_accumulate(x.contiguous()))
    assert torch.equal(H[1024:1792, 1024:1792], binding.hessian_accumulate(x[:, 1024:1792].contiguous()))
