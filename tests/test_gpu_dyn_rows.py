"""The one-pass dynamic quantizer of rows of several 2048-element blocks (a warp per block) against the two calls it stands for, bit for
bit: the smallest and largest number of blocks, more rows than the chip takes at once, the first number that keeps the two passes."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,blocks,row_begin,ld_pad", [(1, 2, 0, 0), (5, 3, 1, 2), (1300, 2, 0, 0), (33, 14, 4, 0), (7, 16, 0, 6), (300, 9, 0, 0), (3, 17, 0, 0)])
def test_rows_of_several_blocks_equal_the_two_calls(M, blocks, row_begin, ld_pad):
    from paper_2410_05265_b200 import binding

    ctx = binding.Context()
    K = 2048 * blocks
    g = torch.Generator().manual_seed(M * 31 + blocks)
    x = (torch.randn((M, K + ld_pad), generator=g) * torch.exp2(torch.randint(-20, 20, (M, 1), generator=g).float())).to(torch.bfloat16).cuda()[:, :K]
    x[M - 1, : K - 2048] = 0  # the maximum sits in the last block
    s_two, s_one = torch.full((M,), -5.0, device="cuda"), torch.full((M,), -5.0, device="cuda")
    q_two, q_one = (torch.full((M, K // 2), 0x5A, dtype=torch.uint8, device="cuda") for _ in range(2))
    ctx.dyn_act_scale(x, 2048, 0.9, row_begin, out=s_two)
    ctx.hadamard_quant_act_rows(x, 2048, s_two, row_begin, out=q_two)
    ctx.dyn_hadamard_quant_act(x, 2048, 0.9, row_begin, s_tok=s_one, out=q_one)
    ctx.check()
    assert torch.equal(s_one, s_two) and torch.equal(q_one, q_two)
    ctx.close()
