"""The weight quantizer that reads a row once against the two-pass kernel (which unaligned rows take) and the oracle: edges of
its vector counts, rows with exact ties, infinities, NaN, zeros and steps far from one."""
import numpy as np
import pytest
import torch

from oracle import pq_oracle as orc
from paper_2410_05265_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2410_05265_b200 import binding

    c = binding.Context()
    yield c
    c.close()


def two_pass(ctx, W):
    """The same rows starting two bytes off a vector boundary."""
    N, K = W.shape
    buf = torch.zeros((N, K + 9), dtype=torch.bfloat16, device="cuda")
    buf[:, 1: K + 1] = W
    return ctx.quant_weights(buf[:, 1: K + 1])


@pytest.mark.parametrize("N,K", [(3, 8), (5, 1000), (7, 4096), (4, 4104), (3, 8192), (2, 8200), (3, 16384), (2, 16392), (2, 32768), (2, 32776)])
def test_one_pass_equals_oracle_and_two_pass(ctx, N, K):
    g = torch.Generator().manual_seed(N * 7 + K)
    W = (torch.randn((N, K), generator=g) * 0.02).to(torch.bfloat16)
    W[0] = (torch.randint(-14, 15, (K,), generator=g) * 0.5).to(torch.bfloat16)  # maximum 7: step 1, every odd half is a tie
    W[0, K // 2] = 7.0
    wq, s_w = ctx.quant_weights(W.cuda())
    wq2, s_w2 = two_pass(ctx, W.cuda())
    ref, s_ref = orc.quant_weights(inputs.bits(W))
    assert np.array_equal(wq.cpu().numpy(), ref) and np.array_equal(s_w.cpu().numpy(), s_ref)
    assert torch.equal(wq, wq2) and torch.equal(s_w, s_w2)


def test_special_rows_keep_the_two_pass_result(ctx):
    K = 4096
    g = torch.Generator().manual_seed(1)
    rows = [torch.zeros(K)]
    base = torch.randn(K, generator=g)
    for scale in (1e-38, 1e-40, 1e-30, 7e-30, 1e30, 1e37):
        rows.append(base * scale)
    for special in (float("inf"), float("-inf"), float("nan")):
        r = base.clone()
        r[17] = special
        rows.append(r)
    both = base.clone()
    both[3], both[4000] = float("nan"), float("inf")
    rows += [both, torch.full((K,), float("nan"))]
    for m in range(128):  # every mantissa of the maximum
        r = (torch.randint(-128, 129, (K,), generator=g).float() / 128) * (1 + m / 128)
        r[0] = 1 + m / 128
        rows.append(r)
    W = torch.stack(rows).to(torch.bfloat16).cuda()
    wq, s_w = ctx.quant_weights(W)
    wq2, s_w2 = two_pass(ctx, W)
    assert torch.equal(wq, wq2)
    assert torch.equal(s_w.view(torch.int32), s_w2.view(torch.int32))
