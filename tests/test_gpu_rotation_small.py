"""Rotation kernel of calls with few wide blocks (16 elements to a thread, a block to a CTA): the codes, steps and normalised rows of the kernel for
many blocks bit for bit, at the borders of the rule between the two (7/16 of a block of 4096 to an SM, four in all with a step per token, two of 2048 to an SM,
five with SwiGLU), for every form."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2410_05265_b200 import binding

    c = binding.Context()
    yield c
    c.check()
    c.close()


def rows(M, width, pitch=0, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = (torch.randn((M, width + pitch), generator=g, device="cuda") * torch.exp(0.5 * torch.randn(width + pitch, generator=g, device="cuda"))).to(torch.bfloat16)
    return x[:, :width]


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("form", ["static", "bytes", "nibbles_in_bytes", "zero_point", "rows", "dynamic"])
@pytest.mark.parametrize("K,block,per_sm", [(4096, 4096, 7 / 16), (4096, 4096, 1), (2048, 2048, 2), (14336, 2048, 2), (8192, 4096, 7 / 16), (8192, 4096, 1)])
@pytest.mark.parametrize("where", ["one", "last", "beyond"])
@pytest.mark.parametrize("pitch,row_begin", [(0, 0), (34, 3)])
def test_same_codes_as_the_kernel_for_many_blocks(ctx, form, K, block, per_sm, where, pitch, row_begin):
    if form == "dynamic" and K != block:
        pytest.skip("rows of several blocks have a kernel of their own")
    per_row = K // block
    most = 4 if block == 4096 and form in ("rows", "dynamic") else int(per_sm * sms())
    M = row_begin + {"one": 1, "last": most // per_row, "beyond": most // per_row + 1}[where]
    x = rows(row_begin + int(per_sm * sms()) // per_row + 40, K, pitch)  # enough rows for the other kernel
    s, z = torch.full((1,), 0.37, device="cuda"), torch.full((1,), 6, dtype=torch.int32, device="cuda")
    s_tok = torch.rand(x.shape[0], device="cuda") + 0.1

    def call(a):
        if form == "static":
            return (ctx.hadamard_quant_act(a, block, s, row_begin),)
        if form == "bytes":
            return (ctx.hadamard_quant_act8(a, block, s / 16, row_begin),)
        if form == "nibbles_in_bytes":
            return (ctx.hadamard_quant_act_c8(a, block, s, row_begin),)
        if form == "zero_point":
            return (ctx.hadamard_quant_act_asym(a, block, s, z, row_begin),)
        if form == "rows":
            return (ctx.hadamard_quant_act_rows(a, block, s_tok[: a.shape[0]], row_begin),)
        return ctx.dyn_hadamard_quant_act(a, block, 0.9, row_begin)

    few, many = call(x[:M]), call(x)
    ctx.check()
    for a, b in zip(few, many):
        assert torch.equal(a, b[:M])
    assert len(torch.unique(few[-1][row_begin:])) > 12  # (not the zeros it was filled with)


@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("F,block,per_sm", [(14336, 2048, 5), (8192, 4096, 1), (8192, 8192, 1)])
def test_swiglu_same_codes_as_the_two_launches(ctx, F, block, per_sm, extra):
    M = per_sm * sms() // (F // block) + extra
    gu = rows(M, 2 * F)
    s = torch.full((1,), 0.2, device="cuda")
    fused = ctx.swiglu_hadamard_quant_act(gu[:, :F], gu[:, F:], block, s)
    two = ctx.hadamard_quant_act(ctx.silu_mul(gu[:, :F], gu[:, F:]), block, s)
    ctx.check()
    assert torch.equal(fused, two) and len(torch.unique(fused)) > 12


@pytest.mark.parametrize("K,per_sm", [(4096, 7 / 16), (4096, 1), (2048, 2)])
@pytest.mark.parametrize("extra", [0, 1])
def test_rmsnorm_fused_and_alone_agree_on_both_sides_of_the_rule(ctx, K, per_sm, extra):
    M = int(per_sm * sms()) + extra
    x, g = rows(M, K), rows(1, K, seed=1)[0].contiguous()
    s = torch.full((1,), 0.5, device="cuda")
    h = ctx.rmsnorm(x, g, 1e-5)
    fused = ctx.rmsnorm_hadamard_quant_act(x, g, 1e-5, s)
    ctx.check()
    assert torch.equal(fused, ctx.hadamard_quant_act(h, K, s))
    xd = x.double()
    want = xd / torch.sqrt((xd * xd).mean(1, keepdim=True) + 1e-5) * g.double()
    # one bf16 rounding of a value that fp32 sums of K squares give within K/512 * 2^-24: half an ulp and a little
    assert bool(((h.double() - want).abs() <= want.abs() * (2.0**-8 + 2.0**-16) + 1e-30).all())


@pytest.mark.parametrize("K,per_sm", [(4096, 7 / 16), (4096, 1), (2048, 2)])
@pytest.mark.parametrize("row_begin", [0, 4])
def test_a_normalised_row_does_not_depend_on_the_rows_beside_it(ctx, K, per_sm, row_begin):
    """Few rows, as many as the kernel of few blocks takes, and two more: the same values, and the fused call the codes of the two
    calls also where row_begin leaves it on one side of the rule and the stand-alone call, which has none, on the other."""
    most = int(per_sm * sms())
    g = rows(1, K, seed=1)[0].contiguous()
    s = torch.full((1,), 0.5, device="cuda")
    for seed in range(8):  # two orders of the sum differ in some five of a million bf16 values
        x = rows(most + 2, K, seed=seed)
        many = ctx.rmsnorm(x, g, 1e-5)
        for M in (3, most):
            assert torch.equal(ctx.rmsnorm(x[:M], g, 1e-5), many[:M])
        fused, two = ctx.rmsnorm_hadamard_quant_act(x, g, 1e-5, s, row_begin), ctx.hadamard_quant_act(many, K, s, row_begin)
        assert torch.equal(fused[row_begin:], two[row_begin:])
    ctx.check()
