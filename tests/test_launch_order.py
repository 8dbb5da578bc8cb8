"""Kernels that write what another kernel reads ahead of its wait for its predecessor (KV-cache rows, lengths and steps; packed
weights, their scales and code sums) must not let their successors start early: the rotation kernels and the small GEMMs trigger ahead of
their own wait, so an early start can be passed on over any number of launches. Read from the sources; the order on the
device is tested in test_gpu_launch_order.py."""
import os
import re

import pytest

import paper_2410_05265_b200

CSRC = os.path.join(os.path.dirname(paper_2410_05265_b200.__file__), "csrc")
TRIGGER = re.compile(r"launch_dependents|pdl_trigger")


def block_from(text, start):
    """The text from the first brace at or after start to the brace that closes it."""
    i = text.index("{", start)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i: j + 1]
    raise ValueError("unbalanced braces")


def kernel_body(source, name):
    with open(os.path.join(CSRC, source)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    found = [m for m in re.finditer(r"__global__[^;{]*?\b%s\s*\(" % name, text)]
    assert len(found) == 1, f"{name} in {source}"
    return block_from(text, found[0].end())


@pytest.mark.parametrize("source,name", [
    ("pq_kv4.cu", "kv4_append_kernel"), ("pq_kv4_dyn.cu", "kv4_append_dyn_kernel"), ("pq_block.cu", "rope_kv4_append_kernel"),
    ("pq_block.cu", "calib_kv_scale_kernel"), ("pq_quant_weights.cu", "quant_weights_kernel"), ("pq_quant_weights.cu", "quant_weights_once_kernel"),
    ("pq_quant_weights.cu", "weight_code_sums_kernel"),
])
def test_writers_of_early_read_data_never_trigger(source, name):
    assert not TRIGGER.search(kernel_body(source, name))


def test_the_one_launch_decode_step_never_triggers():
    body = kernel_body("pq_kv4.cu", "decode_attn_kernel")
    plain_only = block_from(body, body.index("if (!FUSED) {"))
    assert TRIGGER.search(plain_only)
    assert not TRIGGER.search(body.replace(plain_only, "")), "a trigger outside the branch of the plain call"


@pytest.mark.parametrize("source,name", [
    ("pq_gemm_stream.cu", "gemm_w4a4_stream_kernel"), ("pq_gemm_split.cu", "gemm_w4_split_kernel"), ("pq_gemm_tc2.cu", "gemm_w4a4_pair_kernel"),
    ("pq_gemm_tc3.cu", "gemm_w4a4_pair_ts_kernel"), ("pq_hadamard_quant.cu", "hadamard_quant_kernel"),
    ("pq_hadamard_quant.cu", "hadamard_quant_wide_kernel"), ("pq_hadamard_quant.cu", "hadamard_quant_small_kernel"),
    ("pq_quant_weights.cu", "quant_weights_once_kernel"), ("pq_kv4.cu", "decode_attn_kernel"), ("pq_prefill_attn.cu", "prefill_attn_kernel"),
    ("pq_block.cu", "rmsnorm_kernel"), ("pq_block.cu", "rope_kernel"), ("pq_block.cu", "rope_rotate_kernel"), ("pq_block.cu", "silu_mul_kernel"),
    ("pq_block.cu", "add_kernel"), ("pq_block.cu", "rope_kv4_append_kernel"),
])
def test_what_a_predecessor_may_write_is_not_read_through_the_read_only_path(source, name):
    """The compiler may move a read-only load (__ldg, or one through a const __restrict__ pointer) ahead of the wait for the predecessor.
    Only data that no early-triggering kernel writes may be read so: weights with their scales and sums, the cache with its steps and
    prefix, norm weights."""
    body = kernel_body(source, name)
    if name == "gemm_w4_split_kernel":
        with open(os.path.join(CSRC, source)) as f:
            text = f.read()
        body += block_from(text, text.index("void reduce_tile("))
    static = re.compile(r"s_w|wsum|gsrc|\bgr\b|s_k|s_v|p\.len|prefix_|\bkr\b|skb|svb")
    if name == "decode_attn_kernel":  # one helper, which reads so in the one-launch step only
        static = re.compile(r"^ptr$")
    read_only = re.findall(r"__ldg\(((?:[^()]|\([^()]*\))*)\)", body) + re.findall(r'"ld\.global\.nc[^"]*"[^;]*"l"\((\w+)\)', body)
    wrong = [a for a in read_only if not static.search(a)]
    assert not wrong, wrong
    if name.startswith("hadamard"):  # its parameters are const __restrict__: no plain load through them either
        assert not re.search(r"\b(?:x|x2|s_a_in|zp_in)\[", body)
    if name.startswith("quant_weights"):
        assert body.count("row + j") == 1 and not re.search(r"\b(?:W|row)\[|\*row|\*W\b", body) and body.index("pdl_wait") < body.index("row + j")


def test_the_plain_decode_attention_reads_nothing_through_the_read_only_path():
    """The header promises that it waits before it reads anything: a read-only load may be moved ahead of the wait. The one-launch step may."""
    body = kernel_body("pq_kv4.cu", "decode_attn_kernel")
    assert re.findall(r"(FUSED \? )?__ldg\(", body) == ["FUSED ? "]
    for step in ("skb", "svb"):  # (the one-launch step has no steps per vector)
        assert len(re.findall(r"%s \+" % step, body)) == len(re.findall(r"ld_dep\(%s \+" % step, body)) == 1
    assert "FUSED ? __ldcg(p.len + b) : pq::ld_dep(p.len + b)" in body


@pytest.mark.parametrize("source,name", [("pq_gemm_tc2.cu", "gemm_w4a4_pair_kernel"), ("pq_gemm_tc3.cu", "gemm_w4a4_pair_ts_kernel")])
def test_the_kernels_for_any_number_of_tokens_request_nothing_ahead_of_their_wait(source, name):
    """The header asks of a writer of weights that it does not let its successors start early for calls of few rows only."""
    body = kernel_body(source, name)
    assert body.index("griddepcontrol.wait") < body.index("tma_load_2d")
