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
