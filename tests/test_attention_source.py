"""The order of the bf16 attention kernel's set-up, read from its source: a block
takes its tensor memory after it has waited for the kernel before it and before it
lets the next one start.  In any other order two kernels on one SM can each hold
what the other waits for; that is not a thing to try on a GPU."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_tensor_memory_between_wait_and_trigger():
    src = open(os.path.join(ROOT, "paper_2605_06892_gb300", "csrc", "hsa_attention.cu")).read()
    src = re.sub(r"//[^\n]*", "", src)
    body = src[src.index("attn_tc_kernel("):src.index("attn_combine_kernel(")]
    wait, trigger = (body.index(f"{f}();") for f in ("pdl_wait", "pdl_trigger"))
    assert wait < body.index("tcgen05.alloc") < trigger
    assert body.count("tcgen05.alloc") == body.count("pdl_trigger();") == 1
