"""The MLP kernels' parameter copy has no wait that can give up: kt_mlp_forward and
kt_mlp_train_step without a loss return before their kernels run and read no error word, so a
launch that left its outputs unwritten would go unnoticed (csrc/kt_mlp.cu).  Source only."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_04941_gb300", "csrc")


def test_no_wait_with_a_limit_before_the_outputs_are_written():
    with open(os.path.join(CSRC, "kt_mlp.cu")) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    for name in ("stage_table", "mbar_try_wait", "bulk_g2s"):
        assert name not in code, name
    for kernel in ("train_tile", "infer"):
        body = code[code.index(f" {kernel}("):]
        body = body[body.index("{"):body.index("\n}\n")]
        assert "return;" not in body, kernel
