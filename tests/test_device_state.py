"""Sampling and selecting opt in to shared memory for the device of the
context, not once for the process: a context on another device (or in another
thread, before the first one's opt-in is through) asks for itself."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1506_03872_gb300", "csrc")


@pytest.mark.parametrize("source,kernels", [
    ("sample.cu", ("k_sort_scatter", "k_sort_fine", "k_build_x<true>", "k_build_x<false>")),
    ("select.cu", ("k_block_select",))])
def test_opt_ins_belong_to_the_context(source, kernels):
    text = open(os.path.join(CSRC, source)).read()
    for kernel in kernels:
        at = text.index(f"cudaFuncSetAttribute({kernel},")
        guard = re.findall(r"if \((?:build_x && )?!([\w>-]+)\) \{", text[:at])[-1]
        assert guard.startswith("ctx->"), (kernel, guard)
