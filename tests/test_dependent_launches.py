"""The surrogate's kernels start before the kernel in front of them has ended (programmatic dependent
launches) and wait in pass_begin().  A `const T* __restrict__` parameter lets the compiler move its
loads across that wait or take them through the read-only path, so only inputs that no kernel of a pass
writes may carry it.  Read from the source: a wait that runs out cannot be provoked on a GPU."""
import os
import re

SOURCE = os.path.join(os.path.dirname(__file__), "..", "paper_1605_03607_gb300", "csrc", "sg.cu")

# uploaded before a pass: parameters and their packed copies, topology tables, couplers, targets
CONSTANT = {"Wm", "bm", "Wu", "bu", "W", "bias", "WmT", "WuT", "WeT", "W1", "b1", "w2", "b2",
            "in_tab", "out_tab", "msg_tab", "ends", "inter", "J", "target"}


def test_only_constant_inputs_may_be_read_across_the_wait():
    text = open(SOURCE).read()
    kernels = {}
    for k in re.finditer(r"__global__[^;{]*?(\w+_kernel)\((.*?)\)\s*\{(.*?)\n\}", text, flags=re.S):
        if "pass_begin()" in k.group(3):
            kernels[k.group(1)] = re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", k.group(2))
    assert set(kernels) == {"node_fwd_kernel", "edge_fwd_kernel", "node_bwd_kernel", "edge_bwd_kernel",
                            "readout_kernel", "reduce_kernel"}
    for name, restricted in kernels.items():
        assert set(restricted) <= CONSTANT, (name, set(restricted) - CONSTANT)
