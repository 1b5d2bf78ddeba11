"""Every kernel may be launched as a programmatic dependent and run beside the kernel that writes
its inputs.  The read-only loads of the compiler's intrinsics need not stay behind the
grid-dependency wait, so no kernel uses them; those that are spelled out stay there."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_28699_gb300", "csrc")


def test_no_read_only_load_can_pass_the_wait():
    for f in sorted(os.listdir(CSRC)):
        code = "\n".join(line.split("//")[0] for line in open(os.path.join(CSRC, f)))
        assert "__ldg" not in code, f
        for m in re.finditer(r"asm(?P<volatile> volatile)?\s*\((?P<body>[^;]*ld\.global\.nc.*?)\);\n", code, re.S):
            assert m["volatile"] and '"memory"' in m["body"], f
        assert code.count("ld.global.nc") == (2 if f == "write_kernel.cu" else 0), f


def test_the_wait_holds_memory_back():
    code = open(os.path.join(CSRC, "wc_common.cuh")).read()
    assert re.search(r'asm volatile\("griddepcontrol\.wait;"\s*::: "memory"\)', code)
