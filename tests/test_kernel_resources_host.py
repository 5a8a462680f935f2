"""What the compiler says about kernels whose speed hangs on it: no spills, no stack."""
import os
import re
import subprocess

import pytest

from paper_2308_15030_b200 import build

NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def ptxas_properties(source, tmp_path):
    """{mangled kernel name: (stack frame, spill stores, spill loads) in bytes} of `source`, compiled with the library's flags."""
    cu = tmp_path / "kernels.cu"
    cu.write_text(source)
    cmd = [NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xptxas", "-v", "-I", build.CSRC,
           "-cubin", "-o", str(tmp_path / "kernels.cubin"), str(cu)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    props = re.findall(r"Function properties for (\S+)\s+(\d+) bytes stack frame, (\d+) bytes spill stores, (\d+) bytes spill loads",
                       r.stdout + r.stderr)
    return {name: tuple(int(v) for v in rest) for name, *rest in props}


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_permutation_kernel_does_not_spill(tmp_path):
    """Every CTA that copies rows holds four token pieces per thread in registers from before the dependent-launch wait to its
    stores; code of the one CTA that publishes the slot layout must not push them to the stack."""
    forms = ["%s, %s" % (t, top1) for t in ("float", "bf16") for top1 in ("true", "false")]
    source = '#include "permute.cuh"\nnamespace swapmoe {\n' + "".join(
        "template __global__ void permute_gather_kernel<%s>(PermuteArgs);\n" % f for f in forms) + "}\n"
    props = {n: v for n, v in ptxas_properties(source, tmp_path).items() if "permute_gather_kernel" in n}
    assert len(props) == len(forms)
    assert all(v == (0, 0, 0) for v in props.values()), props
