"""What the compiler says about kernels whose speed hangs on it (no spills, no stack), and which tiles the host code picks."""
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


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_gated_small_batches_cover_the_tile_widths(tmp_path):
    """The shapes that the parity tests run get the tile widths and stages noted beside them (on 148 SMs)."""
    from test_gpu_parity import GATED_SMALL_BATCHES
    cu = tmp_path / "widths.cu"
    cu.write_text('''
#include <cstdio>
#include "../../include/swapmoe.h"
#include "common.cuh"
#include "gemm_tc_small.cuh"
using namespace swapmoe;
int main() {
  int T, d, f, K, k;
  while (std::scanf("%d %d %d %d %d", &T, &d, &f, &K, &k) == 5) {
    const int pairs = T * k;
    int a_rows = 16;
    while (a_rows < pairs) a_rows <<= 1;
    TcSmallGeom g;
    if (!tc_small_geometry(2 * f, d / kTcBK, pairs < K ? pairs : K, 148, a_rows * kTcBK * 2, &g)) return 1;
    std::printf("%d %d %d\\n", g.bn, g.kps, g.n_stages);
  }
}
''')
    exe = str(tmp_path / "widths")
    r = subprocess.run([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", build.CSRC, "-o", exe, str(cu)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe], input="\n".join(" ".join(map(str, g[0])) for g in GATED_SMALL_BATCHES), capture_output=True, text=True)
    got = [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    assert [g[:2] for g in got] == [g[1:] for g in GATED_SMALL_BATCHES]
    for (T, d, f, K, k), (bn, kps, stages) in zip((g[0] for g in GATED_SMALL_BATCHES), got):
        blocks = d // 64
        assert -(-blocks // kps) > stages                       # the ring wraps
        assert kps == 1 or blocks % kps != 0                    # the last stage is part empty
        assert bn == 128 or 2 * f % bn != 0                     # the last tile is ragged
    assert {g[1] for g in GATED_SMALL_BATCHES} == {96, 128, 160, 192, 224, 256}
