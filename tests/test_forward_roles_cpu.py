"""What the warps of the tensor-core forward kernel do when a wait runs out, on the CPU: the kernel's own text is compiled with
barriers, copies and products that are emulated by threads (fwd_ws_on_cpu.cpp), and every copy in turn comes too late."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2411_17178_b200 import build

CUDA_INCLUDE = os.path.join(os.path.dirname(os.path.dirname(shutil.which(build._nvcc()) or "/usr/local/cuda/bin/nvcc")), "include")


@pytest.fixture(scope="module")
def roles(tmp_path_factory):
    if not os.path.exists(os.path.join(CUDA_INCLUDE, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    where = tmp_path_factory.mktemp("roles")
    with open(os.path.join(build.CSRC, "litevar_fwd_ws.cu")) as f:
        s = f.read()
    kernel = "template <bool KV8, bool MANY>\n__global__"
    text = s[s.index("constexpr int kChunkKeys"):s.index("// Instruction descriptors")]
    text += s[s.index(kernel):s.index("template <bool KV8, bool MANY>\nlitevar_status_t launch_variant")]
    text, n = re.subn(r'asm volatile\("bar\.(sync|arrive) %0, (\d+);" ::"r"\((.*?)\) : "memory"\);', r"bar_\1(\3, \2);", text)
    assert n >= 7
    text = re.sub(r"asm(?: volatile)?\((?:.|\n)*?\);(?=[ \n])", ";", text)
    assert "asm" not in text
    for old, new in (("__global__ void __launch_bounds__(kThreads, 2)", "void"), ("__grid_constant__ ", ""),
                     ("extern __shared__ __align__(1024) uint8_t smem_raw[];", "uint8_t* smem_raw = cta->smem;")):
        assert old in text
        text = text.replace(old, new)
    (where / "fwd_ws_kernel.inc").write_text(text)
    program = str(where / "roles")
    res = subprocess.run(["g++", "-std=c++20", "-O1", "-w", "-pthread", "-I", str(where), "-I", build.CSRC,
                          "-I", os.path.join(build.ROOT, "include"), "-I", CUDA_INCLUDE,
                          os.path.join(os.path.dirname(__file__), "fwd_ws_on_cpu.cpp"), "-o", program], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[:4000]
    return program


@pytest.mark.parametrize("second_pass", [False, True], ids=["first-pass", "second-pass"])
@pytest.mark.parametrize("kind", ["one-tile", "many-tiles", "8-bit"])
def test_a_late_copy_ends_the_cta(roles, kind, second_pass):
    """Every warp returns, the status word is raised, and no copy or product is in flight."""
    res = subprocess.run([roles, kind] + ["second"] * second_pass, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stdout
