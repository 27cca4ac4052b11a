"""Register shares of warpgroups: what a kernel's warpgroups take together is no more than a block is launched with.  More would
wait for registers that nobody gives back.  Read from the compiler's report, no GPU."""
import os
import re
import subprocess

import pytest

from paper_2507_18181_b200 import build


@pytest.mark.parametrize("variant", [[], ["-DSPECASR_TRACE"]])
def test_shares_add_up_to_what_the_block_is_launched_with(tmp_path, variant):
    source = os.path.join(build.HERE, "csrc", "gemm_fill.cu")
    text = open(source).read()
    roles, epilogue = map(int, re.search(r"ROLE_REGS = (\d+), EPI_REGS = (\d+);", text).groups())
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    res = subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-Xptxas", "-v", *variant,
                          "-I", os.path.join(build.ROOT, "include"), "-c", source, "-o", str(tmp_path / "fill.o")],
                         capture_output=True, text=True, check=True)
    used = re.findall(r"Compiling entry function '\w*k_proj_fill\w*ILi(\d)ELi\d\w*'.*?Used (\d+) registers", res.stderr, re.S)
    with_shares = [int(n) for mode, n in used if mode == "2"]       # mode 2: four warps of roles, eight of the epilogue
    assert with_shares and all(4 * roles + 8 * epilogue <= 12 * n for n in with_shares), res.stderr
