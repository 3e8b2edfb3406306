"""Registers and shared memory of the kernels of single-graph calls, from the
compiler: each block fits an SM beside the serving executor's default blocks,
so that a call beside a busy server does not wait for the executor to leave.
"""
import re
import shutil
import subprocess

import pytest

from paper_2507_03695_gb300 import build

REGISTERS, SHARED, PER_BLOCK = 65536, 228 << 10, 1 << 10
EXECUTOR_BLOCKS = 3
# kernel: (threads, largest dynamic shared memory)
LISTED = {
    "k_select_begin": (256, 0), "k_degree_sampled": (256, 0), "k_degree_certify": (512, 32 << 10),
    "k_select_candidates": (512, 0), "k_argmax_u32": (256, 0), "k_degree": (256, 0), "k_wide_hot_pack": (256, 0),
    "k_init": (256, 0), "k_tiny": (1024, 4 * (48 << 10)), "k_bits_link": (256, 0), "k_bits_build": (256, 0),
    "k_bits_filter": (640, (1504 << 10) // 8 + 20 * 2 * 64 * 4), "k_insert_small": (512, 64 << 10), "k_validate": (256, 0),
    "k_gmin_probe": (256, 0), "k_flatten4": (256, 0), "k_flatten": (256, 0), "k_connected": (256, 0),
    "k_count_roots": (256, 0), "k_csr_maxlen": (256, 0), "k_csr_tile_rows": (256, 0), "k_edge_pass_csr": (256, 0),
}


SOURCES = ("cc_bits.cu", "cc_csr.cu", "cc_kernels.cu", "cc_rootsel.cu", "cc_server.cu", "cc_tiny.cu")


@pytest.mark.skipif(not (shutil.which("nvcc") and shutil.which("c++filt")), reason="no compiler")
def test_blocks_fit_beside_the_executor(tmp_path):
    jobs = [subprocess.Popen(["nvcc", *build.NVCC_FLAGS, "-Xptxas", "-v", "-c", src, "-o", str(tmp_path / f"{i}.o")],
                             stderr=subprocess.PIPE, text=True)
            for i, src in enumerate(build.sources()) if src.endswith(SOURCES)]
    text = "".join(p.communicate()[1] for p in jobs)
    found = re.findall(r"Compiling entry function '(\S+)'(?:.*\n)*?.*?Used (\d+) registers(.*)", text)
    names = subprocess.run(["c++filt"], input="\n".join(f[0] for f in found), capture_output=True, text=True).stdout
    used = {}
    for name, (_, regs, rest) in zip(names.splitlines(), found):
        kernel = re.search(r"\b(k_\w+)[<(]", name).group(1)
        smem = re.search(r"(\d+) bytes smem", rest)
        used.setdefault(kernel, []).append((-(-int(regs) // 8) * 8, int(smem.group(1)) if smem else 0))
    regs, smem = max(used["k_executor"])
    left_regs = (REGISTERS - EXECUTOR_BLOCKS * 256 * regs) // 4  # of each quarter, which takes a quarter of the warps
    left_smem = SHARED - EXECUTOR_BLOCKS * (-(-smem // 128) * 128 + PER_BLOCK)
    for kernel, (threads, dynamic) in LISTED.items():
        for r, s in used[kernel]:
            assert -(-threads // 128) * 32 * r <= left_regs, (kernel, r, threads)
            assert s + dynamic + PER_BLOCK <= left_smem, (kernel, s, dynamic)
