"""The traced library's kernels run as the ordinary ones do: its stamps must not
cost a bandwidth kernel a block per SM, or the timeline times another kernel.
Read from what the compiler prints (no GPU)."""

from __future__ import annotations

import os
import re
import subprocess

from paper_2604_05718_gb300 import build

THREADS = {"prep_kernel": 256, "prep_split_kernel": 256, "pair_average_kernel": 256, "merge_tail_kernel": 256,
           "gather_kernel": 256, "mutual_compact_kernel": 1024}
REGISTERS, SM_THREADS = 65536, 2048


def registers(out, flags):
    src = os.path.join(build.CSRC, "kernels_hbm.cu")
    return subprocess.Popen([build.nvcc(), "-c", src, "-o", str(out), "-Xptxas", "-v"] + build.NVCC_FLAGS + flags,
                            stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)


def blocks_per_sm(proc):
    text = proc.communicate()[0]
    assert proc.returncode == 0, text[-2000:]
    found = {}
    for name, body in re.findall(r"Compiling entry function '(\S+)'(.*?Used \d+ registers)", text, re.S):
        kernel = next((k for k in THREADS if re.search(r"\d" + k, name)), None)
        if kernel is None:
            continue
        instance = re.search(kernel + r"(I(?:L[ib]\d+E)+E)?", name).group(0)
        used = int(re.search(r"Used (\d+) registers", body).group(1))
        threads = THREADS[kernel]
        found[instance] = min(REGISTERS // (-(-used // 8) * 8 * threads), SM_THREADS // threads)
    return found


def test_traced_kernels_keep_their_blocks_per_sm(tmp_path):
    plain = registers(tmp_path / "plain.o", [])
    traced = registers(tmp_path / "traced.o", ["-DMPM_TRACE"])
    plain, traced = blocks_per_sm(plain), blocks_per_sm(traced)
    assert len(plain) >= 15
    assert plain == traced
