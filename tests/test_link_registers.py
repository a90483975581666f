"""The forms of k_link that read the union-find options at run time have the
registers they need: ptxas reports no spill for them (at the register limit of
the default form they do spill, and their link phase takes 3% longer)."""
import os
import re
import subprocess

from paper_2003_11468_gb300 import build


def test_variant_forms_do_not_spill(tmp_path):
    cmd = [build.nvcc(), *build.NVCC_FLAGS, *build.ARCH, "-Xptxas", "-v", "-c",
           os.path.join(build.CSRC, "fof_link.cu"), "-o", str(tmp_path / "link.o")]
    out = subprocess.run(cmd, check=True, capture_output=True, text=True).stderr
    forms = re.findall(r"Compiling entry function '\S*k_linkILb([01])ELb([01])E\S*'.*?(\d+) bytes spill stores", out, re.S)
    assert len(forms) == 4
    for var, split, spilled in forms:
        if var == "1":
            assert int(spilled) == 0, (split, spilled)
