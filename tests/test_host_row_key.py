"""The row keys of the local extension in defined arithmetic (host build with the
undefined-behaviour sanitizer; no GPU needed)."""
import os
import subprocess

import pytest

from paper_2403_06478_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))


def test_row_key_is_exact_and_defined(tmp_path):
    exe = str(tmp_path / "row_key_check")
    cmd = [B._nvcc()] + B.ARCH + ["-std=c++17", "-O1", "-Xcompiler", "-fsanitize=undefined",
                                  "-Xcompiler", "-fno-sanitize-recover=all", "-I" + B.INCLUDE, "-I" + B.CSRC,
                                  os.path.join(HERE, "host", "row_key_check.cu"), "-o", exe, "-lubsan"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        pytest.fail(f"nvcc failed:\n{res.stdout}\n{res.stderr}")
    run = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert run.returncode == 0, run.stdout + run.stderr
    assert " 0 wrong" in run.stdout and "runtime error" not in run.stderr
