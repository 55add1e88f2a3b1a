"""Set-up calls whose allocations fail half-way leave no pointer to freed
memory behind, and their copies are waited for before another stream uses
them: the host side compiled against a stand-in for the CUDA runtime."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2001_11252_gb300", "csrc")


def test_failed_and_reordered_set_up(tmp_path):
    from paper_2001_11252_gb300.build import cuda_home
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "setup_check")
    inc = [os.path.join(cuda_home(), "include"), CSRC, os.path.join(ROOT, "include")]
    subprocess.check_call([cxx, "-O1", "-g", "-std=c++17", "-ffp-contract=off", *["-I" + i for i in inc],
                           os.path.join(HERE, "native", "setup_check.cpp"), os.path.join(CSRC, "host.cpp"), "-o", exe])
    r = subprocess.run([exe], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, timeout=120)
    out = r.stdout.decode()
    assert r.returncode == 0 and out.strip() == "ok", out
