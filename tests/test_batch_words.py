"""The words a prepared batch needs do not depend on what pm_tune does to its
sets afterwards (host code of the batch planner; no GPU)."""
import os
import subprocess

from paper_1407_2889_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_layouts_keep_the_prepared_words(tmp_path):
    lib = build.build()
    exe = tmp_path / "batch_words"
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC,
                    os.path.join(HERE, "batch_words.cpp"), lib, f"-Wl,-rpath,{os.path.dirname(lib)}", "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
