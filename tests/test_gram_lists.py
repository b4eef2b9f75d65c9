"""Lists of the gram tables stay short for small alphabets (host code; no GPU)."""
import os
import subprocess

from paper_1407_2889_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_buckets_hold_their_grams(tmp_path):
    lib = build.build()
    exe = tmp_path / "gram_lists"
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC,
                    os.path.join(HERE, "gram_lists.cpp"), lib, f"-Wl,-rpath,{os.path.dirname(lib)}", "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
