"""Compiles pieces of the device code for the host (simt.h) and runs them."""
import hashlib
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
CSRC = os.path.join(ROOT, "paper_2504_10096_gb300", "csrc")


def _cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


def cut(name, start, end):
    """The text of csrc/`name` from the first line that starts with `start` up to the next one that
    starts with `end`."""
    text = open(os.path.join(CSRC, name)).read()
    i = text.index("\n" + start) + 1
    j = text.index("\n" + end, i) + 1
    return text[i:j]


def run(tmp_path, source, *args):
    """The output lines of `source` (a main() that includes simt.h) as lists of floats."""
    key = hashlib.sha256(source.encode()).hexdigest()[:12]
    src, exe = tmp_path / f"{key}.cpp", tmp_path / key
    src.write_text(source)
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run([shutil.which("g++") or "g++", "-O1", "-std=c++17", "-ffp-contract=off", "-w", f"-I{here}",
                    f"-I{_cuda_include()}", str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe), *map(str, args)], check=True, capture_output=True, text=True, timeout=300).stdout
    return [[float(v) for v in line.split()] for line in out.splitlines()]
