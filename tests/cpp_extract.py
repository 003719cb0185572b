"""Functions of the CUDA sources compiled for the host.

``function(file, head)`` returns the text of the function whose definition
starts with ``head``; ``run(code)`` compiles a program around such text with
g++ and runs it.  For host logic whose failures no call can bring about (a
failing creation, the order of copies) and for device code whose faults must
not be tried on a GPU: the CUDA names it uses are stand-ins of the program."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_03920_gb300", "csrc")


def function(fn: str, head: str) -> str:
    text = open(os.path.join(CSRC, fn)).read()
    at = text.index(head)
    depth, i = 0, text.index("{", at)
    while True:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
        if depth == 0:
            return text[at:i]


def run(tmp_path, code: str) -> str:
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(code)
    r = subprocess.run([cxx, "-std=c++20", "-O1", "-pthread", "-o", str(exe), str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
