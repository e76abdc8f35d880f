"""Builds and asks tests/wide_layout_main.cpp: the host-side rules of the wide passes."""
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2001_09678_gb300")


def compile_rules(tmp_path):
    from paper_2001_09678_gb300 import build
    lib = build.build()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    exe = str(tmp_path / "wide_layout")
    cmd = ["g++", "-std=c++17", "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(ROOT, "include"),
           "-I", cuda, os.path.join(ROOT, "tests", "wide_layout_main.cpp"), lib,
           "-Wl,-rpath," + os.path.dirname(lib), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return exe


def ask(exe, lines):
    r = subprocess.run([exe], input="\n".join(lines) + "\n", capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return [tuple(int(x) for x in l.split()) for l in r.stdout.split("\n") if l]
