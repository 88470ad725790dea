"""What a kernel of a programmatic chain must keep to, read in the sources.

Kernels that may be resident while the one before still writes (those that
call grid_wait) read what the chain writes by plain loads: ld.global.nc, which
__ldg and a const __restrict__ parameter stand for, promises memory that nobody
writes during the kernel's whole life.  A thread that returns before grid_wait
lets its kernel end before the one ahead of it has, and the one behind start on
unfinished data.  No run shows a breach of either reliably."""
import glob
import os
import re

from helpers import ROOT

SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_2608_10139_gb300", "csrc", "*.cu*")))

# weights, gains, biases and RoPE tables: written when a model is loaded or a table is made
READ_ONLY = re.compile(r"xh_gain|rope_cos|rope_sin|\bg4\b|\bc4\b|\bs4\b|load_f32x32")


def _code(path):
    src = re.sub(r"//[^\n]*", "", open(path).read())
    return re.sub(r"/\*.*?\*/", "", src, flags=re.S)


def test_no_restrict_parameters_in_chained_kernels():
    for path in SOURCES:
        for head, body in re.findall(r"__global__(.*?)\{(.*?)\n\}", _code(path), flags=re.S):
            if "grid_wait()" in body:
                assert "__restrict__" not in head, f"{os.path.basename(path)}: {head.strip()[:120]}"


def test_read_only_loads_take_constant_data():
    for path in SOURCES:
        src = _code(path)
        assert "global.nc" not in src, path
        for m in re.finditer(r"__ldg\(([^;]*);", src):
            func = src[:m.start()].rfind("load_f32x32(const float* src")
            inside = func >= 0 and "\n}" not in src[func:m.start()]   # its callers are checked below
            assert inside or READ_ONLY.search(m.group(1)), f"{os.path.basename(path)}: __ldg({m.group(1)}"
        for arg in re.findall(r"\bload_f32x32\(([^)]*)\)", src):
            assert arg.startswith(("const float* src", "ep.bias", "ep.rope_cos", "ep.rope_sin")), arg


def test_no_thread_leaves_before_the_wait():
    for path in SOURCES:
        for head, body in re.findall(r"__global__(.*?)\{(.*?)\n\}", _code(path), flags=re.S):
            if "grid_wait()" in body:
                before = body[:body.index("grid_wait()")]
                assert not re.search(r"\breturn\b(?! ?\w)", before), f"{os.path.basename(path)}: {head.strip()[:120]}"
