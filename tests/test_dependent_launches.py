"""Kernels launched while the launch before them may still be ending read its results coherently.

A kernel launched by launch_dependent() begins before the launch before it on the stream is
over, and what that one wrote is not constant over the kernel's run. So it has to wait
(cudaGridDependencySynchronize) and must not read through the read-only path (__ldg, const
__restrict__), whose loads may be moved above the wait. Checked on the source: a stale read is a
matter of timing.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1409_5474_gb300", "csrc")


def _text(path):
    text = open(path).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    text = re.sub(r"//[^\n]*", "", text)
    return re.sub(r"__launch_bounds__\([^\n]*\)\n", "", text)


def _functions(text):
    """Functions at namespace scope: name -> signature and body."""
    return {m.group(1): m.group(0) for m in
            re.finditer(r"\b(\w+)\([^;{}()]*\)\n\{.*?\n\}", text, flags=re.S)}


def _dependent_kernels(text):
    """Names of the kernels that a file's launch_dependent() calls launch."""
    names = set()
    for m in re.finditer(r"\blaunch_dependent\(((?:<[^;>]*>|[^,;<])*),", text):
        arg = m.group(1)
        if arg.strip() == "kern":
            arg = text[:m.start()].rsplit(" kern =", 1)[1].split(";", 1)[0]
        names |= set(re.findall(r"\bk_\w+", arg))
    return names


FILES = [_text(f) for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))]
FUNCTIONS = [_functions(t) for t in FILES]
KERNELS = sorted((k, f) for f, t in enumerate(FILES) for k in _dependent_kernels(t))


def test_every_kernel_is_found():
    assert {k for k, _ in KERNELS} == {
        "k_force_tile32", "k_force_tiny32", "k_force_tile64", "k_force_jmode64", "k_split_sums",
        "k_force6_tile32", "k_force6_sums", "k_correct6", "k_predict", "k_predict6", "k_correct",
        "k_advance"}


@pytest.mark.parametrize("kernel,file", KERNELS, ids=[k for k, _ in KERNELS])
def test_dependent_kernel_reads_coherently(kernel, file):
    assert "cudaGridDependencySynchronize()" in FUNCTIONS[file][kernel]
    # the kernel and the functions it calls, and theirs
    seen, todo = {kernel}, [FUNCTIONS[file][kernel]]
    while todo:
        code = todo.pop()
        assert "__ldg(" not in code and "__restrict__" not in code
        called = set(re.findall(r"\b([a-z]\w+)(?:<[^;()]*>)?\(", code)) - seen
        seen |= called
        todo += [f[name] for name in called for f in FUNCTIONS if name in f]
