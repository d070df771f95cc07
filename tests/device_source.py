"""Device functions of csrc/, taken from their sources by name and compiled for
the host: for what a test must not try on a GPU (accesses out of range, threads
whose barriers do not pair up)."""
import os
import re
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1708_01159_gb300", "csrc")


def function(path, name):
    """The source text of function (or struct) `name`, its template line included."""
    text = open(os.path.join(CSRC, path)).read()
    at = re.search(r"^(template <[^\n]*>\n)?(struct " + name + r" \{|\w[^\n;{}]*\b" + name + r"\()", text, re.M)
    assert at, f"{name} not found in {path}"
    pos = text.index("{", at.end() - 1)
    depth, end = 0, pos
    while True:
        depth += {"{": 1, "}": -1}.get(text[end], 0)
        end += 1
        if depth == 0:
            break
    return text[at.start():end] + (";" if text[end:end + 1] == ";" else "") + "\n"


def constant(path, name):
    text = open(os.path.join(CSRC, path)).read()
    return re.search(r"^(static )?constexpr [^\n]*\b" + name + r"\b = [^;]*;", text, re.M).group(0) + "\n"


def build(tmp_path, source):
    """Compile `source` after host_cuda.h: the program's path."""
    src, exe = os.path.join(tmp_path, "t.cpp"), os.path.join(tmp_path, "t")
    with open(src, "w") as fh:
        fh.write('#include "host_cuda.h"\n' + source)
    r = subprocess.run(["g++", "-std=c++20", "-O1", "-w", "-fwrapv", "-pthread", "-I", HERE, src, "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    return exe


def execute(exe, *args, timeout=120):
    """(exit status, output)"""
    r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=timeout)
    return r.returncode, r.stdout + r.stderr


def run(tmp_path, source, *args):
    return execute(build(tmp_path, source), *args)
