"""Functions of the CUDA sources, compiled alone for the host with stand-ins for
what they call, so that a test can run their control flow without a GPU."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2103_05694_gb300", "csrc")


def source(name: str) -> str:
    """A source file without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def block(text: str, head: str) -> str:
    """From `head` to the brace that closes the first one opened after it."""
    start = text.index(head)
    depth = 0
    for k in range(text.index("{", start), len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[start:k + 1]
    raise ValueError(f"unbalanced braces after {head!r}")


def run(tmp_path, program: str, *args) -> subprocess.CompletedProcess:
    src, exe = tmp_path / "fragment.cpp", tmp_path / "fragment"
    src.write_text(program)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-pthread", "-w", "-o", str(exe), str(src)], check=True, timeout=300)
    return subprocess.run([str(exe), *map(str, args)], capture_output=True, text=True, timeout=300)
