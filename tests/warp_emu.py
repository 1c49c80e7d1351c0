"""Kernels of the library compiled for the host by their own text (``native/warp_emu.h``): the named top-level
declarations of a source file, and a driver that runs them."""
import os
import re
import subprocess

import paper_1709_03565_gb300._build as _build

NATIVE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native")


def _chunks(text):
    """Top-level declarations of a source file, comments and preprocessor lines removed, namespaces opened."""
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    text = re.sub(r"//[^\n]*", "", text)
    text = re.sub(r"^[ \t]*#(?!pragma unroll)(?:[^\n]*\\\n)*[^\n]*$", "", text, flags=re.M)
    text = re.sub(r"^[ \t]*#pragma unroll.*$", "", text, flags=re.M)
    text = re.sub(r"\bnamespace\s+\w*\s*\{", "", text)
    out, start, depth = [], 0, 0
    for i, c in enumerate(text):
        if c in "({[":
            depth += 1
        elif c in ")}]":
            depth = max(0, depth - 1)
            if c == "}" and depth == 0 and not re.match(r"\s*;", text[i + 1:]):
                out.append(text[start:i + 1])
                start = i + 1
        elif c == ";" and depth == 0:
            out.append(text[start:i + 1])
            start = i + 1
    return [x.strip() for x in out if x.strip()]


def _declares(chunk, name):
    head = re.sub(r"^template\s*<[^>]*>|__launch_bounds__\s*\([^)]*\)|__align__\(\d+\)", "", chunk)
    head = re.split(r"\{|=(?!=)", head, maxsplit=1)[0]
    head = head.split("(", 1)[0] if "(" in head else head
    return re.search(r"\b%s\s*$" % re.escape(name), re.sub(r"\[[^\]]*\]\s*$", "", head.rstrip().rstrip(";"))) is not None


def build(tmp_path, source, names, driver):
    """Compiles ``names`` of ``csrc/source`` and the driver text; the path of the program."""
    chunks = _chunks(open(os.path.join(_build.CSRC, source)).read())
    picked = []
    for c in chunks:
        if any(_declares(c, n) for n in names) and re.search(r"[{=]", c):
            picked.append(c)
    for n in names:
        assert any(_declares(c, n) for c in picked), n
    body = "\n\n".join(picked)
    body = re.sub(r"extern\s+__shared__", "extern", body)
    src = os.path.join(str(tmp_path), "emu.cpp")
    with open(src, "w") as f:
        f.write('#include "warp_emu.h"\n' + driver.replace("//KERNELS//", body))
    exe = os.path.join(str(tmp_path), "emu")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I", NATIVE, src, "-o", exe], check=True)
    return exe
