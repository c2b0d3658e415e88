"""Compiles a kernel file of the library for the host (tests/emulator.h), so that its kernels run on
the CPU under chosen schedules. The source is taken as it is, but for what is no C++: launches become
calls, and the few PTX statements the kernels use become the loads and stores that they stand for."""
from __future__ import annotations

import ctypes
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2410_10094_gb300", "csrc")
HERE = os.path.dirname(os.path.abspath(__file__))


def split_top(text: str):
    """Splits at the commas that no bracket encloses."""
    parts, depth, last = [], 0, 0
    for i, ch in enumerate(text):
        depth += ch in "([{"
        depth -= ch in ")]}"
        if ch == "," and depth == 0:
            parts.append(text[last:i].strip())
            last = i + 1
    return parts + [text[last:].strip()]


def closing(text: str, at: int) -> int:
    """The index of the parenthesis that closes the one at `at` (string literals skipped)."""
    depth, quoted = 0, False
    for i in range(at, len(text)):
        if text[i] == '"' and text[i - 1] != "\\":
            quoted = not quoted
        if quoted:
            continue
        depth += text[i] == "("
        depth -= text[i] == ")"
        if depth == 0:
            return i
    raise ValueError("unbalanced parentheses")


def ptx(statement: str) -> str:
    """What one asm statement does, in C++."""
    code = re.match(r'\s*((?:"(?:[^"\\]|\\.)*"\s*)+)', statement).group(1)
    ops = [statement[m.end():closing(statement, m.end()) + 1] for m in re.finditer(r'"[=+]?[rlfdh]"(?=\()', statement)]
    if "lanemask_lt" in code:
        return f"{ops[0]} = (1u << (threadIdx.x & 31)) - 1u;"
    if "createpolicy" in code:
        return f"{ops[0]} = 0;"
    if "ld.global.nc" in code:
        return f"{ops[0]} = *{ops[1]};"
    if "atom.shared.add" in code:
        return f"{ops[0]} = atomicAdd((uint32_t*){ops[1]}, 1u);"
    m = re.search(r"st\.global.*?(v[24])?\.[sf](?:32|64) ", code)
    if m:
        n = int((m.group(1) or "v1")[1])
        return " ".join(f"({ops[0]})[{k}] = {ops[1 + k]};" for k in range(n))
    return "__builtin_trap();"  # not used by the kernels under test


def host_source(text: str) -> str:
    out, at = [], 0
    for m in re.finditer(r"\basm( volatile)?\(", text):
        if m.start() < at:
            continue
        end = closing(text, m.end() - 1)
        out.append(text[at:m.start()] + "{ " + ptx(text[m.end():end]) + " }")
        at = end + 2  # and the semicolon
    text = "".join(out) + text[at:]
    text = re.sub(r"extern __shared__ __align__\(\d+\) unsigned char (\w+)\[\];",
                  r"unsigned char* const \1 = emu::shared_mem;", text)
    text = re.sub(r"\(uint32_t\)__cvta_generic_to_shared\(p\)", "(uintptr_t)p", text)
    text = text.replace("uint32_t smem_addr(", "uintptr_t smem_addr(")
    while True:
        m = re.search(r"([\w:]+(?:<[\w, :]+>)?)\s*<<<(.*?)>>>\s*\(", text, re.S)
        if not m:
            return text
        end = closing(text, m.end() - 1)
        grid, block = split_top(m.group(2))[:2]
        text = (text[:m.start()] + f"emu::launch({grid}, {block}, [&] {{ {m.group(1)}({text[m.end():end]}); }})" +
                text[end + 1:])


def build(folder, source: str, harness: str) -> ctypes.CDLL:
    """The shared library of csrc/<source> with `harness` (C++, extern "C") behind it, made in `folder`."""
    folder = str(folder)
    for name in os.listdir(CSRC):
        if name.endswith((".cuh", ".h")):
            with open(os.path.join(CSRC, name)) as f, open(os.path.join(folder, name), "w") as g:
                g.write(host_source(f.read()))
    with open(os.path.join(folder, "cuda_runtime.h"), "w") as f:
        f.write('#include "emulator.h"\n')
    cpp, lib = os.path.join(folder, "kernel.cpp"), os.path.join(folder, "libkernel.so")
    with open(os.path.join(CSRC, source)) as f, open(cpp, "w") as g:
        g.write(host_source(f.read()) + "\nnamespace stc { void note_launch(unsigned) {} }\n" + harness)
    cmd = ["g++", "-std=c++20", "-O1", "-w", "-fno-strict-aliasing", "-ffp-contract=off", "-shared", "-fPIC", "-I", folder,
           "-I", HERE, "-I", os.path.join(ROOT, "include"), cpp, "-o", lib]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, "\n".join(l for l in r.stderr.splitlines() if "error" in l)
    return ctypes.CDLL(lib)
