"""Compiles device code of the library for the CPU (see host_cuda.h), so that tests without a GPU run the
source that ships and not a restatement of it."""
import ctypes
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2402_09633_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def between(text, start, end):
    """The part of text from `start` up to `end`, both of which must be there."""
    a = text.index(start)
    return text[a:text.index(end, a)]


def replace(text, old, new):
    """text with every `old` replaced; there must be one."""
    assert old in text, f"not in the source: {old}"
    return text.replace(old, new)


def compile_host(folder, main, files=(), flags=()):
    """main (C++ text) and the named files beside it, compiled into a library that is loaded."""
    with open(os.path.join(HERE, "host_cuda.h")) as f:
        shim = f.read()
    for name, text in [("ptx.cuh", shim), ("main.cpp", main), *files]:
        (folder / name).write_text(text)
    lib = folder / "host.so"
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-ffp-contract=off", "-fno-strict-aliasing", "-w",
                    *flags, "-o", str(lib), str(folder / "main.cpp")], check=True)
    return ctypes.CDLL(str(lib))
