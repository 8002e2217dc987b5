"""Device functions of the library run on the host: their text is taken from the
sources as it stands and compiled with g++ against host stand-ins for the memory
accesses, which a test supplies. What they decide can then be checked for every
order of events, and counted, without a GPU."""

import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1712_09624_gb300", "csrc")

PRELUDE = """
#include <cstdint>
#include <cstddef>
#define __device__
#define __host__
#define __forceinline__ inline
struct uint2 { uint32_t x, y; };
static inline int __ffs(uint32_t v) { return __builtin_ffs((int)v); }
"""


def source(name: str) -> str:
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def between(text: str, start: str, end: str) -> str:
    """The part of text from the line that holds start up to the one that holds end."""
    a = text.rfind("\n", 0, text.index(start)) + 1
    return text[a:text.rfind("\n", 0, text.index(end, a)) + 1]


def definition(text: str, name: str) -> str:
    """The definition of the function, struct or enum of that name at the start of a line."""
    m = re.search(r"^(?:(?:struct|enum) %s\b|[\w ]*[\w*&>] \**&?%s\()" % (name, name), text, re.M)
    assert m, name
    start = m.start()
    if text[:start].rstrip("\n").endswith(">"):  # its template line
        line = text.rfind("\n", 0, start - 1) + 1
        if text.startswith("template", line):
            start = line
    brace = text.index("{", m.end() - 1)
    end = text.index("\n}", brace) + 2 if "\n" in text[brace:text.index("}", brace)] else text.index("}", brace) + 1
    return text[start:text.index("\n", end) + 1] + "\n"


def definitions(file: str, *names: str) -> str:
    text = source(file)
    return "".join(definition(text, n) for n in names)


def layout() -> str:
    """Constants, hashes, timers and addressing of ckpp_device.cuh."""
    return between(source("ckpp_device.cuh"), "constexpr uint32_t kSlots", "place in the stream")


def build(tmp_path, code: str) -> str:
    src, lib = str(tmp_path / "model.cpp"), str(tmp_path / "model.so")
    with open(src, "w") as f:
        f.write(PRELUDE + code)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-o", lib, src], check=True, capture_output=True,
                   text=True)
    return lib
