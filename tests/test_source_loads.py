"""Arrays that a kernel of the step writes are read by ordinary loads.  The step's
kernels start before their predecessor has ended and wait inside; a non-coherent
load (__ldg and the *_const helpers) asks for memory that stays read-only while
the kernel lives and may be moved ahead of that wait."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_06546_gb300", "csrc")
CONST_LOADS = r"(?:__ldg|\b\w+_const(?:<[^<>;()]*>)?|load_uw)\("


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _written_members():
    """The pointer members of DevCase to non-const data."""
    body = re.search(r"struct DevCase \{(.*?)\n\};", _source("ugks_device.cuh"), re.S).group(1)
    out = set()
    for decl in body.split(";"):
        decl = " ".join(decl.split())
        if "*" in decl and not decl.startswith("const"):
            out |= set(re.findall(r"\*\s*(\w+)", decl))
    return out


def _argument(text, at):
    depth, i = 1, at
    while depth:
        depth += {"(": 1, ")": -1}.get(text[i], 0)
        i += 1
    return text[at:i - 1]


def test_arrays_written_in_a_step_are_read_by_ordinary_loads():
    written = _written_members()
    assert {"f_cur", "flux", "krec", "crec", "wrec", "grec", "fside", "xrec", "W"} <= written
    assert not {"uw", "gf", "gi", "eps2", "owned"} & written
    seen = 0
    for name in ("ugks_device.cuh", "ugks_kernels.cu"):
        text = _source(name)
        for m in re.finditer(CONST_LOADS, text):
            arg = _argument(text, m.end())
            members = set(re.findall(r"\bdc\.(\w+)", arg))
            seen += bool(members)
            assert not members & written, (name, m.group(0) + arg)
            # local pointers into f and the flux buffer
            assert not re.search(r"\b(fl|fo|fc|frow|Fr)\b", arg), (name, m.group(0) + arg)
        for m in re.finditer(r"__restrict__\s+\w+\s*=\s*([^;]*);", text):
            assert not set(re.findall(r"\bdc\.(\w+)", m.group(1))) & written, (name, m.group(0))
    assert seen >= 10
