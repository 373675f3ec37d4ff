"""What the library finds out about a device belongs to the context on it: no function keeps such a
value in a variable of its own across calls (an attribute set on one device does not hold on another,
and two threads would find it half set).  Function-local statics of the CUDA sources are constants,
which the language initialises once for all threads."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_07392_gb300", "csrc")


def local_statics(text):
    """Declarations of function-local static variables (indented, not of a constant)."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
    found = re.findall(r"^[ \t]+static\s+(?!const\b|constexpr\b|inline\b)[^;{()]*(?:=[^;]*)?;", text, flags=re.M)
    return [d.strip() for d in found if "(" not in d.split("=")[0]]


def test_the_search_finds_one():
    src = "void f()\n{\n    static bool done = false;\n    static const int k = 3;\n    static constexpr int n = 2;\n}\n"
    assert local_statics(src) == ["static bool done = false;"]


def test_no_function_keeps_state_between_calls():
    files = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))
    assert len(files) >= 6
    bad = {os.path.basename(f): local_statics(open(f).read()) for f in files}
    assert not any(bad.values()), {k: v for k, v in bad.items() if v}
