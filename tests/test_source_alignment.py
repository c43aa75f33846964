"""Wide accesses through a pointer cast need an address that is known to be
aligned: an automatic array has only its element's alignment, so none may be
read or written as a wider vector (it works only while the compiler keeps the
array in registers) unless it is declared alignas(16)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_00387_gb300", "csrc")
WIDE = r"reinterpret_cast<(?:const )?(?:uint[24]|int[24]|double2|float[24]|ulonglong2|longlong2)\s*\*>\(&?(\w+)\b"


def _offenders(text):
    text = re.sub(r"//[^\n]*", "", text)
    out = []
    for m in re.finditer(WIDE, text):
        name = m.group(1)
        # declarations of arrays of that name in the enclosing function (back to
        # the last line that starts in column 0 with a closing brace)
        start = text.rfind("\n}", 0, m.start()) + 1
        for d in re.finditer(r"([^;{}]*?)\b" + name + r"\[[^\];]*\]\s*;", text[start:m.start()]):
            decl = re.sub(r"\([^()]*\)", "()", d.group(1)).strip()  # type words before the name
            if re.fullmatch(r"(?:const |unsigned )*\w[\w:<>]*", decl) and decl != "return":
                out.append(name)
                break
    return out


def test_the_scan_sees_a_plain_array():
    assert _offenders("void f() {\n  double q[8];\n  *reinterpret_cast<uint4*>(q + 2) = z;\n}\n") == ["q"]
    assert _offenders("void f() {\n  alignas(16) double q[8];\n  *reinterpret_cast<uint4*>(q) = z;\n}\n") == []
    assert _offenders("void f(double* q) {\n  q[0] = 1;\n  *reinterpret_cast<uint4*>(q) = z;\n}\n") == []


def test_no_plain_automatic_array_is_accessed_as_a_vector():
    files = sorted(glob.glob(os.path.join(CSRC, "*.cu*")))
    assert files
    bad = {os.path.basename(f): o for f in files for o in [_offenders(open(f).read())] if o}
    assert bad == {}
