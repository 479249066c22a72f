"""Tables that kernels read with loads wider than their elements declare the
loads' alignment: the language gives an array its element's alignment only,
and where the compiler places it depends on the tables around it."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2409_08729_gb300", "csrc")


def test_wide_table_loads_are_declared(tmp_path):
    # sources of the 16-byte reads of constant tables (the others read caller memory, behind a test of its address)
    found = set()
    for f in os.listdir(CSRC):
        if f.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, f)) as fh:
                found |= set(re.findall(r"reinterpret_cast<const (?:ulonglong2|longlong2|double2|int4|uint4|float4)\*>"
                                        r"\((lb_\w+)", fh.read()))
    assert "lb_kt_exp2" in found
    src = str(tmp_path / "a.cpp")
    with open(src, "w") as f:
        f.write('#include "lb_ktrap.cuh"\n#include "lb_uniform.cuh"\n')
        for t in sorted(found):
            f.write('static_assert(__alignof__(%s) >= 16, "%s");\n' % (t, t))
    subprocess.run(["g++", "-std=c++17", "-fsyntax-only", "-I", CSRC, src], check=True)
