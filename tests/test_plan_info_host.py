"""sphynx_plan_info as the C compiler lays it out equals the binding's."""

import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_plan_info_layout(tmp_path):
    import paper_2105_00578_gb300 as spx
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        pytest.skip("no C compiler")
    fields = [f for f, _ in spx.PlanInfo._fields_]
    src = tmp_path / "layout.c"
    src.write_text('#include <stdio.h>\n#include <stddef.h>\n#include "sphynx.h"\nint main(void) {\n' + "".join(
        f'  printf("%zu\\n", offsetof(sphynx_plan_info, {f}));\n' for f in fields) +
        '  printf("%zu\\n", sizeof(sphynx_plan_info));\n  return 0;\n}\n')
    exe = tmp_path / "layout"
    subprocess.run([cc, "-std=c11", "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True)
    got = [int(v) for v in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]
    assert got == [getattr(spx.PlanInfo, f).offset for f in fields] + [ctypes.sizeof(spx.PlanInfo)]
