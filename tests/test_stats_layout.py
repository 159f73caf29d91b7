"""The statistics structure of the C ABI: apply_products lies in what was padding, so that
every other field keeps its place for a program built against an earlier header."""
import ctypes
import os
import subprocess

from paper_1003_0524_gb300 import hfx

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_binding_and_header_agree(tmp_path):
    names = [f for f, _ in hfx.hfx_stats._fields_]
    src = tmp_path / "layout.c"
    src.write_text("#include <stdio.h>\n#include \"hfx.h\"\nint main(void) { printf(\"%zu\\n\", sizeof(hfx_stats));\n" +
                   "".join(f"printf(\"%zu\\n\", offsetof(hfx_stats, {n}));\n" for n in names) + "return 0; }\n")
    exe = tmp_path / "layout"
    subprocess.run(["gcc", "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src)], check=True)
    got = [int(x) for x in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()]
    assert got == [ctypes.sizeof(hfx.hfx_stats)] + [getattr(hfx.hfx_stats, n).offset for n in names]
    assert ctypes.sizeof(hfx.hfx_stats) == 128 and hfx.hfx_stats.flops_apply_exec.offset == 120
