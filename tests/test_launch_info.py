"""kn_get_launch_info on the CPU: the binding's mirror of kn_launch_info and the errors."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_layout_and_errors(tmp_path):
    from paper_1409_5826_gb300 import build, kn
    build.build()
    assert kn.lib().kn_get_launch_info(None, None) == kn.KN_ERR_INVALID_ARG
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        pytest.skip("no C compiler")
    names = [f for f, _ in kn._LaunchInfo._fields_]
    src = tmp_path / "o.c"
    src.write_text('#include <stddef.h>\n#include <stdio.h>\n#include "kn.h"\nint main(void) {\n'
                   + "".join(f'  printf("%zu\\n", offsetof(kn_launch_info, {n}));\n' for n in names)
                   + '  printf("%zu\\n", sizeof(kn_launch_info));\n  return 0;\n}\n')
    subprocess.run([cc, "-std=c99", "-I", os.path.join(ROOT, "include"), str(src), "-o", str(tmp_path / "o")],
                   check=True)
    out = subprocess.run([str(tmp_path / "o")], check=True, capture_output=True, text=True).stdout.split()
    assert [int(x) for x in out] == [getattr(kn._LaunchInfo, n).offset for n in names] + [C.sizeof(kn._LaunchInfo)]
