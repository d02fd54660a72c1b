"""The binding's C module calls the library that the package has loaded, also when the loader's search
path holds another copy of it (CPU only)."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

import pytest

import paper_2606_21848_gb300 as kl
from paper_2606_21848_gb300 import builder

CODE = """
import paper_2606_21848_gb300 as kl
try:
    kl.kl_append_v(kl.make_shape(2, 8, 2, 128, 16, 64, 32), None, 16, 16, 16, None, 0)
except kl.KLError:
    pass
maps = {l.split()[-1] for l in open("/proc/self/maps") if l.rstrip().endswith("libkeyless.so")}
print(len(maps), *maps)
"""


@pytest.mark.skipif(not os.path.exists("/proc/self/maps"), reason="needs /proc")
def test_one_copy_of_the_library(tmp_path):
    kl.build()
    shutil.copy(builder.LIB, tmp_path / "libkeyless.so")
    env = dict(os.environ, LD_LIBRARY_PATH=str(tmp_path))
    r = subprocess.run([sys.executable, "-c", CODE], cwd=builder.ROOT, env=env, capture_output=True, text=True,
                       check=True)
    assert r.stdout.split() == ["1", os.path.realpath(builder.LIB)], r.stdout
