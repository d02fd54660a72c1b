"""What build() makes and when (CPU only)."""
from __future__ import annotations

import os
import sysconfig

import pytest

from paper_2606_21848_gb300 import builder


@pytest.fixture(scope="module", autouse=True)
def built():
    builder.build()


def test_the_module_is_named_for_the_interpreter():
    assert os.path.basename(builder.PYMOD) == "_keyless" + sysconfig.get_config_var("EXT_SUFFIX")


def test_another_interpreter_builds_its_own(tmp_path, monkeypatch):
    """A module built for another interpreter does not stand in for this one's, and the library, which
    has nothing to do with either, is not compiled again."""
    made = []
    monkeypatch.setattr(builder, "PYMOD", str(tmp_path / "_keyless.other.so"))
    monkeypatch.setattr(builder, "_build_library", lambda *a: made.append("library"))
    monkeypatch.setattr(builder, "_build_module", lambda *a: made.append("module"))
    builder.build()
    assert made == ["module"]
