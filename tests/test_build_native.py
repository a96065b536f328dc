"""The build of the binding's marshalling module."""
import os
import shutil

import pytest

from paper_1611_07151_b200 import build


@pytest.fixture
def tree(tmp_path, monkeypatch):
    """A copy of what the module is built from, built once, with the module older than nothing it depends on."""
    shutil.copy(build.NATIVE_SRC, tmp_path / "binding_native.c")
    shutil.copytree(os.path.join(build.ROOT, "include"), tmp_path / "include")
    monkeypatch.setattr(build, "ROOT", str(tmp_path))
    monkeypatch.setattr(build, "NATIVE_SRC", str(tmp_path / "binding_native.c"))
    monkeypatch.setattr(build, "NATIVE", str(tmp_path / os.path.basename(build.NATIVE)))
    build.build_native()
    for f in (build.NATIVE_SRC, str(tmp_path / "include" / "sqn.h"), build.NATIVE):
        os.utime(f, (1000, 1000))
    return tmp_path


@pytest.mark.parametrize("changed", ["binding_native.c", os.path.join("include", "sqn.h")])
def test_built_again_when_a_source_or_the_header_is_newer(tree, changed):
    """The module fills in sqn_conv_opts: a changed struct and an old module would pass the options in the wrong places."""
    build.build_native()
    assert os.path.getmtime(build.NATIVE) == 1000
    os.utime(tree / changed, (2000, 2000))
    build.build_native()
    assert os.path.getmtime(build.NATIVE) > 2000
