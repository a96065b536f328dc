"""The build of the binding's marshalling module."""
import os
import shutil
import subprocess
import sys
import sysconfig

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


IMPORT = """
import sys
sys.path.insert(0, %r)
from paper_1611_07151_b200 import binding
print(binding._native is not None)
"""


def imported(package_parent):
    r = subprocess.run([sys.executable, "-c", IMPORT % str(package_parent)], capture_output=True, text=True, check=True)
    return r.stdout.strip() == "True"


def test_only_the_interpreter_it_is_built_for_takes_the_module(tree):
    """A plain .so is imported by every Python version, whatever its C API."""
    suffix = sysconfig.get_config_var("EXT_SUFFIX")
    assert os.path.basename(build.NATIVE) == "_native" + suffix
    package = tree / "paper_1611_07151_b200"
    package.mkdir()
    for f in ("__init__.py", "binding.py"):
        shutil.copy(os.path.join(build.PKG, f), package / f)
    shutil.copy(build.NATIVE, package / ("_native" + suffix))
    assert imported(tree)
    os.rename(package / ("_native" + suffix), package / "_native.cpython-39-x86_64-linux-gnu.so")
    assert not imported(tree)


def test_a_module_for_another_options_struct_is_left_alone(tree):
    header = tree / "include" / "sqn.h"
    header.write_text(header.read_text().replace("int fuse_global_avgpool;", "int fuse_global_avgpool; double more;"))
    assert "double more" in header.read_text()
    build.build_native(force=True)
    package = tree / "paper_1611_07151_b200"
    package.mkdir()
    for f in ("__init__.py", "binding.py"):
        shutil.copy(os.path.join(build.PKG, f), package / f)
    shutil.copy(build.NATIVE, package)
    assert not imported(tree)


@pytest.mark.parametrize("compiler", ["false", "/nowhere/gcc"])
def test_the_library_builds_without_the_module(tree, monkeypatch, compiler):
    """No compiler or no Python.h: ctypes marshals the calls, and a module older than its sources does not stay."""
    monkeypatch.setenv("CC", compiler)
    monkeypatch.setattr(build, "up_to_date", lambda lib=None: True)
    os.utime(tree / "include" / "sqn.h", (2000, 2000))
    with pytest.warns(UserWarning, match="marshalling module"):
        assert build.build() == build.LIB
    assert not os.path.exists(build.NATIVE)
