"""The build of the library and of the binding's compiled part, with compilers that only write down that they were called."""
import os
import shutil
import stat
import subprocess
import sys

import pytest

from paper_2501_04052_b200 import build


@pytest.fixture
def tree(tmp_path, monkeypatch):
    """A copy of the sources; `calls()` lists the compilers' calls so far, compiler(name, works) sets one up."""
    root = tmp_path / "paper_2501_04052_b200"
    shutil.copytree(build.CSRC, root / "csrc", ignore=shutil.ignore_patterns("*.o"))
    shutil.copytree(os.path.join(os.path.dirname(build.HERE), "include"), tmp_path / "include")
    shutil.copy(os.path.join(build.HERE, "build.py"), root / "build.py")
    log = tmp_path / "log"
    log.write_text("")

    class Tree:
        def compiler(self, variable, works):
            script = tmp_path / variable
            script.write_text('#!/bin/sh\necho %s >> %s\n%s\nwhile [ $# -gt 0 ]; do [ "$1" = -o ] && echo built > "$2"; shift; done\n'
                              % (variable, log, "" if works else "exit 1"))
            script.chmod(script.stat().st_mode | stat.S_IXUSR)
            monkeypatch.setenv(variable, str(script))

        def build(self, *args, torch=True):
            hide = "" if torch else "sys.modules['torch'] = None; "
            code = "import sys; %ssys.argv[0] = 'build'; import runpy; runpy.run_path(%r, run_name='__main__')" % (hide, str(root / "build.py"))
            return subprocess.run([sys.executable, "-c", code, *args], capture_output=True, text=True, timeout=300)

        def calls(self):
            out = log.read_text().split()
            log.write_text("")
            return out

        def path(self, *parts):
            return os.path.join(root, *parts)

        def files(self, end):
            return [f for f in os.listdir(root) if f.endswith(end)]

    t = Tree()
    t.compiler("NVCC", True)
    t.compiler("CXX", True)
    return t


LIBRARY = ["NVCC"] * (len(build.SOURCES) + 1)


def test_library_and_compiled_part_are_built_once(tree):
    assert tree.build().returncode == 0
    assert tree.calls() == LIBRARY + ["CXX"]
    assert sorted(f[:10] for f in tree.files(".so")) == ["librazer.s", "razer_call"]
    assert tree.build().returncode == 0 and tree.calls() == []
    later = os.path.getmtime(tree.path("librazer.so")) + 10
    os.utime(tree.path("csrc", "razer_call.cpp"), (later, later))
    assert tree.build().returncode == 0 and tree.calls() == ["CXX"]


def test_library_is_built_without_torch(tree):
    r = tree.build(torch=False)
    assert r.returncode == 0, r.stderr
    assert tree.calls() == LIBRARY and tree.files(".so") == ["librazer.so"]
    assert tree.build(torch=False).returncode == 0 and tree.calls() == []


def test_library_is_built_without_a_host_compiler_and_not_again(tree):
    tree.compiler("CXX", False)
    assert tree.build().returncode == 0
    assert tree.calls() == LIBRARY + ["CXX"] and tree.files(".so") == ["librazer.so"]
    assert tree.build().returncode == 0 and tree.calls() == []
    assert tree.build("--force").returncode == 0 and tree.calls() == LIBRARY + ["CXX"]


def test_a_compiled_part_that_no_longer_builds_is_not_left_behind(tree):
    assert tree.build().returncode == 0
    tree.calls()
    tree.compiler("CXX", False)
    later = os.path.getmtime(tree.path("librazer.so")) + 10
    os.utime(tree.path("csrc", "razer_call.cpp"), (later, later))
    assert tree.build().returncode == 0
    assert tree.calls() == ["CXX"] and tree.files(".so") == ["librazer.so"]


def test_compiled_part_is_for_one_torch_and_one_interpreter(tree, monkeypatch):
    """Its file says what it was built for; where that is not what is installed it is not loaded, and build() makes another one."""
    import sysconfig

    import torch
    from paper_2501_04052_b200 import binding as b
    assert sysconfig.get_config_var("SOABI") in build.call_path() and build.call_path(torch.__version__) == build.call_path()
    assert len({build.call_path(v) for v in ("2.11.0+cu128", "2.11.0+cpu", "2.12.0+cu128", "none")}) == 4
    assert b._load_call()[0] is not None and b.call_route().startswith("compiled")
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    module, route = b._load_call()
    assert module is None and route.startswith("ctypes") and "torch-0_0_1" in route
    # a file for another torch: built anew, the other one gone
    assert tree.build().returncode == 0
    mine, = (f for f in tree.files(".so") if f.startswith("razer_call."))
    other = tree.path("razer_call.cpython-399-x86_64-linux-gnu.torch-9_9_9.so")
    os.rename(tree.path(mine), other)
    tree.calls()
    assert tree.build().returncode == 0 and tree.calls() == ["CXX"]
    assert os.path.exists(tree.path(mine)) and not os.path.exists(other)
