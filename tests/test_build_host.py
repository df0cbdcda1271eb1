"""The build's generated headers: a generator that was edited without its header is noticed, the slow zones'
tables are what their generator prints, and a failed generator leaves the header in place as it was."""
import os
import re
import shutil
import subprocess
import sys

import pytest

import __graft_entry__

CORE = "rox_core_tables.h"


@pytest.fixture
def build(monkeypatch, tmp_path):
    """The build module on a copy of its generators and headers."""
    m = __graft_entry__._build_module()
    src = tmp_path / "csrc"
    src.mkdir()
    for name in os.listdir(m.CSRC):
        if name.startswith("gen_") or name.endswith("_tables.h"):
            shutil.copy(os.path.join(m.CSRC, name), src)
    monkeypatch.setattr(m, "CSRC", str(src))
    monkeypatch.setattr(m, "BUILD", str(tmp_path))
    return m


def test_committed_headers_are_current(build):
    build.check_tables()


@pytest.mark.parametrize("generator", ["gen_core_tables.py", "gen_faddeeva_tables.py"])
def test_edited_generator_is_noticed(build, generator):
    path = os.path.join(build.CSRC, generator)
    with open(path, "a") as f:
        f.write("\nif __name__ == '__main__':\n    print('/* another line */')\n")
    with pytest.raises(RuntimeError, match="stale"):
        build.check_tables()


def test_failed_generator_leaves_the_header(build):
    build.make_interp_table()
    path = os.path.join(build.BUILD, "rox_interp_table.h")
    whole = open(path).read()
    assert len(whole) > 50_000
    with open(os.path.join(build.CSRC, "gen_interp_table.py"), "w") as f:
        f.write("print('half a', flush=True)\nraise SystemExit(1)\n")
    with pytest.raises(subprocess.CalledProcessError):
        build.make_interp_table()
    assert open(path).read() == whole
    assert sorted(n for n in os.listdir(build.BUILD) if "interp" in n) == ["rox_interp_table.h"]


def test_core_tables_regenerated(build):
    """Every number to within its printed digits (the nodes of the interpolants come from a
    floating-point fit, which may differ in the last digits between machines)."""
    pytest.importorskip("mpmath")
    pytest.importorskip("scipy")
    new = subprocess.run([sys.executable, os.path.join(build.CSRC, "gen_core_tables.py")], check=True,
                         capture_output=True, text=True).stdout
    old = open(os.path.join(build.CSRC, CORE)).read()
    num = re.compile(r"-?\d\.\d+e[+-]\d+")
    assert num.sub("#", new) == num.sub("#", old)
    a, b = ([float(v) for v in num.findall(t)] for t in (new, old))
    assert len(a) > 1500 and all(abs(x - y) <= 1e-6 * abs(y) + 1e-30 for x, y in zip(a, b))
