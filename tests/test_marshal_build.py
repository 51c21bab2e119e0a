"""When the binding's native marshalling is compiled again, and what an import
without it says."""
import os
import shutil
import subprocess
import sys

import pytest
import torch

from paper_2608_02625_gb300 import build


@pytest.fixture(autouse=True)
def built():
    build.build()


def test_up_to_date_after_a_build():
    assert not build._marshal_stale(False)


@pytest.mark.parametrize("version", ["2.9.1+cu130", torch.__version__ + "x"])
def test_stale_under_another_torch(monkeypatch, version):
    """It links against torch's C++ libraries, whose interfaces change with the version."""
    if version == torch.__version__:
        pytest.skip("the version that is here")
    monkeypatch.setattr(torch, "__version__", version)
    assert build._marshal_stale(False)


def test_stale_where_nothing_says_what_it_was_built_for(monkeypatch, tmp_path):
    monkeypatch.setattr(build, "BUILD", str(tmp_path))
    assert build._marshal_stale(False)


@pytest.mark.parametrize("content", [None, b"not a library"], ids=["missing", "unusable"])
def test_import_without_it_says_how_to_build_it(tmp_path, content):
    pkg = tmp_path / "paper_2608_02625_gb300"
    pkg.mkdir()
    for f in os.listdir(build.PKG):
        if f.endswith(".py") or f == "libdlmrefine.so":
            shutil.copy(os.path.join(build.PKG, f), pkg / f)
    if content is not None:
        (pkg / "_marshal.so").write_bytes(content)
    r = subprocess.run([sys.executable, "-c", "import paper_2608_02625_gb300.binding"], cwd=tmp_path, capture_output=True,
                       text=True, env={**os.environ, "PYTHONPATH": str(tmp_path)})
    last = r.stderr.strip().splitlines()[-1]
    assert r.returncode != 0 and last.startswith("ImportError")
    assert "_marshal.so" in last and "python -m paper_2608_02625_gb300.build" in last
