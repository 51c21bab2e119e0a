"""When the binding's native marshalling is compiled again."""
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
