"""The argument-marshalling module depends on the torch and the Python it was compiled for: another one's is built again,
and refused if it is met all the same."""
import os
import shutil

import pytest
import torch

import agtest as T
from paper_2410_12876_b200 import binding as ag
from paper_2410_12876_b200 import build


@pytest.fixture(autouse=True)
def _lib():
    T.ensure_built()


def test_the_tag_is_in_the_module():
    assert build.marshal_matches(build.MARSHAL)
    assert ag._marshal().tag == build.marshal_tag()
    assert torch.__version__ in build.marshal_tag()


def test_a_module_for_another_torch_is_built_again(monkeypatch, tmp_path):
    old = shutil.copy2(build.MARSHAL, tmp_path / "_marshal.so")        # times and all
    monkeypatch.setattr(build, "MARSHAL", str(old))
    calls = []
    monkeypatch.setattr(build.subprocess, "run", lambda cmd, **kw: calls.append(cmd))
    build.build_marshal()
    assert not calls                                                   # as it is: up to date
    monkeypatch.setattr(torch, "__version__", "9.9.9")
    build.build_marshal()
    assert len(calls) == 1 and any("9.9.9" in a for a in calls[0])


def test_a_module_for_another_torch_is_refused(monkeypatch):
    monkeypatch.setattr(torch, "__version__", "9.9.9")
    monkeypatch.setattr(ag, "_m", None)
    with pytest.raises(RuntimeError, match="another torch"):
        ag._marshal()
    assert ag._m is None and os.path.exists(build.MARSHAL)
