"""The call module reads torch's tensors by the layout that it was compiled against: another torch, ABI or Python has to build it again
and must not load it."""
import os

import pytest


@pytest.fixture()
def build():
    from paper_2511_04214_b200 import build
    build.build()
    return build


def other_build(build, path):
    """The module as another torch of the same length of name would have left it."""
    data, tag = open(build.CALL_SO, "rb").read(), build.call_tag().encode()
    assert data.count(tag + b"\0") == 1
    open(path, "wb").write(data.replace(tag, tag.replace(b"torch ", b"t0rch ")))
    return str(path)


def test_a_module_of_another_torch_is_stale(build, monkeypatch, tmp_path):
    assert not build._call_stale()
    monkeypatch.setattr(build, "CALL_SO", other_build(build, tmp_path / "_call.so"))
    assert os.path.getmtime(build.CALL_SO) >= os.path.getmtime(build.CALL_SOURCE)
    assert build._call_stale()


def test_a_module_of_another_torch_is_not_loaded(build, tmp_path):
    from paper_2511_04214_b200 import binding
    assert binding._load_call(build.CALL_SO).TAG == build.call_tag()
    with pytest.raises(ImportError, match="t0rch"):
        binding._load_call(other_build(build, tmp_path / "_call.so"))
