"""When the marshalling extension is compiled again (no GPU, nothing is compiled here)."""
import pytest

import paper_2603_15965_b200 as M
from paper_2603_15965_b200 import binding, build


@pytest.fixture
def compilations(monkeypatch):
    build.build_library()
    calls = []

    def compiler(cmd, **_):
        calls.append(cmd)
        raise RuntimeError("would compile")

    monkeypatch.setattr(build.subprocess, "run", compiler)
    return calls


def test_the_extension_is_not_compiled_again_for_the_torch_it_was_built_for(compilations):
    assert build.marshal_built_for() == build.marshal_abi()
    assert build.build_marshal() == build.MARSHAL_PATH and not compilations


@pytest.mark.parametrize("name,value", [("marshal_abi", lambda: "cpython-399 torch 9.9 cxx11abi 1"),
                                        ("MARSHAL_ABI_PATH", "/nonexistent/_marshal.abi")])        # built for what is not known
def test_the_extension_is_compiled_again_for_another_torch_or_interpreter(compilations, monkeypatch, name, value):
    monkeypatch.setattr(build, name, value)
    with pytest.raises(RuntimeError, match="would compile"):
        build.build_marshal()


def test_an_extension_built_for_another_torch_is_not_loaded(monkeypatch):
    monkeypatch.setattr(binding, "_marshal", None)
    monkeypatch.setattr(binding, "marshal_abi", lambda: "cpython-399 torch 9.9 cxx11abi 1")
    with pytest.raises(ImportError, match="was built for"):
        M.molora_group(None, 2)
