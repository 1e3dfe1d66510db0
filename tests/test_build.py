"""build.py and the loading of what it builds: the library does not hang on the module that makes the usual calls faster."""
import importlib
import subprocess

import pytest


@pytest.fixture()
def build(monkeypatch, tmp_path):
    """build.py with its outputs in a folder of the test's own, and compilers that are only noted."""
    build = importlib.import_module("paper_2609_10937_b200.build")
    monkeypatch.setattr(build, "PKG", tmp_path)
    monkeypatch.setattr(build, "LIB", tmp_path / "libattn_b200.so")
    ran = []

    def run(cmd, check):
        ran.append(cmd[0])
        with open(cmd[cmd.index("-o") + 1], "wb") as fh:
            fh.write(b"built")

    monkeypatch.setattr(build.subprocess, "run", run)
    monkeypatch.setattr(build, "ran", ran, raising=False)
    return build


@pytest.mark.parametrize("failure", [FileNotFoundError("g++"), subprocess.CalledProcessError(1, "g++"), ImportError("torch")])
def test_without_a_compiler_or_headers_for_the_module_the_library_is_built(build, monkeypatch, failure):
    build.fast_path().write_bytes(b"of older sources")

    def command(out):
        out.write_bytes(b"half")
        raise failure

    monkeypatch.setattr(build, "_fast_command", command)
    with pytest.warns(UserWarning, match="binding.py makes every call"):
        assert build.build(force=True) == build.LIB
    assert build.LIB.read_bytes() == b"built" and len(build.ran) == 1
    assert sorted(p.name for p in build.PKG.iterdir()) == [build.LIB.name]


def test_a_module_of_another_version_is_built_anew(build, monkeypatch):
    assert build.build(force=True) == build.LIB and not build.needs_build() and len(build.ran) == 2
    mine = build.fast_path()
    monkeypatch.setattr(build.metadata, "version", lambda name: "1.2.3")
    assert build.needs_build() and build.fast_path() != mine
    build.build()
    assert not build.needs_build() and len(build.ran) == 3                   # the library was not stale
    assert sorted(p.name for p in build.PKG.iterdir()) == sorted([build.LIB.name, build.fast_path().name])


def test_a_module_that_cannot_be_loaded_leaves_the_calls_to_binding(build, monkeypatch):
    torch = importlib.import_module("torch")
    binding = importlib.import_module("paper_2609_10937_b200.binding")
    build.fast_path().write_bytes(b"no module")
    monkeypatch.setattr(binding, "_fast", binding._LazyFast())
    q = torch.zeros(1, 1, 8, 64, dtype=torch.bfloat16)
    with pytest.warns(UserWarning, match="cannot be loaded"), pytest.raises(ValueError, match="CUDA tensors"):
        binding.forward(q, q, q)
    assert binding._fast is binding._NoFast
