"""The build of the in-tree libraries: what makes one out of date (no GPU, no compiler run)."""
import importlib.metadata
import sysconfig

from paper_2511_22972_b200 import build


def test_another_python_or_torch_has_an_extension_of_its_own(monkeypatch):
    # it is bound to one ABI of each: under the same name, an upgrade in place would load what it cannot use
    import importlib.util
    assert importlib.metadata.version("torch") in build.NATIVE_PATH and sysconfig.get_config_var("SOABI") in build.NATIVE_PATH
    real = importlib.metadata.version
    monkeypatch.setattr(importlib.metadata, "version", lambda name: "99.0" if name == "torch" else real(name))
    spec = importlib.util.spec_from_file_location("upgraded_build", build.__file__)
    upgraded = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(upgraded)
    assert upgraded.NATIVE_PATH != build.NATIVE_PATH and upgraded.native_is_stale()
    assert upgraded.LIB_PATH == build.LIB_PATH                # (the library itself knows neither)


def test_a_failing_extension_is_named(monkeypatch):
    from paper_2511_22972_b200 import binding
    import pytest
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(binding._build, "NATIVE_PATH", "/nonexistent/_native.other.so")
    monkeypatch.setattr(binding._build, "ensure_built", lambda: build.LIB_PATH)
    with pytest.raises(ImportError, match="_native.other.so could not be loaded"):
        binding.lib()


def test_a_build_replaces_its_file_only_when_it_is_whole(monkeypatch, tmp_path):
    # ranks that start together each build what is out of date, while others load it
    import os
    import subprocess
    import pytest
    target = tmp_path / "lib.so"
    target.write_text("old")
    written = []

    class Result:
        returncode, stdout, stderr = 0, "", ""

    def compiler(cmd, **kw):
        out = cmd[cmd.index("-o") + 1]
        written.append(out)
        open(out, "w").write("half")
        assert target.read_text() == "old" and os.path.dirname(out) == str(tmp_path)
        open(out, "w").write("new")
        return Result
    monkeypatch.setattr(subprocess, "run", compiler)
    monkeypatch.setattr(build, "LIB_PATH", str(target))
    monkeypatch.setattr(build, "NATIVE_PATH", str(target))
    for make in (build.build_lib, build.build_native):
        target.write_text("old")
        Result.returncode = 1
        with pytest.raises(RuntimeError):
            make()
        assert target.read_text() == "old" and os.listdir(tmp_path) == ["lib.so"]
        Result.returncode = 0
        make()
        assert target.read_text() == "new" and os.listdir(tmp_path) == ["lib.so"]
    assert str(target) not in written
