"""When the native side of the binding is compiled again."""
import subprocess


def test_the_extension_module_is_rebuilt_for_another_torch(monkeypatch, tmp_path):
    from paper_2510_26577_b200 import build
    build.build()
    ran = []

    def compile_only_in_name(cmd, **kw):
        ran.append(cmd[0])
        return subprocess.CompletedProcess(cmd, 0, "", "")

    monkeypatch.setattr(build.subprocess, "run", compile_only_in_name)
    monkeypatch.setattr(build, "OBJ", str(tmp_path))
    build._build_calls()  # no record of what the module was built against
    assert ran == ["g++"]
    build._build_calls()  # the record of the call above
    assert ran == ["g++"]
    monkeypatch.setattr(build, "_built_against", lambda torch_dir: "another torch")
    build._build_calls()
    assert ran == ["g++"] * 2
