"""When the extension module is compiled again (no GPU, nothing is compiled here)."""
import os

from paper_2412_20386_b200 import build as lib_build


def test_extension_is_rebuilt_for_another_torch(monkeypatch, tmp_path):
    so, stamp = tmp_path / "_ptq_torch.so", tmp_path / "versions"
    monkeypatch.setattr(lib_build, "_EXT", str(so))
    monkeypatch.setattr(lib_build, "_EXT_STAMP", str(stamp))
    built = []
    monkeypatch.setattr(lib_build, "up_to_date", lambda target=None, deps=None: target is None or os.path.exists(target))
    monkeypatch.setattr(lib_build, "_run", lambda cmd, target, verbose: (built.append(target), open(target, "w").close()))
    lib_build.build()
    lib_build.build()
    assert built == [str(so)]                                # once: the second call finds it up to date
    real = lib_build.importlib.metadata.version
    monkeypatch.setattr(lib_build.importlib.metadata, "version", lambda name: "0.0" if name == "torch" else real(name))
    lib_build.build()
    lib_build.build()
    assert built == [str(so)] * 2
