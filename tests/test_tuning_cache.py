"""A tuning cached by another version of the library is not taken."""
from paper_1908_06742_gb300 import build as B
from paper_1908_06742_gb300 import ddflb as D
from paper_1908_06742_gb300 import tuning


class _Other:
    def ddflb_version(self):
        return b"ddflb of another day"


def test_version_is_part_of_the_key(tmp_path, monkeypatch):
    B.build()
    monkeypatch.setenv("DDFLB_TUNE_CACHE", str(tmp_path / "tuning.json"))
    cfgs = [D.Config(nx=64, ny=64)]
    k = tuning.key("lattice", cfgs)
    assert D.load().ddflb_version().decode() in k
    tuning.store(k, {"choice": [128, 1, 1]})
    assert tuning.lookup(tuning.key("lattice", cfgs)) == {"choice": [128, 1, 1]}
    monkeypatch.setattr(D, "load", lambda *a: _Other())
    assert tuning.lookup(tuning.key("lattice", cfgs)) is None
