"""The build is repeated when any source it compiles has changed (no GPU, no
compilation)."""
import os
import shutil

from paper_2403_16862_gb300 import build


def test_stamp_covers_every_source_and_header(tmp_path, monkeypatch):
    root = tmp_path / "repo"
    csrc = root / "package" / "csrc"
    shutil.copytree(build.CSRC, csrc)
    shutil.copytree(os.path.join(build.ROOT, "include"), root / "include")
    monkeypatch.setattr(build, "ROOT", str(root))
    monkeypatch.setattr(build, "CSRC", str(csrc))
    before = build._stamp(build._sources())
    assert build._stamp(build._sources()) == before
    files = sorted(csrc.iterdir()) + sorted((root / "include").iterdir())
    assert {f.suffix for f in files} == {".cu", ".cuh", ".h"}
    for f in files:
        text = f.read_text()
        f.write_text(text + "\n// changed\n")
        assert build._stamp(build._sources()) != before, f.name
        f.write_text(text)
    assert build._stamp(build._sources()) == before
