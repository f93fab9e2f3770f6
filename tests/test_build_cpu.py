"""The incremental build: a unit is stale when any header it may include is newer,
the device-code headers (*.cuh) as well as the plain ones."""
import os

from paper_1410_6685_gb300 import build


def test_every_kind_of_header_counts(tmp_path, monkeypatch):
    csrc, include = tmp_path / "csrc", tmp_path / "include"
    csrc.mkdir()
    include.mkdir()
    files = [csrc / "a.h", csrc / "b.cuh", include / "c.h"]
    monkeypatch.setattr(build, "CSRC", str(csrc))
    monkeypatch.setattr(build, "ROOT", str(tmp_path))
    for f in files:
        f.write_text("")
    for newest in files:
        for i, f in enumerate(files):
            t = 2000 if f == newest else 1000 + i
            os.utime(f, (t, t))
        assert build._headers_mtime() == 2000
