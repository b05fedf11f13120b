"""When the built files count as current."""


def test_native_part_is_stale_for_another_torch(tmp_path, monkeypatch):
    from paper_2603_02631_b200 import build
    build.build_library()
    assert not build.is_stale() and build.native_is_for() == build._running()
    note = tmp_path / "for"
    monkeypatch.setattr(build, "NATIVE_FOR_PATH", str(note))
    assert build.is_stale()                                # not on record
    note.write_text("python 3.0, torch 0.1\n")
    assert build.is_stale()
    note.write_text(build._running() + "\n")
    assert not build.is_stale()
