"""The search's traffic record is void once either search source changes (CPU only)."""
import bench


def test_record_hash_covers_both_search_sources(tmp_path, monkeypatch):
    h = bench.device_hash()
    for name in ("PM_SRC", "PM_DIRECT_SRC"):
        src = open(getattr(bench, name), encoding="utf-8").read()
        f = tmp_path / name
        f.write_text("// another build\n" + src, encoding="utf-8")
        with monkeypatch.context() as m:
            m.setattr(bench, name, str(f))
            assert bench.device_hash() not in (None, h), name
    assert bench.device_hash() == h
