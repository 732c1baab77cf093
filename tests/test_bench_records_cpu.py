"""bench.py (no GPU): a record is used only while every header it names is unchanged."""
import hashlib

import bench


def test_records_name_the_headers_they_depend_on(tmp_path, monkeypatch):
    csrc = tmp_path / "paper_2003_03590_gb300" / "csrc"
    csrc.mkdir(parents=True)
    hashes = {}
    for name in ("gp_fft.cuh", "gp_sweep.cuh", "gp_tma.cuh", "gp_plane.cuh", "gp_warp.cuh", "gp_ztile.cuh"):
        (csrc / name).write_text(f"// {name}\n")
        hashes[name] = hashlib.sha256((csrc / name).read_bytes()).hexdigest()[:16]
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    prof = tmp_path / "profiles"
    prof.mkdir()
    cur = bench.kernel_source_hash()
    (prof / "ncu_traffic.txt").write_text(f"# gp_warp.cuh {hashes['gp_warp.cuh']}\n# gp_ztile.cuh {hashes['gp_ztile.cuh']}\n"
                                          f"# k_ztile<1024> (a comment with more words)\nk_ztile<1024> 1024 17.0 {cur}\n")
    assert bench.ncu_traffic("k_ztile<1024>", 1024) == 17.0
    for name in ("gp_ztile.cuh", "gp_warp.cuh"):
        text = (csrc / name).read_text()
        (csrc / name).write_text(text + "// changed\n")
        assert bench.ncu_traffic("k_ztile<1024>", 1024) is None
        (csrc / name).unlink()
        assert bench.ncu_traffic("k_ztile<1024>", 1024) is None
        (csrc / name).write_text(text)
    assert bench.ncu_traffic("k_ztile<1024>", 1024) == 17.0
