"""The bench line's FP64 roofline comes from committed captures (CPU): every entry names a profile
that quotes its source prefix and counts, the fullest pipe is the bound, and a changed source or a
workload without a capture reports none."""
import os

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_entries_are_in_the_profiles():
    assert len(bench.PIPE_INSTRUCTIONS) >= 3
    for key, (counts, src, sha, profile) in bench.PIPE_INSTRUCTIONS.items():
        text = open(os.path.join(ROOT, profile), encoding="utf-8").read()
        assert f"`csrc/{src}` with SHA-1 prefix `{sha}`" in text, key
        for k, v in counts.items():
            shown = [f"{v / 1e6:.{d}f} M" for d in (2, 3)]
            assert k in bench.PIPE_PEAK and any(t in text for t in shown), (key, k)


def test_the_fullest_pipe_is_the_bound(monkeypatch):
    monkeypatch.setattr(bench, "peaks", lambda: {"fp64_gflops": 1250.0, "fp64_src": "given"})
    (kernel, workload), (counts, _, sha, _) = next(iter(bench.PIPE_INSTRUCTIONS.items()))
    monkeypatch.setattr(bench, "source_sha1", lambda name: sha)
    ms, mhz, nsm = 0.125, 2000.0, 152
    line = bench.fp64_roofline(kernel, kernel, workload, 1e9, ms, mhz, nsm)
    clocks = ms * 1e-3 * nsm * mhz * 1e6
    fracs = {k: v / clocks / bench.PIPE_PEAK[k] for k, v in counts.items()}
    assert line["bound"] == max(fracs, key=fracs.get)
    assert abs(line["frac"] - max(fracs.values())) < 1e-12 and line["frac"] < 1.0
    assert abs(line["method"]["gflops"] - 8000.0) < 1e-6
    monkeypatch.setattr(bench, "source_sha1", lambda name: "0" * 12)
    assert bench.fp64_roofline(kernel, kernel, workload, 1e9, ms, mhz, nsm)["frac"] is None
    assert bench.fp64_roofline(kernel, kernel, "other", 1e9, ms, mhz, nsm)["frac"] is None
