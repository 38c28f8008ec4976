"""The DRAM traffic that bench.py reports comes from a profiler capture on record: only one of the kernel as it is counts (CPU)."""
import json

import bench


def test_a_capture_of_another_version_of_the_kernel_does_not_count(tmp_path):
    path = tmp_path / "traffic.json"
    digest = bench.kernel_digest("rabit_gemv_lut.cu")
    for entry, want in [({"dram_bytes_per_step": 7, "kernel_digest": digest}, 7), ({"dram_bytes_per_step": 7, "kernel_digest": digest[::-1] + "x"}, None),
                        ({"dram_bytes_per_step": 7}, None)]:
        path.write_text(json.dumps({"step": entry}))
        assert bench.recorded_traffic("step", str(path)) == want
        assert bench.recorded_traffic("another step", str(path)) is None
    assert bench.recorded_traffic("step", str(tmp_path / "missing.json")) is None


def test_the_digest_ignores_comments_only(tmp_path, monkeypatch):
    csrc = tmp_path / "paper_2602_05367_b200" / "csrc"
    csrc.mkdir(parents=True)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    digests = []
    for text in ("int a = 1;  // one\n", "/* one\n   two */ int  a=1;\n", "int a = 2;\n"):
        (csrc / "k.cu").write_text(text)
        digests.append(bench.kernel_digest("k.cu"))
    assert digests[0] == digests[1] != digests[2]
