"""A recorded DRAM traffic figure counts only for the sources it was taken on,
the headers among them."""
import shutil

import bench


def test_digest_covers_the_headers(tmp_path):
    csrc = str(tmp_path / "csrc")
    shutil.copytree(bench.CSRC, csrc)
    before = {f: bench.source_digest(f, csrc) for f in ("decode.cu", "encode.cu", "hist_lut.cu")}
    assert len(set(before.values())) == 3
    assert before["decode.cu"] == bench.source_digest("decode.cu")
    with open(tmp_path / "csrc" / "decode_span.cuh", "a") as f:
        f.write("// changed\n")
    assert all(bench.source_digest(f, csrc) != d for f, d in before.items())


def test_digest_of_one_source_leaves_the_others(tmp_path):
    csrc = str(tmp_path / "csrc")
    shutil.copytree(bench.CSRC, csrc)
    with open(tmp_path / "csrc" / "encode.cu", "a") as f:
        f.write("// changed\n")
    assert bench.source_digest("encode.cu", csrc) != bench.source_digest("encode.cu")
    assert bench.source_digest("decode.cu", csrc) == bench.source_digest("decode.cu")


def test_figure_is_taken_for_its_source_only(tmp_path):
    path = tmp_path / "traffic.txt"
    path.write_text(f"decode.cu {bench.source_digest('decode.cu')} {bench.WORKLOAD} 123\n"
                    f"encode.cu {'0' * 16} {bench.WORKLOAD} 456\n")
    assert bench._traffic_for("decode.cu", str(path)) == 123.0
    assert bench._traffic_for("encode.cu", str(path)) is None
