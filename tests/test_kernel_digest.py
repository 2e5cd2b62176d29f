"""bench.kernel_digest(): comments do not move it, code in any included file does."""
import os
import shutil
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_digest_follows_the_code_of_every_included_file(tmp_path):
    sys.path.insert(0, ROOT)
    import bench
    csrc = shutil.copytree(os.path.join(ROOT, "paper_1807_04638_gb300", "csrc"), tmp_path / "csrc")
    base = bench.kernel_digest()
    assert bench.kernel_digest(csrc) == base
    for name, moves in (("stage_length.cu", True), ("stage.cuh", True), ("line.cuh", True), ("plane.cuh", True),
                        ("launch_util.cuh", True), ("radix.cuh", True), ("fft_fast.cuh", True), ("common.cuh", True),
                        ("engine.cuh", False)):
        text = (csrc / name).read_text()
        (csrc / name).write_text(text + "\n// a remark\n/* and\n   another */\n")
        assert bench.kernel_digest(csrc) == base, name
        (csrc / name).write_text(text + "\nstatic const int one_more = 1;\n")
        assert (bench.kernel_digest(csrc) != base) == moves, name
        (csrc / name).write_text(text)
