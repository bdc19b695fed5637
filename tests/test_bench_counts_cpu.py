"""bench.py's claims about a step: the kernels of a rebuild by brick size, and what the executed
samples of a rate are."""
import bench


def test_kernels_of_a_rebuild():
    ct = (512, 512, 400)
    assert bench.rebuild_launches(8, ct) == 6
    assert bench.rebuild_launches(16, ct) == 10  # the 8^3 tiles and their fields as well
    assert bench.rebuild_launches(16, (64, 64, 64)) == 6  # too few bricks for tiles
    assert bench.rebuild_launches(16, (128, 64, 64)) == 10 and 8 * 4 * 4 == 128


def test_executed_samples_are_named_by_what_counts_them():
    assert "8^3 tiles" in bench.counted_by(16) and "16^3" in bench.counted_by(16)
    assert bench.counted_by(8) == "samples in occupied 8^3 bricks"
    assert "brick" not in bench.counted_by(0)
