"""The build stores device code uncompressed: unpacking it at a length's first
launch made the first call of a process slower than all of its work."""
from paper_2110_10156_gb300 import build


def test_device_code_is_not_compressed():
    assert "--compress-mode=none" in build.NVCC_FLAGS
