"""The library's device images are stored as they are: unpacking a compressed one
would cost the first context of every process about 11 ms."""
import re

from paper_2311_08872_gb300 import build as libbuild


def test_device_images_are_not_compressed():
    """Every level kernel that the library registers by name has a code section of that
    name in plain sight (the names inside a compressed image are not)."""
    image = open(libbuild.build(), "rb").read()
    names = set(re.findall(rb"\0(_ZN2dk12level_kernelI\w+)(?=\0)", image))
    assert len(names) >= 40
    missing = [n for n in names if b".text." + n not in image]
    assert not missing, (len(missing), len(names), missing[0])
