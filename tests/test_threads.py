"""Contexts belong to a thread each, launchers to all of them: what a launcher keeps from its first call on a device is atomic."""
import glob
import os
import re

from paper_2510_04147_b200 import build


def test_what_launchers_keep_per_device_is_atomic():
    plain = []
    for path in glob.glob(os.path.join(build.CSRC, "*.cu")):
        with open(path) as f:
            plain += [(os.path.basename(path), m) for m in re.findall(r"^\s*static (?!PerDevice|std::atomic)\w[\w:<> ]*\[kMaxDevices\].*", f.read(), re.M)]
    assert plain == []
